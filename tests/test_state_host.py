"""CPDPState's own code, as far as it runs without a GPU."""
import importlib.util
import types

import pytest
import torch

from paper_2607_21224_gb300 import state as state_module


def _fresh_module():
    """state.py executed once more, beside the imported one."""
    spec = importlib.util.spec_from_file_location("paper_2607_21224_gb300._state_again", state_module.__file__)
    module = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(module)
    return module


@pytest.mark.parametrize("private", [True, False])
def test_current_stream_with_and_without_torchs_private_function(private, monkeypatch):
    asked = []
    if private:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda index: asked.append(index) or 0x51, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
        monkeypatch.setattr(torch.cuda, "current_stream",
                            lambda index: asked.append(index) or types.SimpleNamespace(cuda_stream=0x51))
    module = _fresh_module()
    st = object.__new__(module.CPDPState)
    st.ctx, st._device_index = None, 3
    assert st._stream(None) == 0x51 and asked == [3]
    assert st._stream(0x77) == 0x77
    assert st._stream(types.SimpleNamespace(cuda_stream=0x88)) == 0x88
