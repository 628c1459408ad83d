"""Launches of a context alternate between walking the arrays forwards and
backwards; the direction must not change a bit. One context takes a step more
than the other before both start over, so the same steps run in opposite
directions."""
import pytest
import torch

from test_ragged_reconcile_gpu import VARIANTS, _arrays, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [1, 2, 3, 4, 6, 8])
@pytest.mark.parametrize("N", [4, 1028, 1027, 1026, 4 * (256 * 5 + 3), 200_003, 700_006])
def test_either_direction_gives_the_same_bits(N, W):
    gen = torch.Generator(device="cuda").manual_seed(N * 16 + W)
    theta0 = torch.randn(N, device="cuda", generator=gen) * 0.05
    grads = [torch.randn((W, N), device="cuda", generator=gen) * 1e-2 for _ in range(2)]
    for method, opt, state_sync, dtype in VARIANTS:
        with _state(W, N, method, opt, state_sync) as a, _state(W, N, method, opt, state_sync) as b:
            b.init_params(theta0)
            b.local_step(grads[0].to(dtype))
            for st in (a, b):
                st.init_params(theta0)
                for g in grads:
                    st.local_step(g.to(dtype))
                    st.reconcile(g.to(dtype))
            for x, y in zip(_arrays(a), _arrays(b)):
                assert torch.equal(x, y), (method, opt, state_sync, dtype)
