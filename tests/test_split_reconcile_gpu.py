"""The reconcile of many workers over few columns (rows split across the warps
of a block) against the column kernels: the first N columns of a wider problem
must give the same bits, since both add the workers in order. Worker counts
leave partial rounds of 64 and 32 rows and partial row chunks; sizes sit at the
edges of a block's 64 or 32 columns and of the rule that selects the kernel."""
import os
import subprocess
import sys
from pathlib import Path

import pytest
import torch

from launch_rules import split_limit
from test_ragged_reconcile_gpu import VARIANTS, _arrays, _state

pytestmark = pytest.mark.gpu

ROOT = Path(__file__).resolve().parents[1]
WIDE, WIDEST = 160_004, 420_004  # even, and past the sizes the rule takes: the column kernels


def _match(W, N, wide=WIDE):
    gen = torch.Generator(device="cuda").manual_seed(N * 512 + W)
    theta0 = torch.randn(wide, device="cuda", generator=gen) * 0.05
    grads = [torch.randn((W, wide), device="cuda", generator=gen) * 1e-2 for _ in range(2)]
    for method, opt, state_sync, dtype in VARIANTS:
        with _state(W, N, method, opt, state_sync) as a, _state(W, wide, method, opt, state_sync) as b:
            a.init_params(theta0[:N].clone())
            b.init_params(theta0)
            for g in grads:
                for step in ("local_step", "reconcile"):
                    getattr(a, step)(g[:, :N].to(dtype).contiguous())
                    getattr(b, step)(g.to(dtype))
            columns = "reconcile_scalar_kernel" if N % 4 else "reconcile_vec4_kernel"
            split = N <= split_limit(method, opt, state_sync, dtype == torch.bfloat16, W, N % 2 == 1)
            assert a.reconcile_kernel() == ("reconcile_split_kernel" if split else columns)
            assert b.reconcile_kernel() == "reconcile_vec4_kernel"
            for x, y in zip(_arrays(a), _arrays(b)):
                assert torch.equal(x, y[..., :N]), (method, opt, state_sync, dtype)


@pytest.mark.parametrize("W", [9, 15, 24, 33, 64, 65, 131])
@pytest.mark.parametrize("N", [1, 2, 31, 33, 63, 66, 129, 4098, 23_999])
def test_split_rows_match_the_column_kernels(N, W):
    _match(W, N)


@pytest.mark.parametrize("W,N,wide", [
    (8, 1200, WIDE), (9, 64_000, WIDE), (9, 64_004, WIDE), (15, 64_002, WIDE), (16, 80_002, WIDE), (16, 160_000, WIDE),
    (32, 160_002, WIDE), (24, 64_002, WIDE), (23, 24_001, WIDE), (24, 31_999, WIDE), (24, 32_001, WIDE), (24, 63_999, WIDE),
    (24, 64_001, WIDE), (16, 110_001, WIDE), (24, 109_999, WIDE), (48, 110_001, WIDE), (9, 159_999, WIDE),
    (9, 249_999, WIDEST), (9, 250_001, WIDEST), (24, 299_999, WIDEST), (24, 300_001, WIDEST), (24, 419_999, WIDEST),
    (24, 420_001, WIDEST), (100, 60_001, WIDE), (100, 110_001, WIDE), (100, 299_999, WIDEST), (100, 300_001, WIDEST),
    (63, 8_194, WIDE), (65, 8_195, WIDE)])
def test_the_rule_that_selects_it(W, N, wide):
    """Each variant on the side of its limit where it belongs, and the same bits on both."""
    _match(W, N, wide)


def test_the_most_workers():
    W, N = 4096, 66  # a wider problem would be too large: fewer workers instead
    gen = torch.Generator(device="cuda").manual_seed(1)
    with _state(W, N, "cpdp", "sgd", False) as a, _state(W // 16, N, "cpdp", "sgd", False) as b:
        theta0 = torch.randn(N, device="cuda", generator=gen) * 0.05
        g = torch.randn((W // 16, N), device="cuda", generator=gen) * 1e-2
        for st, grads in ((a, g.repeat(16, 1)), (b, g)):
            st.init_params(theta0)
            st.local_step(grads)
            st.reconcile(grads)
        assert a.reconcile_kernel() == "reconcile_split_kernel"
        # 16 copies of 256 workers have the same means, to the rounding of 4,096-term sums
        assert torch.allclose(a.anchor, b.anchor, rtol=0, atol=4096 * 2.0 ** -24 * float(a.anchor.abs().max()))
        assert torch.equal(a.params, a.params[:1].expand_as(a.params))


CHECKED = """
import sys
sys.path[:0] = [{root!r}, {root!r} + "/tests"]
import torch
from test_ragged_reconcile_gpu import VARIANTS, _state
from paper_2607_21224_gb300 import cpdp
bad = 0
for W, N in ((9, 66), (24, 129), (65, 1001), (131, 33), (24, 300_001), (32, 160_000), (3, 1_500_006), (9, 500_003), (8, 3 * 1024 + 126)):
    for method, opt, state_sync, dtype in VARIANTS:
        with _state(W, N, method, opt, state_sync) as st:
            st.init_params(torch.zeros(N, device="cuda"))
            st.reconcile(torch.ones((W, N), device="cuda", dtype=dtype))
            bad += cpdp.cpdp_bad_index_count(st.ctx)
print("bad", bad)
"""


def test_index_checked_build_counts_no_bad_index():
    from paper_2607_21224_gb300 import build
    lib = build.build_library(checked=True)
    r = subprocess.run([sys.executable, "-c", CHECKED.format(root=str(ROOT))], capture_output=True, text=True,
                       env=dict(os.environ, CPDP_LIBRARY=str(lib)), timeout=600)
    assert r.returncode == 0 and r.stdout.split()[-2:] == ["bad", "0"], r.stdout + r.stderr[-2000:]
