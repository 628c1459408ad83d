"""The reconcile for N not a multiple of 4 (pairs of columns where N is even,
single ones where it is odd) against the vector kernel: the same columns padded
to a multiple of 4 must give the same bits, since every sum runs over the
workers in the same order. Sizes sit at the edges of a warp's columns, of a
block's and of the size rule (cpdp_shapes.cuh), and above 2^31 row offsets."""
import itertools

import pytest
import torch

from paper_2607_21224_gb300 import workloads as wls
from paper_2607_21224_gb300.state import CPDPState
from parity import run_and_check, windows

pytestmark = pytest.mark.gpu

VARIANTS = [v for v in itertools.product(("cpdp", "localsgd", "ddp"), ("sgd", "adamw"), (False, True),
                                         (torch.float32, torch.bfloat16)) if not (v[0] == "ddp" and v[2])]


def _state(W, N, method, opt, state_sync):
    hyper = dict(lr=1e-3, momentum=0.0, weight_decay=0.05) if opt == "adamw" else dict(lr=0.1, momentum=0.9, weight_decay=5e-4)
    st = CPDPState(W, N, K=1, beta=0.5, alpha=0.75, **hyper)
    st.set_method(method)
    if opt == "adamw":
        st.set_adamw()
    st.set_state_reconcile(state_sync)
    return st


def _arrays(st):
    return [x for x in (st.params, st.mom, st.anchor, st.slow_v, getattr(st, "exp_avg_sq", None)) if x is not None]


@pytest.mark.parametrize("W,N", [(W, N) for W in (1, 3, 7, 8)
                                 for N in (2, 31, 33, 62, 66, 127, 130, 255, 1022, 1025, 3 * 1024 + 126, 200_001, 400_003,
                                           500_002, 700_002, 1_500_002)]
                         + [(1, 150_003), (1, 330_001), (1, 450_002), (2, 1), (2, 126), (2, 4099), (2, 100_002), (2, 260_001),
                            (2, 330_003), (2, 450_001), (2, 1_500_006), (3, 249_999), (4, 250_001), (7, 329_999), (8, 330_001), (8, 399_999)]
                         + [(W, N) for W in (9, 17, 33) for N in (420_003, 500_002, 1_500_002)])
def test_ragged_columns_match_the_vector_kernel(W, N):
    M = (N + 3) // 4 * 4  # the vector kernel's size: the same columns and up to 3 more
    gen = torch.Generator(device="cuda").manual_seed(N * 16 + W)
    theta0 = torch.randn(M, device="cuda", generator=gen) * 0.05
    grads = [torch.randn((W, M), device="cuda", generator=gen) * 1e-2 for _ in range(2)]
    for method, opt, state_sync, dtype in VARIANTS:
        with _state(W, N, method, opt, state_sync) as a, _state(W, M, method, opt, state_sync) as b:
            a.init_params(theta0[:N].clone())
            b.init_params(theta0)
            for g in grads:  # a local step first, so that the replicas differ when they are averaged
                for step in ("local_step", "reconcile"):
                    getattr(a, step)(g[:, :N].to(dtype).contiguous())
                    getattr(b, step)(g.to(dtype))
            assert a.reconcile_kernel() == "reconcile_scalar_kernel"
            for x, y in zip(_arrays(a), _arrays(b)):
                assert torch.equal(x, y[..., :N]), (method, opt, state_sync, dtype)


@pytest.mark.parametrize("N", [(1 << 28) + 1, (1 << 29) + 2])
def test_ragged_reconcile_with_64_bit_offsets(N):
    """8 rows of 2^28 + 1 single columns, or of 2^28 + 1 pairs: the row offsets pass 2^31."""
    wl = wls.Workload("ragged_largest", W=8, tensors=tuple(wls.flat_tensors(N, 1, 0.05)), K=2, T=3, grad_dtype="bf16")
    run_and_check(wl, cols=windows(wl, width=512, n_random=2048, boundaries=0))
