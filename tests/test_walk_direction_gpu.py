"""Launches of a context alternate between walking the arrays forwards and
backwards where a step's arrays take 30 MB and more; the direction must not
change a bit. One context takes a step more than the other before both start
over, so the same steps run in opposite directions."""
import pytest
import torch

from test_ragged_reconcile_gpu import VARIANTS, _arrays, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,N", [(W, N) for W in (1, 2, 3, 4, 6, 8)
                                 for N in (4, 1028, 1027, 1026, 4 * (256 * 5 + 3), 200_003, 700_006)]
                         + [(W, 8_600_000 // W // 4 * 4 + more) for W in (1, 2, 3, 4, 6, 8, 20)
                            for more in (4 * (64 * 5 + 3), 1027, 1026)])
def test_either_direction_gives_the_same_bits(W, N):
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


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("N", [1_499_999, 1_500_000, 1_500_001, 1 << 23, (1 << 23) + 1])
def test_evict_first_gradients_give_the_same_bits(N, dtype):
    """SGD's local step with its gradients loaded evict-first (6,000,000 to 2^25 elements in all, here 4 workers)
    against single workers, which stay below that."""
    gen = torch.Generator(device="cuda").manual_seed(N)
    theta0 = torch.randn(N, device="cuda", generator=gen) * 0.05
    grads = (torch.randn((4, N), device="cuda", generator=gen) * 1e-2).to(dtype)
    n = 1_000_000  # columns per single worker
    with _state(4, N, "cpdp", "sgd", False) as a:
        a.init_params(theta0)
        for _ in range(2):
            a.local_step(grads)
        for i in range(4):
            for lo in range(0, N, n):
                cols = slice(lo, min(lo + n, N))
                part = grads[i:i + 1, cols].clone()
                with _state(1, part.shape[1], "cpdp", "sgd", False) as b:
                    b.init_params(theta0[cols].clone())
                    for _ in range(2):
                        b.local_step(part)
                    assert torch.equal(a.params[i, cols], b.params[0]) and torch.equal(a.mom[i, cols], b.mom[0])
