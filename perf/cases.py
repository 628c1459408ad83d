"""The workloads that the hot path is timed on.

One pass is one synchronization period as a training program runs it: K calls of
``CPDPState.step`` (or ``HostGradientPipeline.step``) on K different gradient buffers,
K - 1 local steps and one synchronization step (DDP: every call synchronizes). The state
is that of a run under way: the replicas have drifted from the anchor, the momentum
buffers, second moments and SlowMo velocity are not zero. The outputs are the whole state
after the pass.
"""
from __future__ import annotations

import math

import torch

from paper_2607_21224_gb300 import workloads as wls
from paper_2607_21224_gb300.pipeline import HostGradientPipeline
from paper_2607_21224_gb300.state import CPDPState

ADAM_BETA1, ADAM_BETA2, ADAM_EPS = 0.9, 0.999, 1e-8
STEPS_BEFORE = 500  # optimizer steps taken before the pass (AdamW's bias correction)
# A drawn case moves at most the bytes of the ResNet-50 case at 8 workers.
LARGEST_BYTES = 15.6e9
# A host-fed pass copies this much at most: the host link is some 30 times slower than HBM.
LARGEST_HOST_BYTES = 270e6


def _model_size(model: str, classes: int) -> int:
    build = {"resnet50": wls.resnet50_tensors, "vit_s16": wls.vit_s16_tensors}[model]
    return sum(t.numel for t in build(classes))


def _case(N, W, K, *, method="cpdp", opt="sgd", grads="f32", state_reconcile=False, beta=0.5, heavy_tail=False,
          feed="device", **more):
    return dict(more, N=int(N), W=int(W), K=int(K), method=method, opt=opt, grads=grads,
                state_reconcile=state_reconcile, beta=beta, heavy_tail=heavy_tail, feed=feed)


def listed():
    return [
        # A small MLP (16-64-32-1, 3,201 parameters) trained by 4 workers at K = 2, as the training-loop test does:
        # the smallest calls, where the launch and the host call are all there is.
        _case(3201, 4, 2, beta=0.3, name="mlp_w4"),
        # The benchmark's tiny workload: 2 workers of 2^20 parameters; state and gradients fit in L2.
        _case(1 << 20, 2, 2, name="tiny_w2"),
        # Many simulated workers of a small network (60,000 parameters, 64 workers): more rows than columns per SM.
        _case(60_000, 64, 4, name="small_net_w64"),
        # The benchmark's default workload: ResNet-50/CIFAR-100 shapes, 8 workers, K = 4, momentum SGD.
        _case(_model_size("resnet50", 100), 8, 4, name="resnet50_cifar100_w8"),
        # ViT-S/16 with the paper's optimizer for it (AdamW), bf16 gradients, 8 workers, K = 4.
        _case(_model_size("vit_s16", 100), 8, 4, opt="adamw", grads="bf16", name="vit_s16_adamw_w8"),
        # ResNet-50/TinyImageNet shapes: 16 workers, K = 2, heavy-tailed gradients, beta = 0.7.
        _case(_model_size("resnet50", 200), 16, 2, beta=0.7, heavy_tail=True, name="resnet50_tinyimagenet_w16"),
        # A head of 101 classes makes the parameter count odd: every second row starts off a vector boundary.
        _case(_model_size("resnet50", 101), 4, 2, name="resnet50_101_classes_w4"),
        # A head of 10 classes (N = 2 mod 4), ViT-S/16 with AdamW and bf16 gradients.
        _case(_model_size("vit_s16", 10), 8, 2, opt="adamw", grads="bf16", name="vit_s16_10_classes_w8"),
        # The DDP baseline: every step averages the gradients; ViT-S/16, momentum SGD, bf16 gradients.
        _case(_model_size("vit_s16", 100), 8, 1, method="ddp", grads="bf16", name="vit_s16_ddp_w8"),
        # The LocalSGD baseline on a medium model (2^22 parameters), 4 workers, K = 4.
        _case(1 << 22, 4, 4, method="localsgd", name="localsgd_4m_w4"),
        # Optimizer-state reconciliation with AdamW and float32 gradients, 4 workers, K = 2.
        _case(_model_size("vit_s16", 100), 4, 2, opt="adamw", state_reconcile=True, name="vit_s16_reconcile_state_w4"),
        # Gradients that arrive in page-locked host memory, through the double-buffered pipeline.
        _case(1 << 20, 4, 4, feed="host", name="host_fed_1m_w4"),
    ]


def draw(rng):
    """1 to 256 workers, 2,000 parameters to 34 million, K from 1 to 8; half of the sizes are odd or ragged."""
    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        W, N, K = log_uniform(1, 256), log_uniform(2_000, 34_000_000), rng.choice([1, 2, 2, 4, 4, 8])
        N = N if rng.random() < 0.5 else max(4, N // 4 * 4)
        method = rng.choice(["cpdp", "cpdp", "cpdp", "localsgd", "ddp"])
        opt = rng.choice(["sgd", "sgd", "adamw"])
        grads = rng.choice(["f32", "f32", "bf16"])
        c = _case(N, W, 1 if method == "ddp" else K, method=method, opt=opt, grads=grads,
                  state_reconcile=method != "ddp" and rng.random() < 0.2, beta=rng.choice([0.3, 0.5, 0.7]),
                  heavy_tail=rng.random() < 0.2, feed="host" if rng.random() < 0.1 else "device")
        host_bytes = c["K"] * W * N * (4 if grads == "f32" else 2) if c["feed"] == "host" else 0
        if work(c)["bytes"] <= LARGEST_BYTES and host_bytes <= LARGEST_HOST_BYTES:
            return c


def _hyper(case):
    if case["opt"] == "adamw":
        return dict(lr=5e-4, momentum=0.0, weight_decay=0.05, K=case["K"], beta=case["beta"], alpha=1.0)
    return dict(lr=0.1, momentum=0.9, weight_decay=5e-4, K=case["K"], beta=case["beta"], alpha=1.0)


def _inputs(case, seed):
    """theta0, what the state differs by from a fresh one, and the K gradient buffers (on the GPU)."""
    dev, W, N = torch.device("cuda"), case["W"], case["N"]
    gen = torch.Generator(device=dev)
    gen.manual_seed(wls.seed_for(int(seed), "init"))

    def normal(*shape, std):
        return torch.empty(shape, device=dev).normal_(0.0, std, generator=gen)

    adamw = case["opt"] == "adamw"
    theta0 = normal(N, std=0.05)
    drift = normal(W, N, std=1e-4)
    mom = normal(W, N, std=2.3e-4 if adamw else 2.3e-3)  # of gradients N(0, 1e-3) at beta1 = 0.9 / momentum 0.9
    slow_v = normal(N, std=1e-3)
    sq = normal(W, N, std=1e-3).square_() if adamw else None
    grads = []
    for _ in range(case["K"]):
        g = normal(W, N, std=1e-3)
        if case["heavy_tail"]:  # 1 % of the entries are 100 times as large
            g = torch.where(torch.rand((W, N), generator=gen, device=dev) < 0.01, g * 100.0, g)
        grads.append(g.to(torch.bfloat16) if case["grads"] == "bf16" else g)
    return theta0, drift, mom, slow_v, sq, grads


def prepare(case, seed):
    theta0, drift, mom, slow_v, sq, grads = _inputs(case, seed)
    st = CPDPState(case["W"], case["N"], **_hyper(case))
    st.set_method(case["method"])
    if case["opt"] == "adamw":
        st.set_adamw(ADAM_BETA1, ADAM_BETA2, ADAM_EPS)
    st.set_state_reconcile(case["state_reconcile"])
    st.init_params(theta0)
    st.optimizer_step = STEPS_BEFORE
    st.params += drift
    st.mom.copy_(mom)
    st.slow_v.copy_(slow_v)
    if sq is not None:
        st.exp_avg_sq.copy_(sq)
    if case["feed"] == "host":
        feeder = HostGradientPipeline(st, dtype=grads[0].dtype)
        grads = [g.cpu().pin_memory() for g in grads]
    else:
        feeder = st
    return {"state": st, "feeder": feeder, "grads": grads, "steps_per_epoch": 1000 * case["K"]}


def run(state):
    st, step, T = state["state"], state["feeder"].step, state["steps_per_epoch"]
    for t, g in enumerate(state["grads"], start=1):
        step(g, t, T)
    out = {"params": st.params, "mom": st.mom, "anchor": st.anchor, "slow_v": st.slow_v}
    if getattr(st, "exp_avg_sq", None) is not None:
        out["exp_avg_sq"] = st.exp_avg_sq
    return out


def work(case):
    """Each call reads its gradients and the state once and writes the state once (the calls are separate and leave
    their result in memory); a CPDP synchronization step also reads and writes the anchor and the velocity."""
    W, N, K = case["W"], case["N"], case["K"]
    adamw = case["opt"] == "adamw"
    row = (4 if case["grads"] == "f32" else 2) + (24 if adamw else 16)
    flops = W * N * (14 if adamw else 6) * K
    total = W * N * row * K
    if case["method"] == "cpdp":
        total += 16 * N
    return {"bytes": total, "flops": flops}


def tolerance(case):
    """float32 state, sums over W rows. The velocity is a difference of parameter-sized numbers (0.05 against 1e-3),
    which sets the relative error: against 64 bits 3e-6 to 7e-6 at up to 16 workers and 1e-5 to 2e-5 above, where the
    sums are longer (the other outputs are at 2e-7 or below)."""
    return {"rel": 2.5e-5 if case["W"] <= 16 else 8e-5}


def exact(case, seed):
    """Algorithm 1 in 64 bits, whole arrays at a time."""
    theta0, drift, mom, slow_v, sq, grads = _inputs(case, seed)
    f32 = lambda x: float(torch.tensor(x, dtype=torch.float32))  # noqa: E731  the library takes float32 settings
    h = {k: f32(v) for k, v in _hyper(case).items()}
    b1, b2, eps = f32(ADAM_BETA1), f32(ADAM_BETA2), f32(ADAM_EPS)
    p = (theta0 + drift).double()  # the float32 sum that prepare() stores
    m, v, ref = mom.double(), slow_v.double(), theta0.double()
    s = sq.double() if sq is not None else None
    del drift, mom, slow_v, sq, theta0

    def optimizer(g, n):
        if s is None:
            m.mul_(h["momentum"]).add_(g).add_(p, alpha=h["weight_decay"])
            p.sub_(m, alpha=h["lr"])
            return
        p.mul_(1.0 - h["lr"] * h["weight_decay"])
        m.mul_(b1).add_(g, alpha=1.0 - b1)
        s.mul_(b2).add_(g * g, alpha=1.0 - b2)
        denom = s.sqrt().div_(math.sqrt(1.0 - b2 ** n)).add_(eps)
        p.addcdiv_(m, denom, value=-h["lr"] / (1.0 - b1 ** n))

    for t, g in enumerate(grads, start=1):
        g = g.double()
        sync = case["method"] == "ddp" or t == case["K"]
        if sync and case["method"] != "localsgd":
            g = g.mean(dim=0, keepdim=True)
        optimizer(g, STEPS_BEFORE + t)
        if not sync or case["method"] == "ddp":
            continue
        if case["state_reconcile"]:
            m.copy_(m.mean(dim=0, keepdim=True).expand_as(m))
            if s is not None:
                s.copy_(s.mean(dim=0, keepdim=True).expand_as(s))
        new = p.mean(dim=0)
        if case["method"] == "cpdp":
            v = h["beta"] * v + (new - ref)
            new = ref + h["alpha"] * v
            ref = new
        p.copy_(new.expand_as(p))
    out = {"params": p, "mom": m, "anchor": ref, "slow_v": v}
    if s is not None:
        out["exp_avg_sq"] = s
    return out
