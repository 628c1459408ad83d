"""What the rules that choose a reconcile's kernel are meant to say, written
down once for the tests that check them on the CPU and on the GPU."""
import itertools

VARIANTS = [v for v in itertools.product(("cpdp", "localsgd", "ddp"), ("sgd", "adamw"), (False, True), (False, True))
            if not (v[0] == "ddp" and v[2])]  # method, optimizer, state reconciliation, bf16 gradients


def split_limit(method, opt, state_sync, bf16, W, odd):
    """The largest N of which the split kernel takes a reconcile."""
    if W < 9:
        return 0
    if not odd:
        return 64_000 if W < 16 else 160_000
    if state_sync:
        return 300_000 if W >= 100 and (opt, method) != ("sgd", "cpdp") else 64_000 if W >= 24 else 24_000
    if bf16:
        return 110_000 if W >= 48 else 64_000 if W >= 24 else 24_000
    if opt == "sgd":
        if W >= 24:
            return 300_000
        return 250_000 if method == "ddp" else 110_000 if method == "localsgd" and W >= 16 else 24_000
    if W >= 24 and method != "cpdp":
        return 420_000
    return 300_000 if W >= 100 else 110_000 if W >= 16 else 24_000


def edges(limit, odd):
    """The largest N of that parity within the limit and the smallest beyond it."""
    last = limit - (limit % 2 != odd)
    return last, last + 2
