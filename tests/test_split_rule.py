"""The rule that sends a reconcile to the split kernel (split_takes, a host
function), compiled into a small program and run on the CPU."""
import subprocess

import pytest

from paper_2607_21224_gb300 import build

PROGRAM = r"""
#include "cpdp_split.cuh"
#include <cstdio>
int main() {
    cpdp::ReconcileCall c{};
    int method, opt, state_sync, bf16, W;
    long long N;
    while (std::scanf("%d %d %d %d %d %lld", &method, &opt, &state_sync, &bf16, &W, &N) == 6) {
        c.method = method, c.opt = opt, c.state_sync = state_sync != 0, c.bf16 = bf16 != 0, c.W = W, c.N = N;
        std::printf("%d\n", cpdp::split_takes(c) ? 1 : 0);
    }
}
"""


@pytest.fixture(scope="module")
def takes(tmp_path_factory):
    """takes(calls): whether the split kernel gets each (method, opt, state_sync, bf16, W, N)."""
    folder = tmp_path_factory.mktemp("split_rule")
    source, program = folder / "rule.cu", folder / "rule"
    source.write_text(PROGRAM)
    subprocess.run([build.nvcc_path(), "-std=c++17", *build.ARCH, f"-I{build.INCLUDE}", f"-I{build.CSRC}", "-o",
                    str(program), str(source)], check=True, capture_output=True, text=True)
    codes = {"cpdp": 0, "localsgd": 1, "ddp": 2}

    def run(calls):
        lines = "".join(f"{codes[m]} {int(o == 'adamw')} {int(s)} {int(b)} {W} {N}\n" for m, o, s, b, W, N in calls)
        r = subprocess.run([str(program)], input=lines, capture_output=True, text=True, check=True)
        return [line == "1" for line in r.stdout.split()]
    return run


VARIANTS = [(m, o, s, b) for m in ("cpdp", "localsgd", "ddp") for o in ("sgd", "adamw") for s in (False, True) for b in (False, True)
            if not (m == "ddp" and s)]


def test_no_call_that_passes_32_bit_offsets(takes):
    """The kernel's offsets are 32-bit: W rows of N / V loads must stay below 2^31, whatever the limits on W and N."""
    calls = [(*v, W, N) for v in VARIANTS for W in (9, 64, 1000, 4096, 8192, 1 << 15, 1 << 20, 1 << 24, 1 << 28)
             for N in (2, 3, 1_001, 4_096, 60_001, 160_000, 300_001, 419_999, 420_000)]
    taken = takes(calls)
    assert any(taken)
    for (*v, W, N), got in zip(calls, taken):
        if got:
            assert W * (N // (2 if N % 2 == 0 else 1)) < 1 << 31, (*v, W, N)
