"""The rules that choose a launch (host functions of the kernel headers),
compiled into a small program and run on the CPU."""
import subprocess

import pytest

from launch_rules import VARIANTS, edges, split_limit
from paper_2607_21224_gb300 import build

CODES = {"cpdp": 0, "localsgd": 1, "ddp": 2}

PROGRAM = r"""
#include "cpdp_shapes.cuh"
#include "cpdp_split.cuh"
#include <cstdio>
#include <type_traits>
int main() {
    cpdp::ReconcileCall c{};
    int method, opt, state_sync, bf16, W;
    long long N;
    while (std::scanf("%d %d %d %d %d %lld", &method, &opt, &state_sync, &bf16, &W, &N) == 6) {
        c.method = method, c.opt = opt, c.state_sync = state_sync != 0, c.bf16 = bf16 != 0, c.W = W, c.N = N;
        std::printf("%d %d", cpdp::split_takes(c) ? 1 : 0,
                    cpdp::walks_alternate(W, N, opt == cpdp::kOptAdamW, method == cpdp::kMethodCPDP, bf16 ? 2 : 4) ? 1 : 0);
        for (int columns : {1, 2, 4}) std::printf(" %d", cpdp::reconcile_threads(method, opt, state_sync, W, N, columns));
        const auto narrow = [&](auto adamw, auto states) {
            constexpr int O = decltype(adamw)::value ? cpdp::kOptAdamW : cpdp::kOptSGD;
            constexpr bool S = decltype(states)::value;
            const bool ddp = method == cpdp::kMethodDDP;
            std::printf(" %lld %lld\n",
                        (long long)(ddp ? cpdp::ragged_narrow_columns<cpdp::kMethodDDP, 1, O, S>(W)
                                        : cpdp::ragged_narrow_columns<cpdp::kMethodCPDP, 1, O, S>(W)),
                        (long long)cpdp::ragged_narrow_columns<cpdp::kMethodCPDP, 2, O, S>(W));
        };
        const std::true_type yes;
        const std::false_type no;
        if (opt)
            state_sync ? narrow(yes, yes) : narrow(yes, no);
        else
            state_sync ? narrow(no, yes) : narrow(no, no);
    }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    """rules(calls) for each call (method, opt, state_sync, bf16, W, N): taken by the split kernel; walk direction
    alternates; threads per block at 1, 2 and 4 columns per thread; columns to which a ragged row gets one load per
    thread, odd N and N = 2 mod 4."""
    folder = tmp_path_factory.mktemp("launch_rules")
    source, program = folder / "rules.cu", folder / "rules"
    source.write_text(PROGRAM)
    subprocess.run([build.nvcc_path(), "-std=c++17", *build.ARCH, f"-I{build.INCLUDE}", f"-I{build.CSRC}", "-o",
                    str(program), str(source)], check=True, capture_output=True, text=True)

    def run(calls):
        lines = "".join(f"{CODES[m]} {int(o == 'adamw')} {int(s)} {int(b)} {W} {N}\n" for m, o, s, b, W, N in calls)
        r = subprocess.run([str(program)], input=lines, capture_output=True, text=True, check=True)
        return [tuple(map(int, line.split())) for line in r.stdout.splitlines()]
    return run


def test_no_split_call_passes_32_bit_offsets(rules):
    """The kernel's offsets are 32-bit: W rows of N / V loads must stay below 2^31, whatever the limits on W and N."""
    calls = [(*v, W, N) for v in VARIANTS for W in (9, 64, 1000, 4096, 8192, 1 << 15, 1 << 20, 1 << 24, 1 << 28)
             for N in (2, 3, 1_001, 4_096, 60_001, 160_000, 300_001, 419_999, 420_000)]
    taken = [split for split, *_ in rules(calls)]
    assert any(taken)
    for (*v, W, N), got in zip(calls, taken):
        if got:
            assert W * (N // (2 if N % 2 == 0 else 1)) < 1 << 31, (*v, W, N)


@pytest.mark.parametrize("W", [8, 9, 15, 16, 23, 24, 31, 32, 47, 48, 99, 100, 4096])
def test_split_limits(rules, W):
    """Both sides of every limit, for every variant."""
    cases = [(v, odd, N, N <= split_limit(*v, W, odd))
             for v in VARIANTS for odd in (False, True) for N in edges(split_limit(*v, W, odd), odd) if N > 0]
    for (v, odd, N, want), (taken, *_) in zip(cases, rules([(*v, W, N) for v, _, N, _ in cases])):
        assert taken == want, (v, W, N)


def test_walks_alternate_only_past_what_l2_keeps(rules):
    """Below 30 MB a step's arrays are in L2 anyway, and a block whose columns move to another SM each time loses by it."""
    calls = [(*v, W, N) for v in VARIANTS for W in (1, 2, 3, 8, 64, 4096)
             for N in (3201, 30_000, 140_000, 433_007, 600_000, 1 << 20, 3_000_001, 3_750_000, 6_000_000, 1 << 28)]
    for (method, opt, _, bf16, W, N), (_, alternates, *_) in zip(calls, rules(calls)):
        step = W * N * ((12 if opt == "adamw" else 8) + (2 if bf16 else 4)) + (8 * N if method == "cpdp" else 0)
        assert alternates == (step >= 30e6), (method, opt, bf16, W, N, step)


def test_blocks_last_longer_than_the_gpu_takes_to_start_them(rules):
    """Past 65,536 columns a block has 768 elements of each array or the most threads there are; above 4 million
    columns 256 threads, except where smaller blocks gain."""
    sizes = [65_537, 100_000, 855_424, 1 << 20, 1_800_000, 1 << 22]
    calls = [(*v, W, N) for v in VARIANTS for W in (1, 2, 3, 4, 5, 6, 8, 64) for N in sizes]
    for (*v, W, N), (_, _, *threads, _, _) in zip(calls, rules(calls)):
        for columns, t in zip((1, 2, 4), threads):
            assert t in (64, 128, 256) and (t == 256 or t * columns * W >= 768), (*v, W, N, columns, t)
            assert t == 64 or t // 2 * columns * W < 768, (*v, W, N, columns, t)
    small = rules([(*v, W, N) for v in VARIANTS for W in (1, 2, 64) for N in (1, 3201, 65_536)])
    assert all(t == 64 for _, _, *threads, _, _ in small for t in threads)
    large = [(*v, 8, (1 << 22) + 4) for v in VARIANTS]
    for (method, opt, state_sync, *_), (_, _, *threads, _, _) in zip(large, rules(large)):
        assert threads[2] == (64 if opt == "adamw" and state_sync else 256)


@pytest.mark.parametrize("method,opt,state_sync,W,odd,even", [
    ("cpdp", "sgd", False, 1, 150_000, 450_000), ("ddp", "sgd", False, 2, 260_000, 500_000),
    ("cpdp", "sgd", False, 3, 330_000, 500_000), ("ddp", "sgd", False, 3, 250_000, 500_000),
    ("localsgd", "sgd", True, 2, 260_000, 1_500_000), ("cpdp", "sgd", True, 3, 700_000, 1_500_000),
    ("cpdp", "sgd", True, 24, 330_000, 1_500_000), ("cpdp", "adamw", False, 2, 450_000, 1_500_000),
    ("localsgd", "adamw", True, 7, 400_000, 1_500_000), ("ddp", "adamw", False, 8, 400_000, 1_500_000)])
def test_columns_to_which_a_ragged_row_gets_one_load_per_thread(rules, method, opt, state_sync, W, odd, even):
    assert rules([(method, opt, state_sync, False, W, 100_001)])[0][-2:] == (odd, even)
