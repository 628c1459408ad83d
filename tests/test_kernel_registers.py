"""What ptxas reports for the kernels that every training step runs: a register
spill in the local step costs 5 to 13 % where the state sits in L2."""
import re
import subprocess

from paper_2607_21224_gb300 import build

PROGRAM = r"""
#include "cpdp_kernels.cuh"
#include "cpdp_shapes.cuh"
namespace cpdp {
#define STEP(OPT, G, ONCE)                                                                                  \
    template __global__ void local_step_kernel<OPT, G, kLocalUnroll, LocalWarpRuns<OPT, G>::value, ONCE>(   \
        float*, float*, float*, const G*, int64_t, StepArgs, int);
STEP(kOptSGD, float, false)
STEP(kOptSGD, float, true)
STEP(kOptSGD, bf16_bits, false)
STEP(kOptSGD, bf16_bits, true)
STEP(kOptAdamW, float, false)
STEP(kOptAdamW, bf16_bits, false)
}
"""


def test_no_local_step_spills(tmp_path):
    source = tmp_path / "local_step.cu"
    source.write_text(PROGRAM)
    r = subprocess.run([build.nvcc_path(), "-O3", "-std=c++17", *build.ARCH, "-lineinfo", "-Xptxas", "-v",
                        f"-I{build.INCLUDE}", f"-I{build.CSRC}", "-c", "-o", str(tmp_path / "local_step.o"), str(source)],
                       check=True, capture_output=True, text=True)
    report = re.findall(r"Function properties for \S*local_step_kernel(\S*)\s+(\d+) bytes stack frame, "
                        r"(\d+) bytes spill stores, (\d+) bytes spill loads", r.stdout + r.stderr)
    assert len(report) == 6
    assert all((stack, stores, loads) == ("0", "0", "0") for _, stack, stores, loads in report), report
