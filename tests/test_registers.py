"""Register budgets of the FP64 step kernels.

The binary and ternary kernels are compiled for a number of blocks per SM; where that
leaves fewer registers than a node's populations need, the compiler keeps them in local
memory, which no output shows.  The compiler's own count of spilled bytes (-Xptxas -v) is
bounded by what the populations take in their two forms, the double gathered and the
integer collided: a budget beyond that sends every number of a node through memory.
Solvers whose collision runs in FP64 arithmetic have kernels of their own, without a
tighter budget, and spill nothing.
"""

import os
import re
import subprocess

import pytest

from paper_1808_06787_gb300 import build

SOURCE = """
#include "kernels.cuh"
namespace lbms {
template __global__ void k_step<%(lat)s, %(s)d, double, false, false, %(fixed)s>(StepParams<double>);
template __global__ void k_step<%(lat)s, %(s)d, double, true, false, %(fixed)s>(StepParams<double>);
}
"""


@pytest.mark.parametrize("fixed", ["true", "false"])
@pytest.mark.parametrize("s", [1, 2])
@pytest.mark.parametrize("lat", ["LBMS_D2Q9", "LBMS_D3Q7", "LBMS_D3Q15"])
def test_fp64_steps_spill_no_more_than_their_populations(lat, s, fixed, tmp_path):
    src = tmp_path / "k.cu"
    src.write_text(SOURCE % {"lat": lat, "s": s, "fixed": fixed})
    r = subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS
                       + ["-Xptxas", "-v", "-c", str(src), "-o", os.devnull],
                       capture_output=True, text=True, cwd=str(tmp_path))
    assert r.returncode == 0, r.stderr
    spills = [int(v) for v in re.findall(r"(\d+) bytes spill stores", r.stderr)]
    assert len(spills) >= 2 and max(spills) <= (2 * 8 * s * int(lat[8:]) if fixed == "true" else 0), spills


@pytest.mark.parametrize("lat,s,most", [("LBMS_D2Q5", 3, 48), ("LBMS_D2Q4", 3, 48), ("LBMS_D3Q6", 4, 64)])
def test_fp32_steps_leave_room_for_the_next_grid(lat, s, most, tmp_path):
    """Blocks of 256 threads: five per SM with 48 registers, four with 64."""
    src = tmp_path / "k.cu"
    src.write_text('#include "kernels.cuh"\nnamespace lbms {\n'
                   "template __global__ void k_step<%s, %d, float, false, false>(StepParams<float>);\n}\n" % (lat, s))
    r = subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS
                       + ["-Xptxas", "-v", "-c", str(src), "-o", os.devnull],
                       capture_output=True, text=True, cwd=str(tmp_path))
    assert r.returncode == 0, r.stderr
    used = [int(v) for v in re.findall(r"Used (\d+) registers", r.stderr)]
    assert used and max(used) <= most, used


@pytest.mark.parametrize("lat,s,blocks", [("LBMS_D2Q5", 2, 3), ("LBMS_D2Q9", 2, 3), ("LBMS_D3Q7", 2, 3), ("LBMS_D3Q15", 2, 2)])
def test_fp64_batch_steps_keep_their_blocks_per_sm(lat, s, blocks, tmp_path):
    """65536 registers in units of 8 per thread, blocks of 256 threads."""
    src = tmp_path / "k.cu"
    src.write_text('#include "batch.cuh"\nnamespace lbms {\n'
                   "template __global__ void k_batch_step<%s, %d, double, false, false>(BatchParams<double>, "
                   "const double*);\n}\n" % (lat, s))
    r = subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS
                       + ["-Xptxas", "-v", "-c", str(src), "-o", os.devnull],
                       capture_output=True, text=True, cwd=str(tmp_path))
    assert r.returncode == 0, r.stderr
    used = [int(v) for v in re.findall(r"Used (\d+) registers", r.stderr)]
    assert used and max(used) <= 65536 // (256 * blocks) // 8 * 8, used
