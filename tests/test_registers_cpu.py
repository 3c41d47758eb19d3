"""Kernels that change the registers of their warps as they run (setmaxnreg): what they run is inlined, and what they ask for was there at launch.
Checked on the compiler's listing and in the sources."""
import glob
import os
import re
import subprocess

import pytest

from paper_2511_21317_b200 import build as httm_build

CSRC = httm_build.CSRC
CALLED = """
__device__ __noinline__ float helper(float x) { return x * x + 1.f; }
__device__ __forceinline__ float inlined(float x) { return x * x + 2.f; }
__global__ void kernel(float* p) { p[0] = %s(p[1]); }
"""


def test_every_file_that_changes_registers_is_listed():
    using = [os.path.basename(p) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))) if "setmaxnreg" in re.sub(r"//.*", "", open(p).read())]
    assert using and sorted(using) == sorted(httm_build.NO_CALLS)


@pytest.mark.parametrize("name,want", [("helper", True), ("inlined", False)])
def test_a_function_that_is_called_is_found_in_the_listing(tmp_path, name, want):
    src = tmp_path / "f.cu"
    src.write_text(CALLED % name)
    res = subprocess.run([httm_build._nvcc(), *httm_build.NVCC_FLAGS, "-Xptxas", "-v", "-c", str(src), "-o", str(tmp_path / "f.o")],
                         capture_output=True, text=True, check=True)
    found = httm_build.called_functions(res.stdout + res.stderr)
    assert any("helper" in f for f in found) == want and len(found) == want, found


@pytest.mark.parametrize("src", httm_build.NO_CALLS)
def test_nothing_is_called_and_the_registers_were_there(tmp_path, src):
    res = subprocess.run([httm_build._nvcc(), *httm_build.NVCC_FLAGS, "-Xptxas", "-v", "-I", httm_build.INCLUDE, "-c", os.path.join(CSRC, src), "-o",
                          str(tmp_path / "f.o")], capture_output=True, text=True, check=True)
    log = res.stdout + res.stderr
    assert httm_build.called_functions(log) == []
    code = open(os.path.join(CSRC, src)).read()
    role, most = map(int, re.search(r"kScoreRoleRegs = (\d+), kScoreMaxRegs = (\d+)", code).groups())
    groups = int(re.search(r"SC_GROUPS = (\d+)", code).group(1))
    at = log.index("big_scores_kernel")
    used = int(re.search(r"Used (\d+) registers", log[at:]).group(1))
    assert used * (128 + groups * 256) >= 128 * role + groups * 256 * most


def test_calls_with_many_blocks_do_not_pay_for_blocks_shared_out(tmp_path):
    """Both kinds of the score kernel have the registers their split needs, and the kind for many blocks spills no more than the kernel did before there was another."""
    src = os.path.join(CSRC, "httm_big_blocks.cu")
    res = subprocess.run([httm_build._nvcc(), *httm_build.NVCC_FLAGS, "-Xptxas", "-v", "-I", httm_build.INCLUDE, "-c", src, "-o", str(tmp_path / "f.o")],
                         capture_output=True, text=True, check=True)
    log, code = res.stdout + res.stderr, open(src).read()
    role, most = map(int, re.search(r"kScoreRoleRegs = (\d+), kScoreMaxRegs = (\d+)", code).groups())
    groups = int(re.search(r"SC_GROUPS = (\d+)", code).group(1))
    kernels = [m.end() for m in re.finditer(r"Compiling entry function '[^']*big_scores_kernel", log)]
    used = [int(re.search(r"Used (\d+) registers", log[at:]).group(1)) for at in kernels]
    spills = [int(re.search(r"(\d+) bytes spill loads", log[at:]).group(1)) for at in kernels]
    assert len(kernels) == 2 and min(used) * (128 + groups * 256) >= 128 * role + groups * 256 * most
    assert min(spills) <= 368, spills
