"""What holds for the kernels' sources as a whole, in every build."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2207_13962_gb300", "csrc")


def test_no_kernel_waits_for_asynchronous_copies():
    """Bulk and asynchronous copies need a wait for everything in flight on
    every path out of a kernel, a given-up wait included; no kernel, whatever
    macros it is built with, starts one or waits on a barrier in memory."""
    used = []
    for name in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, name)).read()
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)
        used += [(name, w) for w in ("mbarrier", "cp.async", "try_wait") if w in src]
    assert not used, used


@pytest.mark.parametrize("dyn", [0, 1, 4])
def test_every_hand_out_of_the_sweep_compiles(dyn, tmp_path):
    """FSLBM_BULK_DYN: units handed out 1, 4 at a time, or 0 for a fixed stride."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src = tmp_path / "hand_out.cu"
    src.write_text('''#include "fslbm_bulk.cuh"
__global__ void k(int n, int* counter, int* seen) {
  fslbm::hand_out_units<fslbm::StoreF32>(n, counter, [&](int w) { atomicAdd(&seen[w], 1); });
}''')
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", f"-DFSLBM_BULK_DYN={dyn}",
                    "-I", CSRC, "-c", str(src), "-o", str(tmp_path / "hand_out.o")], check=True)
