"""What holds for the kernels' sources as a whole, in every build."""
import os
import re

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
