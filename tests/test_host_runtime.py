"""Host code of the library over a stand-in CUDA runtime (fake_cudart.c), in a
child process: what it does when a launch is rejected, what it allocates and
what it launches.  No GPU is needed or used."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes, os, sys
sys.path.insert(0, {root!r})
import numpy as np
from paper_2207_13962_gb300 import fslbm
fake = ctypes.CDLL({fake!r})
def var(name, kind=ctypes.c_int):
    return kind.in_dll(fake, name)
shape = (40, 9, 5)
fill, flags = np.zeros(1800), np.zeros(1800, np.uint8)
def context(precision="FP32", init=True, shape=shape, vel=None, den=None, **kw):
    n = shape[0] * shape[1] * shape[2]
    c = fslbm.Context(shape, precision=precision, **kw)
    if init:
        c.init(np.zeros(n), np.zeros(n, np.uint8), vel, den)
    return c
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """Runs a script with the stand-in in place of the CUDA runtime."""
    from paper_2207_13962_gb300 import build
    build.build()
    lib = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", lib, os.path.join(HERE, "fake_cudart.c")], check=True)

    def go(script):
        r = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT, fake=lib) + script],
                           env=dict(os.environ, LD_PRELOAD=lib), capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
        return r.stdout
    return go


@pytest.mark.parametrize("precision", ["FP64", "FP32", "FP16SMC"])
def test_a_rejected_launch_is_reported(run, precision):
    """Whichever launch of an init, of a batch's set-up or of a timed step is
    rejected, the call that made it fails: no step graph without one of its
    stages, and a later attempt succeeds."""
    run(f"""
n0 = var("fake_launches").value
c = context({precision!r}, bubble_model=True); c.close()
n = var("fake_launches").value - n0
assert n > 20
def fails(call, k):
    var("fake_fail_at").value = var("fake_launches").value + k
    try:
        call()
    except fslbm.FslbmError as e:
        assert e.status == fslbm.ECUDA, e.status
        return True
    finally:
        var("fake_fail_at").value = -1
    return False
c = context({precision!r}, init=False, bubble_model=True)
init = lambda: c.init(fill, flags)
missed = [k for k in range(n) if not fails(init, k)]
assert not missed, missed
init()
members = [context({precision!r}) for _ in range(2)]
n0 = var("fake_launches").value
b = fslbm.Batch(members)
n = var("fake_launches").value - n0
assert n >= 9
missed = [k for k in range(n) if not fails(lambda: fslbm.Batch(members), k)]
assert not missed, missed
missed = [k for k in range(n) if not fails(lambda: b.set_tuning(1, 2), k)]
assert not missed, missed
b.set_tuning(1, 2)
c.set_timing(True)
missed = [k for k in range(8) if not fails(lambda: c.step(1), k)]
assert not missed, missed
c.step(1)
""")


@pytest.mark.parametrize("precision", ["FP64", "FP32", "FP16S", "BF16S", "FP32MC", "FP16SMC"])
def test_memory_estimate_covers_what_a_context_takes(run, precision):
    """The admission estimate against the bytes that create and init allocate
    at most, with every array staged twice: never less, and above it by no
    more than the partials of the SMs the device does not have (the estimate
    allows for 256 SMs), the bubbles it allows for and the small change."""
    run(f"""
for q in (19, 27):
    for shape in ((1, 1, 1), (3, 2, 1), (40, 9, 5), (64, 33, 17)):
        n = shape[0] * shape[1] * shape[2]
        for sms in (152, 256):
            var("fake_sms").value = sms
            base = var("fake_bytes", ctypes.c_size_t).value
            var("fake_peak", ctypes.c_size_t).value = base
            c = context({precision!r}, shape=shape, q=q, bubble_model=True, vel=np.zeros(3 * n), den=np.ones(n),
                        axis_order=(2, 1, 0))
            took = var("fake_peak", ctypes.c_size_t).value - base
            c.close()
            est = fslbm.memory_estimate(shape, q, {precision!r}, with_velocity=True)
            slack = (256 - sms) * 4 * 8 * 8 + 8192
            assert took <= est <= took + slack, (q, shape, sms, took, est)
""")


@pytest.mark.parametrize("precision,most", [("FP64", 2), ("FP32", 4), ("FP16SMC", 4)])
@pytest.mark.parametrize("fit", [1, 2, 3, 4, 9])
def test_a_batch_launches_no_more_sweep_blocks_than_fit(run, precision, most, fit):
    """Every tuning up to the format's limit is accepted; the persistent sweep
    gets that many blocks per SM, or as many as can be resident at once."""
    run(f"""
var("fake_occupancy").value = {fit}
members = [context({precision!r}, q=27) for _ in range(2)]
block, grid = (ctypes.c_uint * 4096).in_dll(fake, "fake_block"), (ctypes.c_uint * 4096).in_dll(fake, "fake_grid")
def sweep(call):
    first = var("fake_launches").value
    out = call()
    k = first + 1  # after the plan kernel
    assert block[k] == 256
    return out, grid[k]
b, g = sweep(lambda: fslbm.Batch(members))
assert g == 152 * min({most}, {fit}), g
assert b.tuning()["bulk_blocks_per_sm"] == min({most}, {fit})
for t in range(1, {most} + 1):
    _, g = sweep(lambda: b.set_tuning(t, 2))
    assert g == 152 * min(t, {fit}), (t, g)
    assert b.tuning()["bulk_blocks_per_sm"] == t
for t in (0, {most} + 1):
    try:
        b.set_tuning(t, 2)
    except fslbm.FslbmError as e:
        assert e.status == fslbm.EINVAL
    else:
        raise AssertionError(t)
""")
