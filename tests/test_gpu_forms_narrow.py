"""The forms of a stage in the deviation formats: that both sides of a line
are met, and the compact lists at their fullest."""
import numpy as np
import pytest

from oracle import Oracle
from paper_2207_13962_gb300 import scenarios as S

pytestmark = pytest.mark.gpu

# units a warp from which the bulk sweep's list is handed out in chunks
HAND_OUT = {"FP64": 16, "FP32": 4, "FP16S": 4, "BF16S": 4, "FP32MC": 6, "FP16SMC": 16}


@pytest.mark.parametrize("precision,q,copies", [("FP64", 19, 4), ("FP32", 19, 3), ("FP32MC", 27, 3), ("BF16S", 19, 3),
                                                ("FP16SMC", 19, 8), ("FP16SMC", 27, 8)])
def test_both_hand_outs_of_the_sweep(precision, q, copies, gpu_lib):
    """A domain alone below the line and a batch of copies above it, by the
    device's own number of warps and the list's own length, by a sixth at
    least; equal bit for bit."""
    import torch
    from paper_2207_13962_gb300 import fslbm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sc = S.dam_break(nx=128, ny=96, nz=64, W=96, H=72, q=q)
    alone = fslbm.context_for(sc, precision=precision)
    members = [fslbm.context_for(sc, precision=precision) for _ in range(copies)]
    batch = fslbm.Batch(members)
    blocks = batch.tuning()["bulk_blocks_per_sm"]
    units, warps = alone.work_counts()["liquid_segments"], sms * blocks * 8
    assert units * 7 / 6 < HAND_OUT[precision] * warps < copies * units * 6 / 7, (units, warps)
    alone.step(6)
    batch.step(6)
    batch.sync()
    ra = alone.read()
    for m in (members[0], members[-1]):
        rm = m.read()
        for k in ("flags", "fill", "mass", "pdf"):
            np.testing.assert_array_equal(rm[k], ra[k], err_msg=k)
    batch.close()
    for c in [alone] + members:
        c.close()


def _first_step(shape, fill, flags, vel, precision, **kw):
    """The first step against the oracle: types, PDFs within 25 u (u = 2^-24, what one FP32 step may
    round) and fill levels within 1e-4 (a share of the excess mass of cells that convert), and one more
    unit in the last place of what a 16-bit format stores."""
    from paper_2207_13962_gb300 import fslbm
    o = Oracle(*shape, **kw)
    o.init(fill, flags, vel, None)
    g = fslbm.Context(shape, precision=precision, **kw)
    g.init(fill, flags, vel, None)
    mass = g.observables()["total_mass"]
    o.step(1)
    g.step(1)
    ro, rg = o.read(), g.read()
    np.testing.assert_array_equal(rg["flags"], ro["flags"])
    fluid = (ro["flags"] == S.LIQ) | (ro["flags"] == S.IFACE)
    dev = np.abs(ro["pdf"][:, fluid]).max()
    ulp = {"FP32": 0.0, "FP32MC": 2.0 ** -34, "FP16SMC": dev * 2.0 ** -10}[precision]
    assert np.abs(rg["pdf"][:, fluid] - ro["pdf"][:, fluid]).max() <= 25 * 2.0 ** -24 + 28 * ulp
    assert np.abs(rg["fill"][fluid] - ro["fill"][fluid]).max() <= 1e-4 + 28 * ulp
    drift = abs(g.observables()["total_mass"] - mass) / mass
    g.close()
    return int(((ro["flags"] != flags) & (flags == S.IFACE)).sum()), drift


@pytest.mark.parametrize("precision", ["FP32", "FP32MC"])
@pytest.mark.parametrize("q", [19, 27])
def test_more_conversions_than_warps(precision, q, gpu_lib):
    """Thousands of cells convert both ways in the first step.  FP32MC keeps the mass: its liquid links are
    exact, what remains is the FP64 arithmetic of at most 28 terms a cell (1e-13)."""
    nx, ny, nz = shape = (120, 8, 120)
    rng = np.random.default_rng(q)
    fl = np.full((nz, ny, nx), S.GAS, np.uint8)
    ph = np.zeros((nz, ny, nx))
    fl[:, :3], ph[:, :3] = S.LIQ, 1.0
    full = rng.random((nz, nx)) < 0.5
    fl[:, 3], ph[:, 3] = S.IFACE, np.where(full, 0.9999, 0.0001)
    v = np.zeros((3, nz, ny, nx))
    v[1, :, 3] = np.where(full, 0.05, -0.05)
    v[1, :, 2] = v[1, :, 3]
    changed, drift = _first_step(shape, ph.reshape(-1), fl.reshape(-1), v.reshape(-1), precision, q=q,
                                 periodic=(True, False, True), variant="OM", omega=1.5, g=(0.0, -1e-5, 0.0), sigma=1e-4)
    assert changed > 4864
    if precision == "FP32MC":
        assert drift <= 1e-13


@pytest.mark.parametrize("shape", [(17, 9, 10), (8, 8, 8), (3, 16, 1)])
@pytest.mark.parametrize("obstacles", [False, True])
def test_every_cell_an_interface_cell(shape, obstacles, gpu_lib):
    rng = np.random.default_rng(5)
    n = int(np.prod(shape))
    fl = np.full(n, S.IFACE, np.uint8)
    ph = rng.uniform(0.3, 0.7, n)
    if obstacles:
        solid = rng.random(n) < 0.1
        fl[solid], ph[solid] = S.OBST, 0.0
    v = np.where(np.tile(fl, 3) == S.IFACE, rng.uniform(-0.01, 0.01, 3 * n), 0.0)
    _first_step(shape, ph, fl, v, "FP32", q=19, periodic=(True, False, True), variant="NBRC", omega=1.2,
                g=(0.0, -1e-5, 0.0), sigma=1e-3)


def test_mass_conserving_storage_costs_little_more(gpu_lib):
    """FP32MC moves as many bytes as FP32 and adds integer sums (1.07 times a step on this domain); with its
    list of 11 units a warp handed out one by one, sectors were read twice (1.42 times)."""
    import torch
    from paper_2207_13962_gb300 import fslbm
    sc = S.dam_break(nx=384, ny=192, nz=96, W=192, H=96)
    us = {}
    for precision in ("FP32", "FP32MC"):
        c = fslbm.context_for(sc, precision=precision, stream=torch.cuda.current_stream().cuda_stream)
        c.step(20)
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            c.step(40)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b) / 40)
        us[precision] = sorted(times)[3]
        c.close()
    assert us["FP32MC"] <= 1.2 * us["FP32"], us
