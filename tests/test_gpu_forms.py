"""Kernels that take one of several forms by size, at both sides of each line,
and the compact lists at their fullest.

* The interface kernel updates a short band with the lattice directions in the
  lanes of a warp and a long one with a thread a cell.  A domain alone is
  below the line, a batch of copies of it above: the two forms round alike, so
  the results are equal bit for bit.
* The bulk sweep hands a short list out unit by unit and a long one in chunks:
  the same comparison.
* The conversion stages walk their lists with a warp an entry: more converting
  cells than the grid has warps, against the oracle.
* The geometry tiles list the points they need: every cell an interface cell
  (full lists), against the oracle.
* The observables keep FP64 out of the per-cell work of the deviation formats:
  against plain FP64 sums of the state read back.
"""
import numpy as np
import pytest

from oracle import Oracle
from paper_2207_13962_gb300 import scenarios as S

pytestmark = pytest.mark.gpu

FREE_SLIP = 2
BATCH_BAND = {("FP64", 19): 1280, ("FP64", 27): 1280, ("FP32", 19): 5120, ("FP32", 27): 8192,
              ("FP32MC", 19): 5120, ("FP16S", 19): 5120, ("BF16S", 27): 8192, ("FP16SMC", 27): 8192}


def _alone_and_batch(sc, copies, steps, **kw):
    from paper_2207_13962_gb300 import fslbm
    alone = fslbm.context_for(sc, **kw)
    members = [fslbm.context_for(sc, **kw) for _ in range(copies)]
    counts = alone.interface_count(), alone.work_counts()
    alone.step(steps)
    batch = fslbm.Batch(members)
    batch.step(steps)
    batch.sync()
    ra = alone.read()
    for m in (members[0], members[-1]):
        rm = m.read()
        for k in ("flags", "fill", "mass", "pdf"):
            np.testing.assert_array_equal(rm[k], ra[k], err_msg=k)
    batch.close()
    for c in [alone] + members:
        c.close()
    return counts


@pytest.mark.parametrize("precision,q,collision,variant,periodic,cs", [
    ("FP64", 19, "TRT", "NBRC", (1, 0, 1), 0.0),
    ("FP64", 27, "SRT", "OM3", (FREE_SLIP, 0, 1), 0.1),
    ("FP32", 19, "TRT", "OM", (0, 0, 0), 0.0),
    ("FP32", 27, "SRT", "NBKC", (FREE_SLIP,) * 3, 0.1),
    ("FP32", 19, "TRT", "OM3", (1, FREE_SLIP, 1), 0.1),
    ("FP32MC", 19, "TRT", "NBRC", (1, 0, 0), 0.0),
    ("FP16S", 19, "SRT", "OM", (1, 0, 1), 0.0),
    ("BF16S", 27, "TRT", "OM", (1, 0, 1), 0.0),
    ("FP16SMC", 27, "TRT", "OM", (0, 0, 1), 0.0),
])
def test_band_by_lanes_equals_band_by_threads(precision, q, collision, variant, periodic, cs, gpu_lib):
    sc = S.random_interface(shape=(37, 21, 11), seed=7, q=q, collision=collision, variant=variant)
    line = BATCH_BAND[precision, q]
    band = int((sc.flags == S.IFACE).sum())
    copies = line // band + 2
    assert band <= line < copies * band
    _alone_and_batch(sc, copies, 15, precision=precision, periodic=periodic, smagorinsky_cs=cs)


@pytest.mark.parametrize("precision,copies", [("FP32", 2), ("FP16SMC", 6)])
def test_units_one_by_one_equal_units_in_chunks(precision, copies, gpu_lib):
    """442,368 liquid cells at first: with four blocks of eight warps on each
    of 152 SMs, 2.8 units a warp alone, 5.7 (two copies, the line lies at 4)
    and 17 (six, the line at 16) in the batch."""
    sc = S.dam_break(nx=128, ny=96, nz=64, W=96, H=72)
    _alone_and_batch(sc, copies, 6, precision=precision)


def _against_oracle(shape, fill, flags, vel, steps, **kw):
    from paper_2207_13962_gb300 import fslbm
    o = Oracle(*shape, **kw)
    o.init(fill, flags, vel, None)
    g = fslbm.Context(shape, precision="FP64", **kw)
    g.init(fill, flags, vel, None)
    changed = 0  # interface cells that converted in the first step
    for s in range(1, steps + 1):
        o.step(1)
        g.step(1)
        ro, rg = o.read(), g.read()
        np.testing.assert_array_equal(rg["flags"], ro["flags"], err_msg=f"flags at step {s}")
        fluid = (ro["flags"] == S.LIQ) | (ro["flags"] == S.IFACE)
        for k in ("fill", "mass"):
            assert np.all(np.abs(rg[k][fluid] - ro[k][fluid]) <= 1e-12 * np.abs(ro[k][fluid])), (k, s)
        a, b = rg["pdf"][:, fluid], ro["pdf"][:, fluid]
        assert np.all(np.abs(a - b) <= 1e-12 * np.abs(b)), ("pdf", s)
        if s == 1:
            changed = int(((ro["flags"] != flags) & (flags == S.IFACE)).sum())
    g.close()
    return changed


@pytest.mark.parametrize("q", [19, 27])
def test_more_conversions_than_warps(q, gpu_lib):
    """A sheet of 120 x 120 interface cells, nearly full or nearly empty at
    random and moving up or down with it: thousands of cells convert both ways
    in the first step, more than the grid's 4864 warps."""
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
    changed = _against_oracle(shape, ph.reshape(-1), fl.reshape(-1), v.reshape(-1), 4, q=q, periodic=(True, False, True),
                              variant="OM", omega=1.5, g=(0.0, -1e-5, 0.0), sigma=1e-4)
    assert changed > 4864


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
    _against_oracle(shape, ph, fl, v, 4, q=19, periodic=(True, False, True), variant="NBRC", omega=1.2,
                    g=(0.0, -1e-5, 0.0), sigma=1e-3)


@pytest.mark.parametrize("precision", ["FP64", "FP32", "FP32MC", "FP16S", "BF16S", "FP16SMC"])
@pytest.mark.parametrize("shape,q", [((6, 7, 3), 27), ((37, 21, 11), 19), ((101, 67, 33), 19)])
def test_observables_against_the_state_read_back(precision, shape, q, gpu_lib):
    """Mass: the PDFs read back are the stored values plus w, rounded once
    each (27 x 2^-53 of a cell's density), and the float pair carries 2^-44 of
    deviations below 0.1; both stay below 1e-13.  max |u|: sums of Q
    floats of at most 0.1 in all and a division, 30 x 2^-24 x 0.1 = 1.8e-7."""
    from paper_2207_13962_gb300 import fslbm
    sc = S.random_interface(shape=shape, seed=4, q=q)
    c = fslbm.context_for(sc, precision=precision)
    c.step(5)
    o, r = c.observables(), c.read()
    fl, pdf = r["flags"], r["pdf"]
    liq, iface = fl == S.LIQ, fl == S.IFACE
    assert [o["n_gas"], o["n_interface"], o["n_liquid"], o["n_obstacle"]] == [int((fl == k).sum()) for k in range(4)]
    rho = pdf.sum(axis=0)
    mass = rho[liq].sum() + r["mass"][iface].sum()
    assert abs(o["total_mass"] - mass) <= 1e-13 * mass
    vol = liq.sum() + r["fill"][iface].sum()
    assert abs(o["liquid_volume"] - vol) <= 1e-13 * vol
    fluid = liq | iface
    from oracle.oracle import lattice
    cx = np.array(lattice(q)[0], float)
    u = (cx.T @ pdf[:, fluid]) / rho[fluid] - 0.5 * np.array(sc.g)[:, None]
    umax = np.sqrt((u ** 2).sum(axis=0)).max()
    assert abs(o["max_u"] - umax) <= (1e-13 if precision == "FP64" else 1.8e-7)
    assert o["nan_seen"] == 0
    c.close()
