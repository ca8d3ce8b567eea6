"""Observables of states that no run leaves behind: a checkpoint may hold any
numbers, and what is reported for them has to be what the fields say."""
import numpy as np
import pytest

from paper_2207_13962_gb300 import scenarios as S

pytestmark = pytest.mark.gpu

PRECISIONS = ["FP64", "FP32", "FP16S", "BF16S", "FP32MC", "FP16SMC"]
HEADER = 64  # bytes in front of a checkpoint's arrays: PDFs, types, fill levels, masses, ...


def _arrays(raw, c):
    """A checkpoint's PDF bytes, types, and the bytes of its fill levels and masses (views but for the types)."""
    pdf_bytes = int(raw[HEADER - 8:HEADER].view(np.int64)[0])
    at = HEADER + pdf_bytes
    return (raw[HEADER:at], raw[at:at + c.N] & 3, raw[at + c.N:at + 9 * c.N], raw[at + 9 * c.N:at + 17 * c.N])


def _edited(c, which, cell, value):
    """The context's checkpoint with one value of its fill levels (which = 2) or masses (3) replaced."""
    buf = c.save()
    field = _arrays(buf, c)[which]
    field[8 * cell:8 * cell + 8] = np.frombuffer(np.float64(value).tobytes(), np.uint8)
    return buf


@pytest.mark.parametrize("precision", PRECISIONS)
def test_liquid_cells_mass_and_fill_level_count(precision, gpu_lib):
    from paper_2207_13962_gb300 import fslbm
    sc = S.random_interface(shape=(23, 17, 9), seed=4)
    c = fslbm.context_for(sc, precision=precision)
    c.step(2)
    before = c.observables()
    assert before["nan_seen"] == 0
    types = _arrays(c.save(), c)[1]
    cell = int(np.flatnonzero(types == S.LIQ)[7])
    kept = c.save()
    c.load(_edited(c, 2, cell, 0.5))
    o = c.observables()
    # at most 23 * 17 * 9 additions of numbers up to the volume
    assert abs(o["liquid_volume"] - (before["liquid_volume"] - 0.5)) <= c.N * 2.0 ** -53 * before["liquid_volume"]
    assert o["nan_seen"] == 0 and o["total_mass"] == before["total_mass"]
    c.load(kept)
    c.load(_edited(c, 3, cell, np.nan))
    o = c.observables()
    assert o["nan_seen"] == 1 and o["status"] == fslbm.EUNSTABLE
    c.load(kept)
    assert c.observables() == before
    c.close()


def _stored(raw, precision, q, cells):
    """Deviations that the PDF bytes of a checkpoint hold, as float64 (exact), direction-major."""
    pad = (cells + 63) // 64 * 64
    size = {"FP32": 4, "FP16S": 2, "BF16S": 2, "FP32MC": 4, "FP16SMC": 2}[precision]
    body, rest = raw[:q * pad * size], raw[q * pad * size:]
    if precision.startswith("FP32"):
        d = body.view(np.float32).astype(np.float64)
    elif precision == "BF16S":
        d = (body.view(np.uint16).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    else:
        d = body.view(np.float16).astype(np.float64) * 2.0 ** -15
    d = d.reshape(q, pad)[:, :cells].copy()
    if precision.endswith("MC"):
        d[0] = rest.view(np.int32)[:cells] * 2.0 ** (-34 if precision == "FP32MC" else -30)
    return d


def _draw(rng, precision, q, cells, kind):
    """PDF bytes of `cells` cells: deviations of one size, of sizes over 40 powers of two, or beyond 2."""
    d = rng.uniform(-1.0, 1.0, (q, cells))
    if kind == "spread":
        d = np.sign(d) * 2.0 ** -rng.uniform(3.2, 40.0, d.shape)
    elif kind == "far":
        d *= 2.0 ** rng.uniform(0.0, 20.0, d.shape)
    elif precision == "FP32MC":
        d *= 0.1249
    pad = (cells + 63) // 64 * 64
    out = np.zeros((q, pad))
    out[:, :cells] = d
    if precision == "FP32":
        return np.frombuffer(out.astype(np.float32).tobytes(), np.uint8)
    if precision == "BF16S":
        return np.frombuffer((out.astype(np.float32).view(np.uint32) >> 16).astype(np.uint16).tobytes(), np.uint8)
    if precision == "FP16S":
        return np.frombuffer((out * 2.0 ** 15).astype(np.float16).tobytes(), np.uint8)
    shift = 34 if precision == "FP32MC" else 30
    if precision == "FP32MC":  # stored values lie on the grid
        body = (np.rint(out * 2.0 ** shift) * 2.0 ** -shift).astype(np.float32).tobytes()
    else:
        x = out * 2.0 ** 15
        body = np.where(np.abs(x) < 0.0625, np.rint(x * 2.0 ** 15) * 2.0 ** -15, x).astype(np.float16).tobytes()
    rest = rng.integers(-2 ** 31 + 1, 2 ** 31, pad, dtype=np.int64).astype(np.int32)
    return np.frombuffer(body + rest.tobytes(), np.uint8)


@pytest.mark.parametrize("kind", ["even", "spread", "far"])
@pytest.mark.parametrize("precision,q", [("FP32", 19), ("FP32", 27), ("FP16S", 27), ("BF16S", 19), ("FP32MC", 27),
                                         ("FP16SMC", 19)])
def test_mass_and_velocity_of_any_cell(precision, q, kind, gpu_lib):
    """One liquid cell.  Its mass is 1 + the exact sum of what is stored to 2^-53 (once rounded) and 2^-54
    (the sum), as close as a sum in FP64; deviations of 2 and more are summed in FP64 (q roundings of
    partial sums).  |u| is what FP32 gives with that density rounded once, bit for bit."""
    import math
    from fractions import Fraction
    from oracle.oracle import lattice
    from paper_2207_13962_gb300 import fslbm
    if kind == "far" and precision not in ("FP32", "BF16S"):
        pytest.skip("the format holds no such deviation")
    f4 = np.float32
    cx = np.array(lattice(q)[0])
    rng = np.random.default_rng(q)
    c = fslbm.Context((1, 1, 1), precision=precision, q=q, periodic=(True, True, True))
    c.init(np.ones(1), np.full(1, S.LIQ, np.uint8))
    for _ in range(150):
        buf = c.save()
        _arrays(buf, c)[0][:] = _draw(rng, precision, q, 1, kind)
        d = _stored(_arrays(buf, c)[0], precision, q, 1)[:, 0]
        exact = 1 + sum(Fraction(float(x)) for x in d)
        c.load(buf)
        o = c.observables()
        err = abs(Fraction(o["total_mass"]) - exact)
        if np.abs(d).max() < 2.0 or precision.endswith("MC"):
            assert err <= Fraction(2) ** -53 * max(abs(exact), 1) + Fraction(2) ** -54, (float(err), float(exact))
        else:
            assert err <= Fraction(2) ** -53 * (q + 2) * sum(abs(Fraction(float(x))) for x in d) + Fraction(2) ** -53
        if precision.endswith("MC") or abs(float(exact)) < 2.0 ** -6:
            continue
        rho = f4(float(exact))
        j = [f4(0.0)] * 3
        for i in range(q):
            for a in range(3):
                if cx[i, a]:
                    j[a] = f4(j[a] + f4(d[i])) if cx[i, a] > 0 else f4(j[a] - f4(d[i]))
        u = [float(f4(x / rho)) for x in j]
        assert o["max_u"] == math.sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
        assert (o["nan_seen"] != 0) == (not rho > 0)
    c.close()


@pytest.mark.parametrize("precision,q", [("FP32", 19), ("BF16S", 27), ("FP16S", 19), ("FP32MC", 19), ("FP16SMC", 27)])
def test_mass_of_many_cells(precision, q, gpu_lib):
    """More cells than the reduction has threads, every deviation anywhere in its range: the mass is the
    exact one to the roundings of the reduction's tree (some 40 additions of FP64 sums)."""
    import math
    from paper_2207_13962_gb300 import fslbm
    shape = (101, 97, 53)
    n = int(np.prod(shape))
    rng = np.random.default_rng(3)
    c = fslbm.Context(shape, precision=precision, q=q, periodic=(True, True, True))
    c.init(np.ones(n), np.full(n, S.LIQ, np.uint8))
    buf = c.save()
    raw = _arrays(buf, c)[0]
    raw[:] = _draw(rng, precision, q, n, "spread")
    d = _stored(raw, precision, q, n)
    exact = math.fsum(d.reshape(-1)) + n
    c.load(buf)
    o = c.observables()
    assert abs(o["total_mass"] - exact) <= 40 * 2.0 ** -53 * exact
    c.close()
