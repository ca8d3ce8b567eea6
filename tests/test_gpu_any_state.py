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
