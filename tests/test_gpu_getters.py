"""The FP32-mixed getters widen the stored 32-bit values exactly: zeros of both
signs, subnormals, the ends of the normal range; positions are (cell + offset)
times the cell size, and one that rounds up to the end of the box reads 0."""
import numpy as np
import pytest

from paper_2101_12149_gb300 import pic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

VALUES = np.array([0.0, -0.0, 1e-45, -3e-42, 1.1754942e-38, 1.17549435e-38, -1.2e-38, 1.0, -0.1, 1 / 3, 2.0 ** 24 + 1,
                   -3.4e38, 3.4028235e38, 1e-7], dtype=np.float64)


@pytest.mark.parametrize("d", [(1.0, 1.0, 1.0), (0.5, 1.0, 0.7)])
@pytest.mark.parametrize("n", [(6, 5, 7), (8, 8, 32)])
def test_fp32_mixed_getters_are_exact(n, d):
    m = VALUES.size
    frac = np.array([0.0, 1e-46, 2.0 ** -40, 0.25, 0.5, 1 - 2.0 ** -24, 1 - 2.0 ** -30, 1 / 3, 0.9, 0.1, 0.7, 1e-3, 0.6,
                     0.999])
    parts = {}
    for a, k in enumerate("xyz"):
        cell = np.arange(m) % n[a]
        cell[6] = n[a] - 1  # its fraction rounds to 1 in 32 bits: the next cell, which wraps to 0
        parts[k] = (cell + frac) * d[a]
    for k in ("ux", "uy", "uz"):
        parts[k] = VALUES.copy()
    parts["w"] = np.abs(VALUES[::-1]).copy()
    c = pic.Context(n, d=d, precision=pic.FP32_MIXED, order=1)
    c.load_particles(-1.0, 1.0, parts)
    got = c.get_particles()
    o = np.argsort(got["id"])
    for k in ("ux", "uy", "uz", "w"):
        want = parts[k].astype(np.float32).astype(np.float64)
        assert np.array_equal(got[k][o].view(np.int64), want.view(np.int64)), k
    for a, k in enumerate("xyz"):
        p = parts[k] / d[a]
        cell = np.minimum(np.floor(p), n[a] - 1)
        f = (p - cell).astype(np.float32)
        up = f >= 1.0
        cell, f = np.where(up, (cell + 1) % n[a], cell), np.where(up, np.float32(0), f)
        want = (cell + f.astype(np.float64)) * d[a]
        want = np.where(want >= n[a] * d[a], want - n[a] * d[a], want)
        assert np.array_equal(got[k][o], want), (k, got[k][o] - want)


def test_fp32_mixed_field_getter_is_exact():
    n = (6, 5, 7)
    F = np.resize(VALUES, (9,) + n)
    c = pic.Context(n, precision=pic.FP32_MIXED, order=1)
    c.set_fields(F)
    want = F.astype(np.float32).astype(np.float64)
    assert np.array_equal(c.get_fields()[:6].view(np.int64), want[:6].view(np.int64))
