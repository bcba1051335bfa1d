"""The table of the inverse Maxwellian speed distribution (CPU)."""
import numpy as np
import pytest

from paper_2309_08655_gb300 import maxwell


def test_series_reproduces_the_distribution():
    special = pytest.importorskip("scipy.special")
    t = np.array(maxwell.table())
    assert t.shape == (maxwell.CELLS, maxwell.DEGREE + 1)
    cell = np.arange(maxwell.CELLS)
    x0 = np.array([maxwell.centre(int(c)) for c in cell])
    octave = np.floor(np.log2(x0))
    half = 0.5 * 2.0 ** octave / np.where(x0 < maxwell.X_MID, 2.0 ** maxwell.LOW_BITS,
                                          2.0 ** maxwell.HIGH_BITS)
    for s in (-1.0, -0.4, 0.0, 0.7, 1.0):
        x = x0 + s * half
        up = cell >= maxwell.first_upper_cell()
        v = np.where(up, special.gammaincc(1.5, x * x), special.gammainc(1.5, x * x))
        d = (v - t[:, 0]) * t[:, 1]
        p = np.zeros_like(d)
        for k in range(maxwell.DEGREE, 1, -1):
            p = p * d + t[:, k]
        # scipy's distribution is good to a few 1e-15 relative, which moves x by at most
        # v / (x f) <= 1/2 of that
        assert np.abs((x0 + (d + d * d * p)) / x - 1).max() < 1e-14
