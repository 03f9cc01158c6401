"""The FP64 nonlinear term of a uniform u_r and one mode of u_z, N_z = -u_r
u_z', at the ends of the FP64 range: each row of the transforms has an exponent
of its own, down to the subnormal numbers and up to the largest.  A value that
is not finite spoils its own rows and no others.

Tolerance: 4 N^2 eps of the largest derivative, the rounding of the wall's
weights."""
import numpy as np
import pytest

from paper_1705_03838_gb300 import opf

pytestmark = pytest.mark.gpu

N, K, M, ALPHA = 20, 3, 4, 1.25


def _run(scale, bad=None):
    r = np.cos(np.pi * (N - np.arange(1, N + 1)) / (2 * N - 1))
    r[-1] = 1.0
    h = opf.opf_create(N, K, M, 1, ALPHA, 1000.0, 0.01)
    d1 = opf.opf_setup_query(N, K, M, 1, ALPHA, 1000.0, 0.01, "d1").reshape(2, N, 9)[1]
    col = scale * r * (1 - r * r)
    U = np.zeros((3, M, 2 * K - 1, N), dtype=np.complex128)
    U[0, 0, K - 1] = 1.0
    U[2, 1, K - 1] = col * (1 - 0.5j)
    if bad is not None:
        U[2, 1, K - 1, 12] = bad
    got = opf.opf_nonlinear(h, U)[2, 1, K - 1]
    terms = d1 * (col / scale)[np.clip(np.arange(N) - 4, 0, N - 9)[:, None] + np.arange(9)]
    return got, -terms.sum(1) * (1 - 0.5j)


@pytest.mark.parametrize("scale", [1e-305, 1e-290, 1e-255, 1e-240, 1e-100, 1e263, 1e266, 1e290, 1e303])
def test_scale(scale):
    got, want = _run(scale)
    eps = 2.0**-53 + 2.0**-1074 / scale  # (a unit of the subnormal numbers)
    assert np.isfinite(got).all()
    assert np.abs(got / scale - want).max() <= 4 * N**2 * eps * np.abs(want).max()


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_not_finite(bad):
    got, want = _run(1.0, bad)
    lo = np.clip(np.arange(N) - 4, 0, N - 9)
    reach = (lo <= 12) & (12 <= lo + 8)
    assert not np.isfinite(got[reach]).any()
    assert np.abs(got[~reach] - want[~reach]).max() <= 4 * N**2 * 2.0**-53 * np.abs(want).max()
