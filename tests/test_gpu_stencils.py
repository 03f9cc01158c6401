"""Radial derivatives row by row where columns are steep: r^m~ towards the axis,
(1 - r)^2 at the wall, against extended precision.

The nonlinear term of a uniform u_r (its vorticity is exactly zero) and one
mode of u_z or u_theta is that mode's derivative: N_z = -u_r u_z', N_theta =
-u_r (u_theta' + u_theta / r).  Bound per row, eps the rounding unit: 9 eps S, S the
sum of |weight x value| over the row's stencil (the multiply-adds' a priori
bound), and 32 eps of the result (and of u_theta / r) for the transforms of
one harmonic and 15 points."""
import numpy as np
import pytest

from paper_1705_03838_gb300 import opf

pytestmark = pytest.mark.gpu


def _mesh(N):
    r = np.cos(np.pi * (N - np.arange(1, N + 1)) / (2 * N - 1))
    r[-1] = 1.0
    return r


COLUMNS = {
    "axis": lambda r, mt: r**mt * (1 - r * r) ** 2 * (1 + 0.1 * np.cos(7 * r * r)),
    "wall": lambda r, mt: r ** (mt % 2) * (1 - r) ** 2,
    "axis_tiny": lambda r, mt: 1e-20 * r ** (mt / 2) * (1 - r),
    "jump": lambda r, mt: np.where(np.arange(r.size) % 7 < 3, 1.0, 1e-25) * np.cos(9 * r),
}


# (in mixed precision u_z' is the FP64 one, and what is left of the base flow's
# vorticity, 1e-15, joins its products)
@pytest.mark.parametrize("precision,component", [(0, 2), (0, 1), (1, 1)])
@pytest.mark.parametrize("N", [9, 21, 48, 64, 100])
def test_derivative_of_steep_columns(N, precision, component):
    K, M, alpha, Re = 1, 5, 1.25, 1000.0
    r = _mesh(N)
    rl = r.astype(np.longdouble)
    eps = 2.0**-53 if precision == 0 else 2.0**-24
    for m_p in (10, 11):
        h = opf.opf_create(N, K, M, m_p, alpha, Re, 0.01)
        opf.opf_set_option(h, "precision", precision)
        d1 = opf.opf_setup_query(N, K, M, m_p, alpha, Re, 0.01, "d1").reshape(2, N, 9)
        for m in (1, 2, 4):
            mt = m * m_p
            w = d1[(mt & 1) if component == 2 else (mt & 1) ^ 1].astype(np.longdouble)
            for name, f in COLUMNS.items():
                col = f(r, mt) * (1.0 - 0.7j)
                U = np.zeros((3, M, 2 * K - 1, N), dtype=np.complex128)
                U[0, 0, 0] = 1.0
                if precision == 1:
                    U[2, 0, 0] = 1 - r * r  # (taken off there: the perturbation has no axial mean)
                U[component, m, 0] = col
                got = opf.opf_nonlinear(h, U)[component, m, 0]
                for part in (np.real, np.imag):
                    c = part(col).astype(np.longdouble)
                    lo = np.clip(np.arange(N) - 4, 0, N - 9)
                    terms = w * c[lo[:, None] + np.arange(9)]
                    want, S = -terms.sum(1), np.abs(terms).sum(1)
                    scale = np.abs(want)
                    if component == 1:
                        want = want - c / rl
                        scale = scale + np.abs(c / rl)
                    err = np.abs(part(got).astype(np.longdouble) - want)
                    bound = eps * (9 * S + 32 * scale)
                    rows = np.arange(N)
                    if precision == 1:
                        rows = rows[S[rows] > 1e-27]  # (above FP32's subnormals)
                    worst = (err[rows] / np.where(bound[rows] > 0, bound[rows], 1)).max() if rows.size else 0.0
                    assert worst <= 1.0, (name, mt, part.__name__, int(rows[np.argmax(err[rows] / bound[rows])]), float(worst))
