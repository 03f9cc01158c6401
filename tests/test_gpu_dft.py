"""The FP64 nonlinear term at transform lengths around the tiling of the
tensor-core transforms (harmonics 1..32, points in tiles of 8 and 16, odd
lengths, many m columns) and just past their range, against the oracle."""
import numpy as np
import pytest

from oracle.opf_oracle import Oracle, Params
from paper_1705_03838_gb300 import inputs, opf

pytestmark = pytest.mark.gpu


def _check(N, K, M, m_p, rot, amplitude=0.1):
    alpha, Re = 1.25, 900.0
    U = inputs.seeded_state(N, K, M, m_p, alpha, amplitude, 40 * K + M,
                            envelope=inputs.envelope_broadband)
    h = opf.opf_create(N, K, M, m_p, alpha, Re, 0.001)
    for key, v in zip(("rot_x", "rot_y", "rot_z"), rot):
        opf.opf_set_option(h, key, v)
    want = Oracle(Params(N, K, M, m_p, alpha, Re, 0.001, rotation=rot)).nonlinear(U)
    got = opf.opf_nonlinear(h, U)
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
    assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)


@pytest.mark.parametrize("K,M", [(1, 1), (1, 6), (2, 3), (3, 16), (5, 9), (8, 18), (9, 2), (15, 15), (16, 32),
                                 (18, 20), (25, 24), (27, 5), (32, 16), (30, 40), (36, 8), (32, 32)])
def test_nonlinear_matches_oracle(K, M):
    _check(10 if K * M > 300 else 13, K, M, 1, (0.0, 0.0, 0.0))


@pytest.mark.parametrize("rot,m_p", [((0.3, -0.2, 0.5), 1), ((0.0, 0.0, 0.7), 3)])
def test_rotation(rot, m_p):
    _check(12, 6, 10, m_p, rot)


@pytest.mark.parametrize("amplitude", [1e-120, 1e-8, 1e60])
def test_scales(amplitude):
    """Each row of data has an exponent of its own."""
    _check(12, 5, 8, 1, (0.0, 0.0, 0.0), amplitude)
