"""The FP64 nonlinear term on grids of many blocks, where the tensor-core
transforms take several row tiles per block (across rows and fields of the
z synthesis) and the forms for more blocks than SMs, against the oracle."""
import numpy as np
import pytest

from oracle.opf_oracle import Oracle, Params
from paper_1705_03838_gb300 import inputs, opf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M", [(80, 16, 16), (81, 10, 12), (161, 5, 3), (60, 32, 24), (78, 20, 18)])
def test_nonlinear_matches_oracle_on_many_blocks(N, K, M):
    alpha, Re = 1.25, 900.0
    U = inputs.seeded_state(N, K, M, 1, alpha, 0.1, 40 * K + M, envelope=inputs.envelope_broadband)
    h = opf.opf_create(N, K, M, 1, alpha, Re, 0.001)
    want = Oracle(Params(N, K, M, 1, alpha, Re, 0.001)).nonlinear(U)
    got = opf.opf_nonlinear(h, U)
    # the wall's derivative weights are of order N^2: their rounding, N^2 eps, on top of the transforms'
    tol = 1e-12 + 4 * N**2 * 2.3e-16
    assert np.abs(got - want).max() <= tol * np.abs(want).max()
    assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
