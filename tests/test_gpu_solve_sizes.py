"""One time step at radial sizes around the substitution's blocking (rounds of
16 columns counted back from the nine wall columns, and both halves of the
split solve) against the oracle."""
import numpy as np
import pytest

from oracle.opf_oracle import Oracle, Params
from paper_1705_03838_gb300 import inputs, opf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,split", [(9, 0), (10, 0), (12, 0), (24, 0), (25, 0), (26, 0), (26, 1), (28, 1), (33, 0),
                                     (41, 0), (42, 0), (50, 1)])
def test_step_matches_oracle_at_every_alignment(N, split):
    K, M, m_p, alpha, Re, dt = 3, 4, 1, 1.25, 300.0, 0.005
    U = inputs.seeded_state(N, K, M, m_p, alpha, 0.05, 9100 + N)
    h = opf.opf_create(N, K, M, m_p, alpha, Re, dt)
    opf.opf_set_option(h, "spike", split)
    assert opf.opf_get_option(h, "spike") == split
    opf.opf_set_state(h, U)
    opf.opf_step(h, 1)
    ref = Oracle(Params(N, K, M, m_p, alpha, Re, dt)).step(U, 1)
    got = opf.opf_get_state(h)
    assert np.linalg.norm(got - ref) <= 1e-10 * np.linalg.norm(ref)
