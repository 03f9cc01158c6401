"""The solve around N = 64, from where its radial derivatives are digit
products: every tile gives the same bits, and a step follows the oracle."""
import numpy as np
import pytest

from oracle.opf_oracle import Oracle, Params
from paper_1705_03838_gb300 import inputs, opf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [63, 64, 65, 71])
def test_step_at_every_tile(N):
    K, M, m_p, alpha, Re, dt = 9, 5, 4, 1.25, 700.0, 0.002  # 17 k: a ragged last tile of each size
    U = inputs.seeded_state(N, K, M, m_p, alpha, 0.05, 700 + N)
    out = []
    for tile in (4, 8, 16):
        h = opf.opf_create(N, K, M, m_p, alpha, Re, dt)
        opf.opf_set_option(h, "spike", 0)
        opf.opf_set_option(h, "tile", tile)
        opf.opf_set_state(h, U)
        opf.opf_step(h, 1)
        out.append(opf.opf_get_state(h))
    ref = Oracle(Params(N, K, M, m_p, alpha, Re, dt)).step(U, 1)
    assert np.linalg.norm(out[0] - ref) <= 1e-10 * np.linalg.norm(ref)
    for got in out[1:]:
        assert np.array_equal(got, out[0])
