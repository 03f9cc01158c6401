"""The solve's tiles (4, 8 and 16 modes, and the 4-mode form that takes the
curl of its new state on a grid of a block per SM) go through the same
arithmetic per mode: equal bit for bit."""
import numpy as np
import pytest

from paper_1705_03838_gb300 import inputs, opf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [9, 16, 20, 23, 33, 48])
@pytest.mark.parametrize("precision", [0, 1])
def test_tiles_and_batches_agree_bit_for_bit(N, precision):
    K, M, m_p, alpha, Re, dt, copies = 9, 5, 2, 1.25, 700.0, 0.005, 8  # 17 k: a ragged last tile of each size
    U0 = inputs.seeded_state(N, K, M, m_p, alpha, 0.05, 4100 + N)

    def single(tile):
        h = opf.opf_create(N, K, M, m_p, alpha, Re, dt)
        opf.opf_set_option(h, "precision", precision)
        opf.opf_set_option(h, "spike", 0)
        opf.opf_set_option(h, "tile", tile)
        opf.opf_set_state(h, U0)
        opf.opf_step(h, 3)
        return opf.opf_get_state(h)

    want = single(4)
    assert np.isfinite(want).all()
    for tile in (8, 16):
        assert np.array_equal(single(tile), want)
    e = opf.opf_ens_create(*([v] * copies for v in (N, K, M, m_p, alpha, Re, dt)))
    opf.opf_ens_set_option(e, "precision", precision)
    opf.opf_ens_set_option(e, "spike", 0)
    for i in range(copies):
        opf.opf_ens_set_state(e, i, U0)
    opf.opf_ens_step(e, 3)
    for i in (0, copies - 1):
        assert np.array_equal(opf.opf_ens_get_state(e, i), want)
