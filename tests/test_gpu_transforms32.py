"""FP32 transforms of the mixed-precision step at every compiled length (48,
72, 96, 192, 384) in both directions, against the FP64 step."""
import numpy as np
import pytest

from paper_1705_03838_gb300 import inputs, opf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,M", [(16, 24), (24, 32), (32, 16), (64, 5), (128, 3), (5, 64), (3, 128)])
def test_mixed_step_follows_fp64(K, M):
    N, m_p, alpha, Re, dt = 10, 1, 1.25, 900.0, 0.001
    U0 = inputs.seeded_state(N, K, M, m_p, alpha, 0.2, 70 + K + M, envelope=inputs.envelope_broadband)
    out = []
    for precision in (0, 1):
        h = opf.opf_create(N, K, M, m_p, alpha, Re, dt)
        opf.opf_set_option(h, "precision", precision)
        opf.opf_set_state(h, U0)
        opf.opf_step(h, 1)
        out.append(opf.opf_get_state(h))
    # FP32 rounding of the nonlinear term (a few 2^-24 per transform pass) against the step's change
    assert np.linalg.norm(out[1] - out[0]) <= 1e-5 * np.linalg.norm(out[0] - U0)
