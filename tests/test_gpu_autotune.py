"""Autotuned launch shapes against the default ones in mixed precision, bit
for bit, at the theta lengths whose product takes a compiled plan and on grids
where its blocks are small: the tuner tries up to 16 rows per block, more than
a block has threads for at once."""
import ctypes

import numpy as np
import pytest

from paper_1705_03838_gb300 import inputs, opf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M", [(60, 32, 16), (128, 32, 24), (128, 32, 32), (128, 32, 64), (10, 9, 128),
                                   (110, 32, 20)])
def test_every_shape(N, K, M):
    """Each candidate of the tuner in turn, on few and on many blocks."""
    alpha, Re, dt = 1.25, 900.0, 0.001
    U0 = inputs.seeded_state(N, K, M, 1, alpha, 0.2, 60 + K + M, envelope=inputs.envelope_broadband)
    h = opf.opf_create(N, K, M, 1, alpha, Re, dt)
    opf.opf_set_option(h, "precision", 1)

    def step():
        opf.opf_set_state(h, U0)
        opf.opf_step(h, 1)
        return opf.opf_get_state(h)

    want, taken = step(), 0
    assert np.isfinite(want).all()
    for c in (1, 2, 4, 8, 16):
        for mcz, zc, mca in ((c, 4, 4), (4, c, 4), (4, 4, c)):
            if opf.lib().opf_test_launch_shape(ctypes.c_void_p(h.ptr), mcz, zc, mca) == 0:
                taken += 1
                assert np.array_equal(step(), want), (mcz, zc, mca)
    assert taken >= 12


@pytest.mark.parametrize("N,K,M", [(10, 3, 128), (24, 10, 128), (40, 6, 64)])
def test_single(N, K, M):
    alpha, Re, dt = 1.25, 900.0, 0.001
    U0 = inputs.seeded_state(N, K, M, 1, alpha, 0.2, 60 + K + M, envelope=inputs.envelope_broadband)
    out = []
    for tune in (0, 1):
        h = opf.opf_create(N, K, M, 1, alpha, Re, dt)
        opf.opf_set_option(h, "precision", 1)
        opf.opf_set_option(h, "autotune", tune)
        opf.opf_set_state(h, U0)
        opf.opf_step(h, 2)
        out.append(opf.opf_get_state(h))
    assert np.array_equal(*out)


@pytest.mark.parametrize("M", [24, 32, 64, 128])
def test_ensemble_of_many_blocks(M):
    N, K, alpha, dt, copies = 16, 6, 1.25, 0.001, 24  # 18 z rows: 2 x 16 x 24 blocks of 16 rows
    U0 = [inputs.seeded_state(N, K, M, 1, alpha, 0.2, 600 + i, envelope=inputs.envelope_broadband)
          for i in range(copies)]
    out = []
    for tune in (0, 1):
        e = opf.opf_ens_create(*([v] * copies for v in (N, K, M, 1, alpha, 900.0, dt)))
        opf.opf_ens_set_option(e, "precision", 1)
        opf.opf_ens_set_option(e, "autotune", tune)
        for i, U in enumerate(U0):
            opf.opf_ens_set_state(e, i, U)
        opf.opf_ens_step(e, 2)
        out.append([opf.opf_ens_get_state(e, i) for i in range(copies)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
