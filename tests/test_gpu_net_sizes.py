"""Network passes at sizes around the GEMM tiles and the vector widths of the
kernels that lay the operands out: one point, one sample, odd channel counts,
just past a tile of 64 channels and 128 rows, against the FP64 oracle network.

Tolerance: as for the network's other parity tests, BF16 factors of relative
error 4e-3 over three layers, held to 3e-2 in relative L2."""
import numpy as np
import pytest

from oracle import net_oracle as nn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,hidden,L,B,nout", [(24, 16, 1, 5, 1), (33, 47, 2, 9, 1), (65, 129, 43, 3, 3),
                                                 (72, 64, 32, 4, 5), (200, 66, 13, 20, 2)])
def test_passes_match_oracle(cin, hidden, L, B, nout):
    torch = pytest.importorskip("torch")
    from paper_1705_03838_gb300 import opf

    rel = lambda a, b: np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b))
    rng = np.random.default_rng(cin + hidden)
    net = opf.opf_net_create(cin, hidden, L, nout, seed=3)
    p = nn.split(opf.opf_net_get_params(net).astype(np.float64), cin, hidden, nout)
    for k in ("b1", "b2", "b3", "bh"):
        p[k] = rng.normal(size=p[k].shape) * 0.1
    flat = nn.flatten(p).astype(np.float32)
    opf.opf_net_set_params(net, flat)
    assert np.array_equal(opf.opf_net_get_params(net), flat)
    p = nn.split(flat.astype(np.float64), cin, hidden, nout)
    for batch in (B, 1, B):  # buffers sized for the larger batch serve the smaller
        x = rng.normal(size=(batch, L, cin)).astype(np.float32)
        ty = rng.normal(size=(batch, L, cin)).astype(np.float32) * 0.5
        tz = rng.normal(size=(batch, nout)).astype(np.float32)
        dx, dty, dtz = (torch.from_numpy(a).cuda() for a in (x, ty, tz))
        loss_ref, g_ref, y_ref, z_ref = nn.loss_and_grads(p, x.astype(np.float64), ty, tz, 0.5)
        loss = opf.opf_net_gradients(net, dx.data_ptr(), dty.data_ptr(), dtz.data_ptr(), batch, 0.5)
        g = nn.split(opf.opf_net_get_params(net, grads=True).astype(np.float64), cin, hidden, nout)
        dy, dz = torch.empty_like(dx), torch.empty_like(dtz)
        opf.opf_net_forward(net, dx.data_ptr(), batch, dy.data_ptr(), dz.data_ptr())
        assert abs(loss - loss_ref) <= 3e-2 * loss_ref
        assert rel(dy.cpu().numpy(), y_ref) < 3e-2
        assert rel(dz.cpu().numpy(), z_ref) < 3e-2
        for k in nn.NAMES:
            assert rel(g[k], g_ref[k]) < 3e-2, k
