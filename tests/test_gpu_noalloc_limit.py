"""The radial limit of opf_nonlinear_noalloc does not depend on the calls made
before: with 3 x 2 modes, three columns per block, N up to 1263 is accepted."""
import pytest

from paper_1705_03838_gb300 import opf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", [1264, 16])
def test_limit_after_any_first_call(first):
    torch = pytest.importorskip("torch")
    K, M, alpha, Re = 2, 2, 1.0, 500.0

    def call(N):
        d_in = torch.zeros(3 * M * (2 * K - 1) * N * 2, dtype=torch.float64, device="cuda")
        d_out = torch.empty_like(d_in)
        torch.cuda.synchronize()
        opf.opf_nonlinear_noalloc(N, K, M, 1, alpha, Re, d_in.data_ptr(), d_out.data_ptr())
        assert torch.isfinite(d_out).all()

    for N in (first, 16, 1264, 1263, 1264):
        if N > 1263:
            with pytest.raises(opf.OpfError) as e:
                call(N)
            assert e.value.code == opf.OPF_EINVAL and "shared memory" in str(e.value)
        else:
            call(N)
