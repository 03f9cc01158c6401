"""The bounded waits of the tensor-core GEMM give a warp one verdict: true only
where every lane saw its phase complete, and false, after the limit, on all
lanes where some ran out."""
import ctypes

import pytest

from paper_1705_03838_gb300 import opf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("done_lanes", [0, 1, 16, 31, 32])
def test_verdict_is_the_same_on_every_lane(done_lanes):
    verdict = (ctypes.c_int * 32)(*([-1] * 32))
    assert opf.lib().opf_test_wait_verdict(done_lanes, verdict) == 0
    assert list(verdict) == [int(done_lanes == 32)] * 32
