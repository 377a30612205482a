"""conv_get_info reports where the FP64 passes' twiddles lie: in shared memory at the compile-time
lengths, in global memory at the others."""
import pytest

from paper_2107_03958_gb300.api import ConvPlan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,period,compact,staged", [(256, 3, True, 1), (1024, 3, True, 1), (64, 3, False, 0),
                                                     (256, 3, False, 0)])
def test_info_says_where_the_twiddles_are(n, period, compact, staged):
    info = ConvPlan("log", n=n, period=period, precision="fp64", compact=compact).info
    assert info.smem_twiddles == staged and (info.static_len > 0) == bool(staged)
