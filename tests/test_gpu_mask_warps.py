"""Mask polynomials of which some warps (128 coefficients) and whole CTAs (1024) carry no
output, beside ones that do: ct_out and both shares against the oracle, bit for bit."""
import pytest

from oracle.protocol import FWD, Layer
from tests.test_gpu_linear import check_forward

pytestmark = pytest.mark.gpu


# (h, kernel, Co, partition): 3 x 3 outputs in rows 22 and 46 coefficients apart, the first
# at word 440 and word 2100; one and two channels a polynomial; one output at the last word
@pytest.mark.parametrize("h,s,co,part", [(22, 20, 3, (1, 1, 1, 3, 3, 20, 20)), (22, 20, 3, (1, 1, 2, 3, 3, 20, 20)),
                                         (46, 44, 2, (1, 1, 1, 3, 3, 44, 44)), (64, 64, 1, (1, 1, 1, 1, 1, 64, 64))])
def test_polynomials_with_empty_warps(h, s, co, part):
    from paper_2403_11166_gb300 import he
    check_forward(he, (12, 2, 60), Layer("conv", B=2, Ci=1, Co=co, h=h, w=h, s=s, pad=0), FWD, part, 33, [], [], [0], True)
