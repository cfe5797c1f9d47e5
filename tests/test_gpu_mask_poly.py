"""Mask polynomials of outputs at every stride: ct_out (the mask's element words and its
padding words) and both shares against the oracle, bit for bit."""
import pytest

from oracle.protocol import FWD, Layer
from tests.test_gpu_linear import check_forward

pytestmark = pytest.mark.gpu


# (B, Ci, Co, partition (bb, cib, cob)) at N = 4096: one output channel per polynomial puts
# neighbouring elements into different blocks of the stream, cib - 1 coefficients of padding
# between them: 1024, 768, 597, 512 and 461 different blocks per 1024 coefficients; then runs
# of 2, 3, 5 and 7 elements with gaps of 0 and 1, and one output alone
@pytest.mark.parametrize("shape", [(1100, 1, 5, (1100, 1, 1)), (1030, 2, 5, (1030, 2, 1)), (700, 3, 5, (700, 3, 1)),
                                   (520, 4, 5, (520, 4, 1)), (500, 5, 3, (500, 5, 1)), (600, 1, 7, (600, 1, 2)),
                                   (300, 1, 3, (300, 1, 3)), (300, 2, 5, (300, 2, 5)), (300, 1, 7, (300, 1, 7)),
                                   (1, 8, 1, (1, 8, 1))])
def test_mask_words_match_oracle(shape):
    from paper_2403_11166_gb300 import he
    b, ci, co, (bb, cib, cob) = shape
    check_forward(he, (12, 2, 60), Layer("fc", b, ci, co), FWD, (bb, cib, cob, 1, 1, 1, 1), 31, [], [], [0], True)
