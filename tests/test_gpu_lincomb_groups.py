"""Linear combinations: every remainder of the groups of terms (8, 4, 2, 1), one and two
elements a thread at the size where the rule changes and past it, exactly."""
import numpy as np
import pytest

from tests import rules_lib
from tests.gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu
MASK = np.uint64((1 << 41) - 1)


@pytest.mark.parametrize("count,pairs", [(1000, False), ((1 << 17) - 2, False), (1 << 17, True), ((1 << 20) + 6, True)])
@pytest.mark.parametrize("terms,terms2", [(0, 1), (1, 1), (2, 1), (3, 1), (4, 1), (5, 2), (7, 1), (8, 1), (13, 2), (15, 4),
                                          (64, 1)])
def test_groups_of_terms(count, pairs, terms, terms2):
    from paper_2403_11166_gb300 import he
    assert rules_lib.lincomb_pairs(count) is pairs
    ctx = he.Context(12, 1, 60, 41)
    r = np.random.default_rng(count + 100 * terms + terms2)
    inner, outer, ts, ts2, off = count // 2, count // 2 + 10, 2, 40, 6
    size = off + 2 * outer + terms * ts + terms2 * ts2 + 8
    src = r.integers(0, 1 << 63, size, dtype=np.uint64)
    add = r.integers(0, 1 << 63, count, dtype=np.uint64)
    k = [int(v) for v in r.integers(0, 1 << 63, max(1, terms * terms2), dtype=np.uint64)][:terms * terms2]
    out = to_dev(np.full(count + 2, 7, dtype=np.uint64))
    he.pencil_lincomb2(ctx, to_dev(src), k, terms, terms2, count, out, addend=to_dev(add), src_offset=off, inner=inner,
                       outer_stride=outer, term_stride=ts, term_stride2=ts2)
    e = np.arange(count)
    at = off + (e // inner) * outer + e % inner
    want = add.copy()
    with np.errstate(over="ignore"):
        for i2 in range(terms2):
            for i in range(terms):
                want += np.uint64(k[i2 * terms + i]) * src[at + i * ts + i2 * ts2]
    got = to_np(out)
    assert (got[:count] == (want & MASK)).all()
    assert (got[count:] == 7).all()   # nothing past the result
