"""The small kernels' vector, cluster and alignment branches, exactly."""
import numpy as np
import pytest
import torch

from tests.gpu_util import as_u64, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def he():
    from paper_2403_11166_gb300 import he
    return he


# B HW at and above the size that is split over a cluster; ragged parts; the most
# channels (the y extent of the grid)
@pytest.mark.parametrize("layer", [("fc", 4096, 1, 3), ("fc", 4097, 1, 3), ("fc", 5, 1, 1), ("fc", 1, 1, 65535),
                                   ("conv", 63, 1, 5, 8, 9, 1, 0), ("conv", 1, 1, 1, 65, 64, 1, 0),
                                   ("conv", 3, 2, 17, 37, 37, 1, 0)])
def test_bias_grad_parts(he, layer):
    kind, b, ci, co, *rest = layer
    h, w = rest[:2] if rest else (1, 1)
    ctx = he.Context(12, 1, 60, 41)
    plan = he.Plan(ctx, he.Layer(he.FC if kind == "fc" else he.CONV, b, ci, co, h, w, 1, 0), he.ROLE_FWD)
    g = np.random.default_rng(1).integers(0, 1 << 41, (b, co, h * w), dtype=np.uint64)
    out = torch.empty(co, dtype=torch.int64, device="cuda")
    he.pencil_bias_grad(ctx, plan, to_dev(g), out)
    assert (to_np(out) == g.sum(axis=(0, 2), dtype=np.uint64) & np.uint64((1 << 41) - 1)).all()


# two elements per thread against one: a shift of the source, the output or the addend by
# one word, an odd offset, an odd count, inner extent or stride
@pytest.mark.parametrize("shift", [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)])
@pytest.mark.parametrize("count,inner,outer,tstride,off", [(64, 16, 40, 200, 2), (2, 2, 0, 64, 0), (1030, 1030, 0, 1100, 0),
                                                           (63, 21, 40, 200, 2), (64, 16, 41, 200, 2),
                                                           (64, 16, 40, 201, 2), (64, 16, 40, 200, 3)])
@pytest.mark.parametrize("terms", [1, 7, 9])
def test_lincomb_pairs(he, shift, count, inner, outer, tstride, off, terms):
    ctx = he.Context(12, 1, 60, 41)
    r = np.random.default_rng(count + terms)
    size = off + (count // inner) * outer + inner + (terms - 1) * tstride + 8
    buf = r.integers(0, 1 << 63, (3, max(size, count) + 2), dtype=np.uint64)
    k = [int(v) for v in r.integers(0, 1 << 63, terms, dtype=np.uint64)]
    dev = [to_dev(row.copy()) for row in buf]
    src, out, add = (t[s:] for t, s in zip(dev, shift))
    he.pencil_lincomb(ctx, src, k, count, out, addend=add, negate=True, src_offset=off, inner=inner,
                      outer_stride=outer, term_stride=tstride)
    e = np.arange(count)
    at = shift[0] + off + (e // inner) * outer + e % inner
    with np.errstate(over="ignore"):
        want = buf[2][shift[2]:shift[2] + count] - sum(np.uint64(k[i]) * buf[0][at + i * tstride] for i in range(terms))
    assert (to_np(out[:count]) == (want & np.uint64((1 << 41) - 1))).all()
    assert (to_np(out[count:]) == buf[1][shift[1] + count:]).all()   # nothing past the result


@pytest.mark.parametrize("layer", [("fc", 3, 2, 7), ("fc", 1, 1, 1), ("conv", 2, 1, 3, 5, 5, 3, 1)])
def test_share_store_at_odd_addresses(he, layer):
    kind, b, ci, co, *rest = layer
    ctx = he.Context(12, 2, 60, 41)
    plan = he.Plan(ctx, he.Layer(he.FC if kind == "fc" else he.CONV, b, ci, co, *rest), he.ROLE_FWD)
    s = plan.sizes
    x0 = torch.zeros(b * ci * (rest[0] * rest[1] if rest else 1), dtype=torch.int64, device="cuda")
    bias = torch.arange(1, co + 1, dtype=torch.int64, device="cuda")
    ws = plan.new_ws(s.ws_forward)
    got = []
    for shift in (0, 1):
        y0 = torch.full((s.out_elems + 8,), -5, dtype=torch.int64, device="cuda")
        he.he_linear_forward_prepare(ctx, plan, x0, bias, 9, y0[shift:], ws)
        assert (y0[:shift] == -5).all() and (y0[shift + s.out_elems:] == -5).all()
        got.append(y0[shift:shift + s.out_elems].clone())
    assert torch.equal(*got)
