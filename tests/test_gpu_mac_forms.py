"""Every form of the multiply-accumulate (digit products, bulk copies, few input blocks,
per-thread ring, shared-memory staged, generic) at sizes that take it, asserted with the
library's own rule, against the per-thread ring kernel (60-bit primes) or the generic one
(54-bit): ct_out bit for bit."""
import pytest
import torch

from tests import rules_lib

pytestmark = pytest.mark.gpu

# digit products, both primes: every remainder class of a chunk of 16 input blocks (1 .. 4, 5 .. 8, 9 .. 12,
# 13 .. 16) alone and behind a full chunk, part rows of tiles of 4, 8 and 16, part columns of 16
FORWARD = [(16, 7, 16), (24, 8, 32), (8, 9, 16), (24, 11, 32), (12, 13, 48), (40, 13, 33), (28, 15, 61), (40, 16, 33),
           (16, 20, 16), (20, 21, 16), (21, 22, 32), (41, 24, 49), (16, 25, 16), (16, 28, 32), (19, 29, 16)]
# chunks of 8: remainders 1 .. 4 and 5 .. 8, alone and behind full ones
DUAL = [(32, 3, 32), (16, 5, 16), (24, 6, 17), (33, 9, 48), (16, 12, 32), (40, 12, 33), (17, 13, 47)]
BULK = [(5, 9, 7), (2, 7, 5), (3, 13, 9), (1, 8, 1), (5, 20, 2)]
BULK_DUAL = [(3, 2, 5), (2, 5, 3), (1, 1, 1), (5, 7, 2)]


def _residues(ctx, shape, fill, seed):
    """[..., L, N] canonical words: uniform, or the largest residue everywhere."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.empty(shape, dtype=torch.int64, device="cuda")
    for j, q in enumerate(ctx.primes()[0]):
        t[..., j, :] = q - 1 if fill == "max" else torch.randint(0, q, t[..., j, :].shape, generator=g, device="cuda",
                                                                 dtype=torch.int64)
    return t


def _ctx(bits, columns, staging):
    from paper_2403_11166_gb300 import he
    ctx = he.Context(12, 2, bits, 41)
    ctx.tune(he.TUNE_MAC_COLUMNS, columns)
    ctx.tune(he.TUNE_MAC_STAGING, staging)
    return ctx


def _forward(ctx, m, k, nc, fill, slices=()):
    from paper_2403_11166_gb300 import he
    plan = he.Plan(ctx, he.Layer(he.FC, m, k, nc), he.ROLE_FWD, (1, 1, 1, 1, 1, 1, 1))
    s = plan.sizes
    assert (s.ct_in, s.pt, s.ct_out) == (m * k, k * nc, m * nc)
    ct = _residues(ctx, (s.ct_in, 2, ctx.L, ctx.n), fill, 1)
    pt = _residues(ctx, (s.pt, ctx.L, ctx.n), fill, 2)
    x0 = torch.full((m, k), (1 << 41) - 1, dtype=torch.int64, device="cuda")
    out, ws = plan.new_ct(s.ct_out), plan.new_ws(s.ws_forward)
    y0 = torch.empty(s.out_elems, dtype=torch.int64, device="cuda")
    he.he_linear_forward(ctx, plan, ct, pt, x0, None, 7, out, y0, ws)
    parts = torch.zeros_like(out)
    for first, count in slices:
        he.he_linear_forward_apply(ctx, plan.slice(first, count), ct, pt, parts, ws)
    return out, parts


def _dual(ctx, m, k, nc, fill):
    from paper_2403_11166_gb300 import he
    plan = he.Plan(ctx, he.Layer(he.FC, k, m, nc), he.ROLE_WGRAD, (1, 1, 1, 1, 1, 1, 1))
    s = plan.sizes
    assert (s.ct_in, s.pt, s.ct_out) == (m * k, k * nc, m * nc)
    ct_x = _residues(ctx, (s.ct_in, 2, ctx.L, ctx.n), fill, 3)
    ct_g = _residues(ctx, (s.pt, 2, ctx.L, ctx.n), fill, 4)
    x0 = torch.full((k, m), 1 << 40, dtype=torch.int64, device="cuda")
    g0 = torch.full((k, nc), (1 << 40) + 12345, dtype=torch.int64, device="cuda")
    out, ws = plan.new_ct(s.ct_out), plan.new_ws(s.ws_backward)
    mask = torch.empty(s.out_elems, dtype=torch.int64, device="cuda")
    he.he_linear_backward(ctx, None, plan, None, None, ct_x, ct_g, g0, x0, 0, 9, None, None, out, mask, ws)
    return out


def _plain(bits):
    """(columns, staging, form) of the integer kernel compared with."""
    return (4, 0, "ring") if bits == 60 else (0, 1, "generic")


def _check_form(want, m, k, nc, dual, bits, columns, staging):
    assert rules_lib.mac_form(m, k, nc, dual, bits == 60, columns, staging) == want


@pytest.mark.parametrize("fill", ["uniform", "max"])
@pytest.mark.parametrize("bits", [60, 54])
@pytest.mark.parametrize("shape", FORWARD)
def test_digit_products_forward(shape, bits, fill):
    columns, staging, form = _plain(bits)
    _check_form("digits", *shape, False, bits, 4, 1)
    _check_form(form, *shape, False, bits, columns, staging)
    got, _ = _forward(_ctx(bits, 4, 1), *shape, fill)
    want, _ = _forward(_ctx(bits, columns, staging), *shape, fill)
    assert torch.equal(got, want)


@pytest.mark.parametrize("fill", ["uniform", "max"])
@pytest.mark.parametrize("bits", [60, 54])
@pytest.mark.parametrize("shape", DUAL)
def test_digit_products_weight_gradient(shape, bits, fill):
    columns, staging, form = _plain(bits)
    _check_form("digits", *shape, True, bits, 4, 1)
    _check_form(form, *shape, True, bits, columns, staging)
    assert torch.equal(_dual(_ctx(bits, 4, 1), *shape, fill), _dual(_ctx(bits, columns, staging), *shape, fill))


@pytest.mark.parametrize("bits", [60, 54])
@pytest.mark.parametrize("shape,slices", [((43, 24, 47), ((0, 16), (16, 8), (24, 19))), ((40, 13, 32), ((0, 24), (24, 16))),
                                          ((28, 16, 48), ((0, 4), (4, 12), (16, 12)))])
def test_digit_products_of_row_slices(shape, slices, bits):
    for _, count in slices:
        _check_form("digits", count, *shape[1:], False, bits, 4, 1)
    whole, parts = _forward(_ctx(bits, 4, 1), *shape, "uniform", slices)
    assert torch.equal(whole, parts)
    columns, staging, _ = _plain(bits)
    assert torch.equal(whole, _forward(_ctx(bits, columns, staging), *shape, "uniform")[0])


@pytest.mark.parametrize("shape", BULK)
@pytest.mark.parametrize("columns", [2, 4, 8])
def test_bulk_copies_forward(shape, columns):
    _check_form("bulk", *shape, False, 60, columns, 1)
    _check_form("ring", *shape, False, 60, columns, 0)
    _check_form("smem", *shape, False, 60, 0, 1)
    got, _ = _forward(_ctx(60, columns, 1), *shape, "uniform")
    for other in ((columns, 0), (0, 1)):
        assert torch.equal(got, _forward(_ctx(60, *other), *shape, "uniform")[0])


@pytest.mark.parametrize("shape", BULK_DUAL)
@pytest.mark.parametrize("columns", [2, 4, 8])
def test_bulk_copies_weight_gradient(shape, columns):
    _check_form("bulk", *shape, True, 60, columns, 1)
    got = _dual(_ctx(60, columns, 1), *shape, "uniform")
    for other in ((columns, 0), (0, 1)):
        assert torch.equal(got, _dual(_ctx(60, *other), *shape, "uniform"))


@pytest.mark.parametrize("columns", [2, 4, 8])
def test_bulk_copies_prepare_apply(columns):
    """A ragged convolution of seven input blocks: prepare and apply, on two streams, give the
    whole call's ciphertexts, and the shared-memory staged kernel's."""
    from paper_2403_11166_gb300 import he
    outs = []
    for cols, staging in ((columns, 1), (0, 1)):
        ctx = he.Context(13, 3, 60)
        ctx.tune(he.TUNE_MAC_COLUMNS, cols)
        ctx.tune(he.TUNE_MAC_STAGING, staging)
        plan = he.Plan(ctx, he.Layer(he.CONV, 1, 7, 7, 9, 8, 3, 1), he.ROLE_FWD, (1, 1, 3, 5, 4, 3, 3))
        s = plan.sizes
        m, nc = plan.rows, s.pt // 7
        assert s.ct_in == m * 7
        _check_form("bulk" if cols else "smem", m, 7, nc, False, 60, cols, staging)
        ct = _residues(ctx, (s.ct_in, 2, ctx.L, ctx.n), "uniform", 5)
        pt = _residues(ctx, (s.pt, ctx.L, ctx.n), "uniform", 6)
        x0 = torch.arange(7 * 72, dtype=torch.int64, device="cuda")
        whole, parts = plan.new_ct(s.ct_out), plan.new_ct(s.ct_out)
        y0 = torch.empty(s.out_elems, dtype=torch.int64, device="cuda")
        ws, ws2 = plan.new_ws(s.ws_forward), plan.new_ws(s.ws_forward)
        he.he_linear_forward(ctx, plan, ct, pt, x0, None, 4, whole, y0, ws)
        torch.cuda.synchronize()
        a, b = torch.cuda.Stream(), torch.cuda.Stream()
        he.he_linear_forward_prepare(ctx, plan, x0, None, 4, y0, ws2, stream=a)
        b.wait_stream(a)
        he.he_linear_forward_apply(ctx, plan, ct, pt, parts, ws2, stream=b)
        torch.cuda.synchronize()
        assert torch.equal(whole, parts)
        outs.append(whole)
    assert torch.equal(*outs)
