"""The digit-product multiply-accumulate (tensor cores) against the integer
kernels: ct_out bit for bit, at the edges of its tiles and chunks."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# (log2 N, primes, prime bits, knobs of the integer form: MAC columns, MAC staging)
RINGS = {"60-bit": (12, 2, 60, 4, 0), "54-bit": (12, 2, 54, 0, 1)}
# (M, K, NC): part and whole tiles of 4 / 8 / 16 rows and 16 columns, chunks of 4 / 8 /
# 12 / 16 input blocks and their remainders, more than eight chunks (a lazy sum folded)
SHAPES = [(4, 16, 16), (5, 9, 16), (8, 13, 17), (9, 16, 33), (16, 17, 16), (17, 33, 31), (12, 147, 16), (3, 43, 64),
          (10, 20, 32), (16, 12, 16)]


def _ctx(name):
    from paper_2403_11166_gb300 import he
    log_n, limbs, bits, cols, staging = RINGS[name]
    plain, mma = he.Context(log_n, limbs, bits, 41), he.Context(log_n, limbs, bits, 41)
    plain.tune(he.TUNE_MAC_COLUMNS, cols)
    plain.tune(he.TUNE_MAC_STAGING, staging)
    return plain, mma


def _residues(ctx, shape, fill, seed):
    """[..., L, N] canonical words: uniform, or the largest residue everywhere."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.empty(shape, dtype=torch.int64, device="cuda")
    for j, q in enumerate(ctx.primes()[0]):
        t[..., j, :] = q - 1 if fill == "max" else torch.randint(0, q, t[..., j, :].shape, generator=g, device="cuda",
                                                                 dtype=torch.int64)
    return t


@pytest.mark.parametrize("fill", ["uniform", "max"])
@pytest.mark.parametrize("ring", list(RINGS))
@pytest.mark.parametrize("shape", SHAPES)
def test_forward_product_matches_integer_kernels(ring, shape, fill):
    from paper_2403_11166_gb300 import he
    m, k, nc = shape
    outs = []
    for ctx in _ctx(ring):
        plan = he.Plan(ctx, he.Layer(he.FC, m, k, nc), he.ROLE_FWD, (1, 1, 1, 1, 1, 1, 1))
        s = plan.sizes
        assert (s.ct_in, s.pt, s.ct_out) == (m * k, k * nc, m * nc)
        ct = _residues(ctx, (s.ct_in, 2, ctx.L, ctx.n), fill, 1)
        pt = _residues(ctx, (s.pt, ctx.L, ctx.n), fill, 2)
        x0 = torch.full((m, k), (1 << 41) - 1, dtype=torch.int64, device="cuda")
        out, ws = plan.new_ct(s.ct_out), plan.new_ws(s.ws_forward)
        y0 = torch.empty(s.out_elems, dtype=torch.int64, device="cuda")
        he.he_linear_forward(ctx, plan, ct, pt, x0, None, 7, out, y0, ws)
        outs.append(out)
    assert torch.equal(*outs)


@pytest.mark.parametrize("fill", ["uniform", "max"])
@pytest.mark.parametrize("ring", list(RINGS))
@pytest.mark.parametrize("shape", [(8, 8, 16), (9, 5, 17), (17, 20, 31), (8, 77, 16), (3, 12, 33)])
def test_weight_gradient_product_matches_integer_kernels(ring, shape, fill):
    from paper_2403_11166_gb300 import he
    m, k, nc = shape
    outs = []
    for ctx in _ctx(ring):
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
        outs.append(out)
    assert torch.equal(*outs)


def test_row_slices_match_the_whole_product():
    from paper_2403_11166_gb300 import he
    ctx = he.Context(12, 2, 60, 41)
    plan = he.Plan(ctx, he.Layer(he.FC, 21, 18, 19), he.ROLE_FWD, (1, 1, 1, 1, 1, 1, 1))
    s = plan.sizes
    ct, pt = _residues(ctx, (s.ct_in, 2, ctx.L, ctx.n), "uniform", 5), _residues(ctx, (s.pt, ctx.L, ctx.n), "uniform", 6)
    x0 = torch.arange(21 * 18, dtype=torch.int64, device="cuda").view(21, 18)
    ws, y0 = plan.new_ws(s.ws_forward), torch.empty(s.out_elems, dtype=torch.int64, device="cuda")
    whole, parts = plan.new_ct(s.ct_out), plan.new_ct(s.ct_out)
    he.he_linear_forward(ctx, plan, ct, pt, x0, None, 7, whole, y0, ws)
    for first, count in ((0, 9), (9, 1), (10, 11)):
        he.he_linear_forward_apply(ctx, plan.slice(first, count), ct, pt, parts, ws)
    assert torch.equal(whole, parts)
