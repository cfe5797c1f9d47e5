"""The multiply-accumulate of few input blocks against the per-thread ring kernel:
ct_out bit for bit, at the edges of its row pairs and column strips."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# (M, K, NC): every K, odd and single rows, strips of 8 and (76 rows) of 16 columns with
# remainders and one column
SHAPES = [(1, 1, 1), (2, 2, 8), (3, 3, 9), (5, 4, 7), (7, 5, 16), (4, 6, 33), (77, 1, 16), (76, 2, 17), (79, 6, 31)]


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
@pytest.mark.parametrize("shape", SHAPES)
def test_short_product_matches_ring_kernel(shape, fill):
    from paper_2403_11166_gb300 import he
    m, k, nc = shape
    outs, parts = [], []
    for staging in (0, 1):
        ctx = he.Context(12, 2, 60, 41)
        ctx.tune(he.TUNE_MAC_STAGING, staging)
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
        if m > 1 and staging:   # the same rows in two slices
            part = torch.zeros_like(out)
            for first, count in ((0, 1), (1, m - 1)):
                he.he_linear_forward_apply(ctx, plan.slice(first, count), ct, pt, part, ws)
            parts.append(part)
    assert torch.equal(*outs)
    assert all(torch.equal(outs[0], part) for part in parts)
