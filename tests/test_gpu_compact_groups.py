"""compact_returned where a warp's groups of 32 coefficients are empty, half empty or full:
every engine, radix and N.  The compact form is the inverse transform of c0 at the
coefficients that carry outputs (one by one through pencil_ntt_batch), and decrypts to the
same share."""
import pytest
import torch

pytestmark = pytest.mark.gpu

RINGS = [(12, 2, 60, 4, 1), (12, 2, 50, 4, 0), (13, 2, 60, 4, 1), (13, 2, 60, 5, 1), (13, 2, 60, 4, 0), (14, 2, 60, 4, 1),
         (14, 2, 60, 5, 1), (14, 2, 50, 5, 0)]
# (B, Ci, Co, H, kernel, pad), role, partition: 3 x 3 outputs a channel 400 words on; full rows; every 40th coefficient
LAYERS = [((1, 2, 3, 20, 18, 0), 0, (1, 1, 1, 3, 3, 18, 18)), ((2, 1, 2, 30, 1, 0), 0, (2, 1, 1, 30, 30, 1, 1)),
          ((60, 40, 2, 1, 1, 0), 0, (30, 40, 2, 1, 1, 1, 1)), ((1, 1, 1, 1, 1, 0), 0, (1, 1, 1, 1, 1, 1, 1))]


@pytest.mark.parametrize("copies", [1, 150])   # one CTA each, and few enough for a cluster each
@pytest.mark.parametrize("layer,role,part", LAYERS)
@pytest.mark.parametrize("log_n,limbs,bits,radix,arith", RINGS)
def test_compact_form_is_the_output_coefficients(log_n, limbs, bits, radix, arith, layer, role, part, copies):
    from paper_2403_11166_gb300 import he
    b, ci, co, h, k, pad = layer
    b, part = b * copies, tuple(part)
    ctx = he.Context(log_n, limbs, bits, 20)
    ctx.tune(he.TUNE_NTT_LOG_RADIX, radix)
    if bits == 60:
        ctx.tune(he.TUNE_NTT_ARITH, arith)
    sk = ctx.keygen(3)
    plan = he.Plan(ctx, he.Layer(he.FC if (h, k) == (1, 1) else he.CONV, b, ci, co, h, h, k, pad), role, part)
    s = plan.sizes
    g = torch.Generator(device="cuda").manual_seed(5)
    ct = plan.new_ct(s.ct_out)
    words = ct.view(s.ct_out, 2, limbs, ctx.n)
    for j, q in enumerate(ctx.primes()[0]):
        words[:, :, j] = torch.randint(0, q, words[:, :, j].shape, generator=g, device="cuda", dtype=torch.int64)
    c0c = torch.full((limbs, s.out_elems), -1, dtype=torch.int64, device="cuda")
    he.compact_returned(ctx, plan, ct, c0c)
    coeff = words[:, 0].clone()
    he.pencil_ntt_batch(ctx, coeff, inverse=True)
    # every output is one coefficient of its polynomial: the same words, each as often
    assert (c0c >= 0).all()
    for j in range(limbs):
        row, _ = torch.sort(coeff[:, j].reshape(-1))
        at = torch.searchsorted(row, c0c[j].contiguous())
        assert torch.equal(row[at.clamp(max=row.numel() - 1)], c0c[j])
        assert torch.unique(c0c[j]).numel() == s.out_elems   # (uniform residues: no two alike)
    ws, y, z = plan.new_ws(s.ws_decrypt), *(torch.empty(s.out_elems, dtype=torch.int64, device="cuda") for _ in range(2))
    ws.fill_(-1)   # (residues of empty groups are not written, and not read)
    he.decrypt_to_share(ctx, sk, plan, ct, y, False, ws)
    ws.fill_(7)
    he.decrypt_compact_to_share(ctx, sk, plan, ct, c0c, z, False, ws)
    assert torch.equal(y, z)
