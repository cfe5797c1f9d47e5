"""Small launches, whose transforms run on clusters of four CTAs each, against the same
work as ordinary launches (radix 2^5 selects those): ciphertexts, plaintexts and shares
bit for bit at every size, both prime families, and raw transforms against the same
polynomials inside a large batch."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _ctxs(log_n, limbs, bits, t_bits=41):
    from paper_2403_11166_gb300 import he
    quad, plain = he.Context(log_n, limbs, bits, t_bits), he.Context(log_n, limbs, bits, t_bits)
    plain.tune(he.TUNE_NTT_LOG_RADIX, 5)
    return quad, plain


@pytest.mark.parametrize("log_n", [12, 13, 14])
@pytest.mark.parametrize("limbs", [1, 2, 3, 4])
@pytest.mark.parametrize("bits", [60, 54])
def test_raw_transforms(log_n, limbs, bits):
    from paper_2403_11166_gb300 import he
    ctx = he.Context(log_n, limbs, bits, 41)
    g = torch.Generator(device="cuda")
    g.manual_seed(log_n * 10 + limbs)
    big = torch.empty((330, limbs, 1 << log_n), dtype=torch.int64, device="cuda")
    for j, q in enumerate(ctx.primes()[0]):
        big[:, j] = torch.randint(0, q, (330, 1 << log_n), generator=g, device="cuda", dtype=torch.int64)
        big[0, j], big[1, j] = q - 1, 0
        big[2, j] = torch.where(torch.arange(1 << log_n, device="cuda") % 2 == 0, q - 1, 0)
    for count in (1, 5):
        for inverse in (False, True):
            want, got = big.clone(), big[:count].clone()
            he.pencil_ntt_batch(ctx, want, inverse)
            he.pencil_ntt_batch(ctx, got, inverse)
            assert torch.equal(got, want[:count]), (count, inverse)


@pytest.mark.parametrize("log_n,limbs,bits,t_bits", [(12, 2, 54, 41), (13, 3, 60, 59), (14, 4, 60, 41), (12, 1, 60, 30)])
@pytest.mark.parametrize("layer", [("fc", 2, 9, 5, 1, 1, 0), ("conv", 2, 2, 3, 6, 3, 1), ("conv", 1, 1, 2, 9, 5, 0)])
def test_protocol_steps(log_n, limbs, bits, t_bits, layer):
    from paper_2403_11166_gb300 import he
    kind, b, ci, co, h, s, pad = layer
    lay = he.Layer(he.FC if kind == "fc" else he.CONV, b, ci, co, h, h, s, pad)
    g = torch.Generator().manual_seed(5)
    w = torch.randint(-4096, 4096, (co * ci * s * s,), generator=g).cuda()
    x0, x1 = (torch.randint(0, 1 << t_bits, (b * ci * h * h,), generator=g).cuda() for _ in range(2))
    outs = []
    for ctx in _ctxs(log_n, limbs, bits, t_bits):
        sk = ctx.keygen(3)
        pk = ctx.pk_keygen(sk, 4)
        if limbs > 2:
            ctx.flooding(50)
        plan = he.Plan(ctx, lay, he.ROLE_FWD)
        z = plan.sizes
        ws = plan.new_ws(max(z.ws_encrypt, z.ws_encrypt_pk, z.ws_forward, z.ws_decrypt))
        pt, px = plan.new_pt(z.pt), plan.new_pt(z.ct_in)
        ct, ctp, out = plan.new_ct(z.ct_in), plan.new_ct(z.ct_in), plan.new_ct(z.ct_out)
        y0, y1, y2 = (torch.empty(z.out_elems, dtype=torch.int64, device="cuda") for _ in range(3))
        c0c = torch.empty((limbs, z.out_elems), dtype=torch.int64, device="cuda")
        he.encode_weights(ctx, plan, he.OPERAND_KERNEL, w, pt)
        he.encode_weights(ctx, plan, he.OPERAND_INPUT, x0, px)
        he.encrypt_share(ctx, sk, plan, he.OPERAND_INPUT, x1, 11, ct, ws)
        he.encrypt_share_pk(ctx, pk, plan, he.OPERAND_INPUT, x1, 12, ctp, ws)
        he.he_linear_forward(ctx, plan, ct, pt, x0, None, 13, out, y0, ws)
        he.decrypt_to_share(ctx, sk, plan, out, y1, False, ws)
        he.compact_returned(ctx, plan, out, c0c)
        he.decrypt_compact_to_share(ctx, sk, plan, out, c0c, y2, False, ws)
        assert torch.equal(y1, y2)
        outs.append((pt, px, ct, ctp, out, y0, y1, c0c))
    for a, b_ in zip(*outs):
        assert torch.equal(a, b_)
