"""Launches of N = 8192 transforms that give no SM two of them (compiled for one CTA per SM)
at both ends of their range, against the same work elsewhere: raw transforms against the
same polynomials inside a large batch, the protocol's steps against radix 2^5, bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _counts(limbs):
    """Polynomials: the fewest past the clusters' forward range, and the most on one SM each."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return sms // (4 * limbs) + 1, sms // limbs


@pytest.mark.parametrize("limbs,bits", [(1, 60), (2, 54), (3, 60), (4, 59)])
def test_raw_transforms(limbs, bits):
    from paper_2403_11166_gb300 import he
    ctx = he.Context(13, limbs, bits, 41)
    g = torch.Generator(device="cuda").manual_seed(limbs)
    big = torch.empty((330, limbs, 8192), dtype=torch.int64, device="cuda")
    for j, q in enumerate(ctx.primes()[0]):
        big[:, j] = torch.randint(0, q, (330, 8192), generator=g, device="cuda", dtype=torch.int64)
        big[0, j], big[1, j] = q - 1, 0
    for count in _counts(limbs):
        for inverse in (False, True):
            want, got = big.clone(), big[:count].clone()
            he.pencil_ntt_batch(ctx, want, inverse)
            he.pencil_ntt_batch(ctx, got, inverse)
            assert torch.equal(got, want[:count]), (count, inverse)


@pytest.mark.parametrize("limbs,bits,t_bits,flood", [(3, 60, 59, 50), (2, 54, 41, 0)])
@pytest.mark.parametrize("most", [False, True])
def test_protocol_steps(limbs, bits, t_bits, flood, most):
    from paper_2403_11166_gb300 import he
    b = _counts(limbs)[most]
    g = torch.Generator().manual_seed(7)
    w = torch.randint(-4096, 4096, (2 * 4096,), generator=g).cuda()
    x0, x1 = (torch.randint(0, 1 << t_bits, (b * 4096,), generator=g).cuda() for _ in range(2))
    outs = []
    for radix in (4, 5):
        ctx = he.Context(13, limbs, bits, t_bits)
        ctx.tune(he.TUNE_NTT_LOG_RADIX, radix)
        sk = ctx.keygen(3)
        pk = ctx.pk_keygen(sk, 4)
        if flood:
            ctx.flooding(flood)
        plan = he.Plan(ctx, he.Layer(he.FC, b, 4096, 2), he.ROLE_FWD, (1, 4096, 2, 1, 1, 1, 1))
        z = plan.sizes
        assert z.ct_in == z.ct_out == b
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
    for a, c in zip(*outs):
        assert torch.equal(a, c)
