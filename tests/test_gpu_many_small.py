"""N = 4096 transforms four to an SM (large launches) against the same polynomials in
launches that run two to an SM, and around the size where the form changes."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _words(ctx, count, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.empty((count, ctx.L, ctx.n), dtype=torch.int64, device="cuda")
    for j, q in enumerate(ctx.primes()[0]):
        t[:, j] = torch.randint(0, q, (count, ctx.n), generator=g, device="cuda", dtype=torch.int64)
        t[0, j], t[-1, j] = q - 1, 0
    return t


@pytest.mark.parametrize("limbs,bits", [(1, 60), (2, 54), (3, 60)])
@pytest.mark.parametrize("inverse", [False, True])
def test_raw_transforms(limbs, bits, inverse):
    from paper_2403_11166_gb300 import he
    ctx = he.Context(12, limbs, bits, 41)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    edge = (4 if inverse else 3) * sms // limbs
    for count in (edge, edge + 1, 3 * edge + 7):
        x = _words(ctx, count, count)
        want = x.clone()
        for part in want.split(100):   # at most two or three transforms per SM
            he.pencil_ntt_batch(ctx, part, inverse)
        he.pencil_ntt_batch(ctx, x, inverse)
        assert torch.equal(x, want), count


@pytest.mark.parametrize("bits", [60, 54])
@pytest.mark.parametrize("flood", [0, 30])
def test_protocol_steps(bits, flood):
    """A layer of many polynomials, default (64 registers) and radix 2^5 launches."""
    from paper_2403_11166_gb300 import he
    outs = []
    for radix in (4, 5):
        ctx = he.Context(12, 2, bits, 20)
        ctx.tune(he.TUNE_NTT_LOG_RADIX, radix)
        if flood:
            ctx.flooding(flood)
        sk = ctx.keygen(5)
        plan = he.Plan(ctx, he.Layer(he.CONV, 40, 16, 16, 32, 32, 3, 1), he.ROLE_FWD)
        s = plan.sizes
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        assert min(2 * s.pt, 2 * s.ct_in + 2 * s.ct_out) > 3 * sms
        g = torch.Generator(device="cuda")
        g.manual_seed(1)
        r = lambda n: torch.randint(0, 1 << 20, (n,), generator=g, device="cuda", dtype=torch.int64)
        w, x1, x0 = r(16 * 16 * 9), r(40 * 16 * 1024), r(40 * 16 * 1024)
        pt, ct, out = plan.new_pt(s.pt), plan.new_ct(s.ct_in), plan.new_ct(s.ct_out)
        y0, y1 = (torch.empty(s.out_elems, dtype=torch.int64, device="cuda") for _ in range(2))
        ws = plan.new_ws(max(s.ws_encrypt, s.ws_forward, s.ws_decrypt))
        he.encode_weights(ctx, plan, he.OPERAND_KERNEL, w, pt)
        he.encrypt_share(ctx, sk, plan, he.OPERAND_INPUT, x1, 7, ct, ws)
        he.he_linear_forward(ctx, plan, ct, pt, x0, None, 9, out, y0, ws)
        he.decrypt_to_share(ctx, sk, plan, out, y1, True, ws)
        assert ctx.sync_status() == 0
        outs.append((plan.part, pt, ct, out, y0, y1))
    assert outs[0][0] == outs[1][0]
    for a, b in zip(outs[0][1:], outs[1][1:]):
        assert torch.equal(a, b)
