"""Contexts of the shortest primes (30 and 31 bits), which have no split products: keys, both
encryptions, the products and decryption; and the memory of their keys."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n,bits", [(12, 30), (13, 31), (14, 31)])
def test_layer_forward(log_n, bits):
    from paper_2403_11166_gb300 import he
    t = 16
    ctx = he.Context(log_n, 4, bits, t)
    sk = ctx.keygen(3)
    pk = ctx.pk_keygen(sk, 4)
    b, ci, co = 3, 50, 7
    plan = he.Plan(ctx, he.Layer(he.FC, b, ci, co), he.ROLE_FWD)
    s = plan.sizes
    g = torch.Generator().manual_seed(bits)
    w = torch.randint(-128, 128, (co, ci), generator=g)
    x0, x1 = (torch.randint(0, 1 << t, (b, ci), generator=g) for _ in range(2))
    ws = plan.new_ws(max(s.ws_encrypt, s.ws_encrypt_pk, s.ws_forward, s.ws_decrypt))
    pt, ct, out = plan.new_pt(s.pt), plan.new_ct(s.ct_in), plan.new_ct(s.ct_out)
    y0, y1 = (torch.empty(s.out_elems, dtype=torch.int64, device="cuda") for _ in range(2))
    he.encode_weights(ctx, plan, he.OPERAND_KERNEL, w.cuda(), pt)
    want = ((x0 + x1) @ w.T).reshape(-1) & ((1 << t) - 1)
    for encrypt in ("secret", "public"):
        if encrypt == "secret":
            he.encrypt_share(ctx, sk, plan, he.OPERAND_INPUT, x1.cuda(), 5, ct, ws)
        else:
            he.encrypt_share_pk(ctx, pk, plan, he.OPERAND_INPUT, x1.cuda(), 5, ct, ws)
        he.he_linear_forward(ctx, plan, ct, pt, x0.cuda(), None, 9, out, y0, ws)
        he.decrypt_to_share(ctx, sk, plan, out, y1, True, ws)
        assert ctx.sync_status() == 0
        assert torch.equal((y0 + y1).cpu() & ((1 << t) - 1), want)


def test_keys_hold_one_form_where_the_context_has_one():
    """256 secret keys of 4 limbs at N = 16384: 1 MiB each with Shoup companions alone."""
    from paper_2403_11166_gb300 import he
    ctx = he.Context(14, 4, 50, 20)
    first = ctx.keygen(1)   # (module loading)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    keys = [ctx.keygen(i) for i in range(256)]
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    assert used < 256 * 1.5 * (1 << 20), used
    del keys, first
