"""The MO's prepared terms with and without flooding: the Shoup engine's words against the
split products' (returned ciphertexts of a zero plaintext are minus the prepared masks)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flood", [0, 1, 50, 62])
@pytest.mark.parametrize("b", [2, 40])
def test_prepared_terms_agree(flood, b):
    from paper_2403_11166_gb300 import he
    outs = []
    for arith in (0, 1):
        ctx = he.Context(13, 3, 60, 41)
        ctx.tune(he.TUNE_NTT_ARITH, arith)
        ctx.flooding(flood)
        plan = he.Plan(ctx, he.Layer(he.FC, b, 300, 7), he.ROLE_FWD, (1, 300, 7, 1, 1, 1, 1))
        s = plan.sizes
        g = torch.Generator(device="cuda").manual_seed(b)
        x0 = torch.randint(0, 1 << 41, (b * 300,), generator=g, device="cuda", dtype=torch.int64)
        ct, pt = plan.new_ct(s.ct_in).zero_(), plan.new_pt(s.pt)
        he.encode_weights(ctx, plan, he.OPERAND_KERNEL, torch.arange(2100, device="cuda"), pt)
        out, y0 = plan.new_ct(s.ct_out), torch.empty(s.out_elems, dtype=torch.int64, device="cuda")
        he.he_linear_forward(ctx, plan, ct, pt, x0, None, 11, out, y0, plan.new_ws(s.ws_forward))
        outs.append((out, y0))
    for a, c in zip(*outs):
        assert torch.equal(a, c)
