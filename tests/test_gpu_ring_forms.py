"""Every form of the plaintext correlations over Z_t (tile, offsets and outputs on the
integer pipe, digit products on the tensor cores) against int64 PyTorch (wrap-around is
exact mod t), at the edges of its threads, tiles and chunks.  The form a size takes is
asserted with the library's own rule, so that a change of the rule cannot leave one
without a test."""
import pytest
import torch

from tests import rules_lib

pytestmark = pytest.mark.gpu

# (B, Ci, Co, H, kernel, pad), role -> form (both t).  Roles: 0 forward, 1 input gradient, 2 weight gradient
CASES = {
    "tile": [((1, 1, 1, 1, 1, 0), 0), ((5, 2, 7, 1, 1, 0), 0), ((513, 4, 9, 1, 1, 0), 0), ((70, 17, 2, 1, 1, 0), 1),
             ((1, 130, 17, 1, 1, 0), 2), ((2, 65, 33, 1, 1, 0), 2), ((40, 1, 3, 41, 3, 1), 0), ((40, 1, 1, 39, 3, 2), 0),
             ((4, 2, 1, 30, 1, 0), 1)],
    "offsets": [((1, 1, 1, 28, 5, 2), 2), ((1, 3, 9, 16, 3, 1), 2), ((2, 2, 3, 17, 1, 0), 2), ((1, 4, 2, 20, 3, 0), 2),
                ((1, 2, 5, 24, 5, 4), 2)],
    "outputs": [((1, 1, 2, 20, 4, 2), 2), ((1, 2, 1, 16, 2, 1), 2), ((1, 1, 3, 28, 7, 3), 2)],
    "digits": [((64, 37, 17, 1, 1, 0), 0), ((33, 100, 65, 1, 1, 0), 0), ((7, 700, 3, 1, 1, 0), 0), ((65, 9, 33, 1, 1, 0), 2),
               ((300, 6, 5, 1, 1, 0), 2), ((3, 20, 18, 9, 3, 1), 0), ((2, 5, 33, 11, 5, 2), 1), ((60, 4, 3, 20, 3, 1), 2),
               ((2, 16, 2, 7, 5, 4), 0), ((40, 3, 40, 18, 1, 0), 2), ((90, 5, 20, 17, 2, 0), 2)],
}
FLAT = [(form, layer, role) for form, cases in CASES.items() for layer, role in cases]


def _correlate(v, w):
    """y[a, o, i, j] = sum_{c, u, x} w[o, c, u, x] v[a, c, i + u, j + x] in int64."""
    a, _, h, wd = v.shape
    o, _, kh, kw = w.shape
    ho, wo = h - kh + 1, wd - kw + 1
    y = torch.zeros((a, o, ho, wo), dtype=torch.int64)
    for u in range(kh):
        for x in range(kw):
            win = v[:, :, u:u + ho, x:x + wo].permute(0, 2, 3, 1).reshape(-1, v.shape[1])
            y += (win @ w[:, :, u, x].T).view(a, ho, wo, o).permute(0, 3, 1, 2)
    return y


@pytest.mark.parametrize("t_bits", [41, 59])
@pytest.mark.parametrize("form,layer,role", FLAT)
def test_matches_int64(form, layer, role, t_bits):
    from paper_2403_11166_gb300 import he
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert rules_lib.ring_form(layer, role, t_bits, sms) == form
    b, ci, co, h, s, pad = layer
    kind = he.FC if (h, s) == (1, 1) else he.CONV
    ctx = he.Context(12, 2, 60, t_bits)
    plan = he.Plan(ctx, he.Layer(kind, b, ci, co, h, h, s, pad), role)
    g = torch.Generator().manual_seed(b * 100 + ci * 10 + co)
    mask, ho = (1 << t_bits) - 1, h + 2 * pad - s + 1

    def draw(*shape):
        return torch.randint(0, 1 << t_bits, shape, generator=g, dtype=torch.int64)
    x, w, gy = draw(b, ci, h, h), draw(co, ci, s, s), draw(b, co, ho, ho)
    w[0, 0, 0, 0] = -5   # weights are signed
    pd = torch.nn.functional.pad
    if role == 0:
        kern, inp, ref = w, x, _correlate(pd(x, (pad,) * 4), w)
    elif role == 1:
        kern, inp, ref = w, gy, _correlate(pd(gy, (s - 1 - pad,) * 4), w.flip(2, 3).transpose(0, 1))
    else:
        kern, inp = gy, x
        ref = _correlate(pd(x, (pad,) * 4).transpose(0, 1), gy.transpose(0, 1)).transpose(0, 1)
    ref = ref.reshape(-1)
    a1, a2 = draw(ref.numel()), draw(ref.numel())
    dev = [t.contiguous().cuda() for t in (kern, inp, a1, a2)]
    out = torch.empty(ref.numel(), dtype=torch.int64, device="cuda")
    he.pencil_ring_linear(ctx, plan, dev[0], dev[1], None, out)
    assert torch.equal(out.cpu(), ref & mask)
    acc = dev[2].clone()   # the output may be its own addend
    he.pencil_ring_linear(ctx, plan, dev[0], dev[1], acc, acc, addend2=dev[3])
    assert torch.equal(acc.cpu(), (ref + a1 + a2) & mask)
