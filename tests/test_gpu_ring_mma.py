"""Plaintext correlations over Z_t on the tensor cores against int64 PyTorch (wrap-around is
exact mod t): part tiles of output channels and positions, reductions of one chunk, of
remainders and split over the grid, both digit counts, every role's strides."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# kind, B, Ci, Co, H, kernel, pad
LAYERS = [("fc", 1, 1, 1, 1, 1, 0), ("fc", 5, 37, 17, 1, 1, 0), ("fc", 33, 16, 65, 1, 1, 0), ("fc", 64, 700, 3, 1, 1, 0),
          ("conv", 1, 1, 1, 1, 1, 0), ("conv", 2, 3, 5, 7, 3, 1), ("conv", 3, 2, 16, 9, 5, 2), ("conv", 2, 17, 33, 6, 3, 0),
          ("conv", 9, 4, 3, 20, 3, 1), ("conv", 2, 2, 2, 5, 5, 4), ("conv", 4, 3, 40, 18, 1, 0), ("conv", 3, 5, 4, 17, 2, 0)]


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
@pytest.mark.parametrize("role", [0, 1, 2])
@pytest.mark.parametrize("layer", LAYERS)
def test_matches_int64(layer, role, t_bits):
    from paper_2403_11166_gb300 import he
    kind, b, ci, co, h, s, pad = layer
    ctx = he.Context(12, 2, 60, t_bits)
    plan = he.Plan(ctx, he.Layer(he.FC if kind == "fc" else he.CONV, b, ci, co, h, h, s, pad), role)
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
