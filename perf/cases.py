"""Timed workloads of the homomorphic linear layers, through the public calls of
`paper_2403_11166_gb300` (he, autograd, prep).

Every case is one pass a party pair makes: the data owner's encryption and
decryption and the model owner's evaluation of one layer (`linear`), of one layer
forward and backward (`train`), of one layer served with kept weights, public-key
ciphertexts, flooding and the compact send form (`serve`), of many uneven layers
in one captured graph (`batch`), the HE-free online phase of the preprocessing
protocol (`online`), a training step of the 3-layer network (`cnn`), and the
batched transforms alone (`ntt`).  Weights and activations are N(0, 1) clipped to
+-8 in fixed point, shares and masks uniform in Z_t.
"""
import math

import torch

from paper_2403_11166_gb300 import autograd, he, prep

CONV, FC = "conv", "fc"


def _linear(name, family, kind, b, ci, co, hw=1, k=1, pad=0, log_n=13, limbs=3, bits=60, t=41, frac=12, **more):
    return {"name": name, "family": family, "kind": kind, "b": b, "ci": ci, "co": co, "hw": hw, "k": k, "pad": pad,
            "log_n": log_n, "limbs": limbs, "bits": bits, "t": t, "frac": frac, **more}


def _ntt(name, log_n, limbs, bits, count, inverse):
    return {"name": name, "family": "ntt", "log_n": log_n, "limbs": limbs, "bits": bits, "count": count,
            "inverse": inverse}


def listed():
    return [
        # one sample through a small classifier head at the paper's parameters (t = 2^59, f = 25): latency
        _linear("fc256_100_b1_fwd_t59", "linear", FC, 1, 256, 100, t=59, frac=25),
        # a transform of a few polynomials (one small layer's worth), two 54-bit primes: latency
        _ntt("intt_n4096_l2x54_16", 12, 2, 54, 16, True),
        # small layer, N = 4096, two 54-bit primes: forward, input gradient and weight gradient
        _linear("fc784_100_b32_train", "train", FC, 32, 784, 100, log_n=12, limbs=2, bits=54),
        # the ordinary convolution layer, forward (products per second are quoted on it)
        _linear("conv16_16_32_b64_fwd", "linear", CONV, 64, 16, 16, 32, 3, 1),
        # ragged sizes: 3 input channels, 58 x 58 padded images, the paper's parameters
        _linear("conv3_64_56_b64_fwd_t59", "linear", CONV, 64, 3, 64, 56, 3, 1, t=59, frac=25),
        # serving: weights encoded once, public-key ciphertexts, flooded and compacted replies, odd widths
        _linear("fc2048_1001_b64_serve", "serve", FC, 64, 2048, 1001, flood=62),
        # 96 uneven layers as one captured graph
        {"name": "batch96_uneven_fwd", "family": "batch", "each": 32, "log_n": 13, "limbs": 3, "bits": 60, "t": 41},
        # preprocessing protocol's online phase, m = 8 masks per party
        _linear("online_conv16_m8", "online", CONV, 64, 16, 16, 32, 3, 1, m=8),
        # a private training step of the 3-layer network: logits and all gradients
        {"name": "cnn3_b64_step", "family": "cnn", "b": 64, "hw": 32, "c1": 16, "c2": 32, "classes": 10},
        # a wide layer, forward and both gradients
        _linear("conv128_128_16_b128_train", "train", CONV, 128, 128, 128, 16, 3, 1),
        # sustained transforms
        _ntt("ntt_n8192_l3_10000", 13, 3, 60, 10000, False),
        _ntt("intt_n16384_l4_2500", 14, 4, 60, 2500, True),
    ]


# ------------------------------------------------------------------ sizes of a case
def _shapes(c):
    if c["kind"] == FC:
        return (c["co"], c["ci"]), (c["b"], c["ci"]), (c["b"], c["co"])
    ho = c["hw"] + 2 * c["pad"] - c["k"] + 1
    return ((c["co"], c["ci"], c["k"], c["k"]), (c["b"], c["ci"], c["hw"], c["hw"]), (c["b"], c["co"], ho, ho))


def _ring_macs(c):
    """64-bit multiply-adds of the plain layer over Z_t."""
    w, _, y = _shapes(c)
    return math.prod(w) * c["b"] * (math.prod(y[2:]) if len(y) > 2 else 1)


def _poly_counts(c):
    """(input polynomials, kernel polynomials, output polynomials, products) a layer cannot do without."""
    n = 1 << c["log_n"]
    hw, kk = (c["hw"] + 2 * c["pad"]) ** 2, c["k"] ** 2   # padded window, kernel elements
    counts = (c["b"] * c["ci"] * hw, c["ci"] * c["co"] * kk, c["b"] * c["co"] * hw, c["b"] * c["ci"] * c["co"] * hw)
    return tuple(max(1.0, v / n) for v in counts)


def _ntt_ops(log_n):
    """32-bit multiply-adds (2 operations each) of one limb's transform: N/2 log2 N modular products of 10 each."""
    return 2.0 * 10 * (1 << (log_n - 1)) * log_n


def _he_work(c, roles):
    n, limbs = 1 << c["log_n"], c["limbs"]
    i, w, o, p = _poly_counts(c)
    ntts = limbs * (2 * i + w + 2 * o)
    flops = roles * (ntts * _ntt_ops(c["log_n"]) + p * 2 * limbs * n * 8.0)
    return flops, 16.0 * limbs * n


def work(case):
    f = case["family"]
    if f == "ntt":
        polys = float(case["count"] * case["limbs"])
        return {"bytes": 16.0 * polys * (1 << case["log_n"]), "flops": polys * _ntt_ops(case["log_n"])}
    if f == "batch":
        flops = bytes_ = 0.0
        for c in _batch_layers(case["each"]):
            c = {**case, **c}
            flops += _he_work(c, 1)[0]
            w, x, y = _shapes(c)
            bytes_ += 8.0 * (math.prod(w) + 2 * math.prod(x) + 2 * math.prod(y))
        return {"bytes": bytes_, "flops": flops}
    if f == "cnn":
        flops = bytes_ = 0.0
        hw, b = case["hw"], case["b"]
        for kind, ci, co, k in ((CONV, 3, case["c1"], 3), (CONV, case["c1"], case["c2"], 3),
                                (FC, case["c2"] * hw * hw // 4, case["classes"], 1)):
            c = _linear("", "", kind, b, ci, co, hw if kind == CONV else 1, k, k // 2)
            flops += _he_work(c, 3)[0]
            w, x, y = _shapes(c)
            bytes_ += 8.0 * (2 * math.prod(w) + 2 * math.prod(x) + 2 * math.prod(y))
        return {"bytes": bytes_, "flops": flops}
    w, x, y = (math.prod(s) for s in _shapes(case))
    if f == "online":
        m = case["m"]
        # masks, operands and both parties' m^2 shares in; the masked operands and the shares out
        return {"bytes": 8.0 * ((m + 2) * w + (m + 2) * x + (2 * m * m + 2) * y),
                "flops": 6.0 * (m + 1) * _ring_macs(case)}
    flops, ct = _he_work(case, 3 if f == "train" else 1)
    i, _, o, _ = _poly_counts(case)
    if f == "linear":   # operands in; both shares and the ciphertexts that travel out
        return {"bytes": 8.0 * (w + 2 * x + 2 * y) + ct * (i + o), "flops": flops}
    if f == "serve":
        k = max(1.0, case["ci"] * case["co"] / (1 << case["log_n"]))
        return {"bytes": 8.0 * (2 * x + 2 * y) + ct * (i + o + k / 2), "flops": flops}
    return {"bytes": 8.0 * (2 * w + 4 * x + 4 * y), "flops": flops + 12.0 * _ring_macs(case)}   # train


# ------------------------------------------------------------------ drawn cases
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


_RINGS = [(12, 2, 54), (12, 2, 60), (13, 3, 60), (13, 3, 60), (13, 3, 60), (13, 4, 60), (14, 3, 60), (14, 4, 60)]


def _draw_layer(rng, family):
    log_n, limbs, bits = rng.choice(_RINGS)
    t, frac = rng.choice([(41, 12), (41, 12), (59, 25)]) if limbs > 2 else (41, 12)
    ring = dict(log_n=log_n, limbs=limbs, bits=bits, t=t, frac=frac)
    if rng.random() < 0.4:
        return _linear("", family, FC, _log_int(rng, 1, 64), _log_int(rng, 10, 2048), _log_int(rng, 4, 1100), **ring)
    k = rng.choice([1, 3, 3, 3, 5])
    hw = _log_int(rng, 4, 56)
    return _linear("", family, CONV, _log_int(rng, 1, 128), _log_int(rng, 1, 128), _log_int(rng, 1, 128),
                   max(hw, k), k, rng.choice([0, k // 2]), **ring)


def draw(rng):
    big = listed()[9]
    most = work(big)["flops"]
    while True:
        family = rng.choice(["linear", "linear", "train", "ntt", "ntt", "serve", "online"])
        if family == "ntt":
            log_n, limbs = rng.choice([12, 13, 14]), rng.choice([1, 2, 3, 4])
            most_polys = (1 << 31) // ((8 << log_n) * limbs)
            c = _ntt("", log_n, limbs, rng.choice([60, 60, 54]), _log_int(rng, 1, min(10000, most_polys)),
                     rng.random() < 0.5)
        else:
            c = _draw_layer(rng, family)
            if family == "serve":
                c.update(flood=rng.choice([0, 62]) if c["limbs"] > 2 else 0)
            if family == "online":
                c.update(m=rng.choice([2, 4, 8]))
                if c["limbs"] < 3:
                    continue   # products of two uniform masks need the noise room of three primes
            # a drawn case costs at most half of the largest listed one, buffers included
            x, y = math.prod(_shapes(c)[1]), math.prod(_shapes(c)[2])
            i, _, o, p = _poly_counts(c)
            scale = c.get("m", 1)
            if c["family"] == "online" and (scale * scale * y > 1 << 25 or scale * _ring_macs(c) > 1 << 31):
                continue
            pts = c["ci"] * c["co"] if c["kind"] == CONV else c["ci"] * c["co"] / (1 << c["log_n"])
            ct = 16.0 * c["limbs"] * (1 << c["log_n"])
            if max(scale * scale * work(c)["flops"], ct * pts * 500) > most / 2 or ct * (i + o + pts) > 4e9:
                continue
            if max(x, y) > 1 << 24:
                continue
        del c["name"]
        return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _fixed(g, shape, frac):
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64).clamp_(-8, 8)
    return torch.floor(x * (1 << frac)).to(torch.int64)


def _uniform(g, shape, t):
    return torch.randint(0, 1 << t, shape, generator=g, device="cuda", dtype=torch.int64)


def _shares(g, shape, frac, t):
    x1 = _uniform(g, shape, t)
    return ((_fixed(g, shape, frac) - x1) & ((1 << t) - 1)), x1


def _layer(c):
    return he.Layer(he.FC if c["kind"] == FC else he.CONV, c["b"], c["ci"], c["co"], c["hw"], c["hw"], c["k"],
                    c["pad"])


def _words(count):
    return torch.empty(count, dtype=torch.int64, device="cuda")


class _Linear:
    """Alg. 1 for one layer: encode the weights, encrypt the data owner's share, evaluate and re-mask, decrypt."""

    def __init__(self, c, seed):
        g = _gen(seed)
        self.ctx = he.Context(c["log_n"], c["limbs"], c["bits"], c["t"])
        self.sk = self.ctx.keygen(seed + 1)
        w, x, _ = _shapes(c)
        self.w = _fixed(g, w, c["frac"])
        self.x0, self.x1 = _shares(g, x, c["frac"], c["t"])
        self.bias = _uniform(g, (c["co"],), c["t"])
        self.plan = he.Plan(self.ctx, _layer(c), he.ROLE_FWD)
        s = self.plan.sizes
        self.pt, self.ct_in, self.ct_out = (self.plan.new_pt(s.pt), self.plan.new_ct(s.ct_in),
                                            self.plan.new_ct(s.ct_out))
        self.ws = self.plan.new_ws(max(s.ws_encrypt, s.ws_forward, s.ws_decrypt))
        self.y0, self.y1 = _words(s.out_elems), _words(s.out_elems)
        self.seed = seed << 20

    def run(self):
        self.seed += 2
        he.encode_weights(self.ctx, self.plan, he.OPERAND_KERNEL, self.w, self.pt)
        he.encrypt_share(self.ctx, self.sk, self.plan, he.OPERAND_INPUT, self.x1, self.seed, self.ct_in, self.ws)
        he.he_linear_forward(self.ctx, self.plan, self.ct_in, self.pt, self.x0, self.bias, self.seed + 1,
                             self.ct_out, self.y0, self.ws)
        he.decrypt_to_share(self.ctx, self.sk, self.plan, self.ct_out, self.y1, True, self.ws)
        return {"y0": self.y0, "y1": self.y1, "ct_in": self.ct_in, "ct_out": self.ct_out}


class _Serve(_Linear):
    """Alg. 1 with the weights encoded once, public-key encryption, flooding and the compact send form."""

    def __init__(self, c, seed):
        super().__init__(c, seed)
        self.pk = self.ctx.pk_keygen(self.sk, seed + 2)
        if c["flood"]:
            self.ctx.flooding(c["flood"])
        s = self.plan.sizes
        self.ws = self.plan.new_ws(max(s.ws_encrypt_pk, s.ws_forward, s.ws_decrypt))
        self.c0c = torch.empty((c["limbs"], s.out_elems), dtype=torch.int64, device="cuda")
        he.encode_weights(self.ctx, self.plan, he.OPERAND_KERNEL, self.w, self.pt)

    def run(self):
        self.seed += 2
        he.encrypt_share_pk(self.ctx, self.pk, self.plan, he.OPERAND_INPUT, self.x1, self.seed, self.ct_in, self.ws)
        he.he_linear_forward(self.ctx, self.plan, self.ct_in, self.pt, self.x0, self.bias, self.seed + 1,
                             self.ct_out, self.y0, self.ws)
        he.compact_returned(self.ctx, self.plan, self.ct_out, self.c0c)
        he.decrypt_compact_to_share(self.ctx, self.sk, self.plan, self.ct_out, self.c0c, self.y1, True, self.ws)
        return {"y0": self.y0, "y1": self.y1, "ct_in": self.ct_in, "ct_out": self.ct_out, "c0c": self.c0c}


class _Train:
    """One layer's forward pass, input gradient (Alg. 1 form) and weight gradient (Alg. 2) through a session."""

    def __init__(self, c, seed):
        g = _gen(seed)
        self.sess = autograd.HeSession(c["log_n"], c["limbs"], c["bits"], c["t"], c["frac"], seed=seed)
        self.layer = _layer(c)
        w, x, y = _shapes(c)
        self.w = _fixed(g, w, c["frac"]) & self.sess.mask
        self.bias = _uniform(g, (c["co"],), c["t"])
        self.x0, self.x1 = _shares(g, x, c["frac"], c["t"])
        self.g0, self.g1 = _shares(g, y, c["frac"], c["t"])

    def run(self):
        y0, y1 = self.sess.forward(self.layer, self.w, self.bias, self.x0, self.x1)
        gx0, gx1, gw, gb = self.sess.backward(self.layer, self.w, self.x0, self.x1, self.g0, self.g1, True)
        return {"y0": y0, "y1": y1, "gx0": gx0, "gx1": gx1, "gw": gw, "gb": gb}


def _batch_layers(each):
    return ([{"kind": FC, "b": 16, "ci": 512, "co": 10, "hw": 1, "k": 1, "pad": 0}] * each
            + [{"kind": CONV, "b": 32, "ci": 64, "co": 64, "hw": 8, "k": 3, "pad": 1}] * each
            + [{"kind": CONV, "b": 8, "ci": 128, "co": 256, "hw": 4, "k": 1, "pad": 0}] * each)


class _Batch:
    """Many layers' forward passes, committed once and replayed as one captured graph."""

    def __init__(self, c, seed):
        g = _gen(seed)
        self.ctx = he.Context(c["log_n"], c["limbs"], c["bits"], c["t"])
        self.sk = self.ctx.keygen(seed + 1)
        layers = _batch_layers(c["each"])
        self.plans = [he.Plan(self.ctx, _layer(p), he.ROLE_FWD) for p in layers]
        self.batch = he.Batch(self.ctx, self.plans)
        total = sum(p.sizes.out_elems for p in self.plans)
        self.y0, self.y1 = _words(total), _words(total)
        at = 0
        for i, (p, plan) in enumerate(zip(layers, self.plans)):
            w, x, _ = _shapes(p)
            x0, x1 = _shares(g, x, 12, c["t"])
            n = plan.sizes.out_elems
            self.batch.bind(i, _fixed(g, w, 12), x1, x0, None, self.y0[at:at + n], self.y1[at:at + n])
            at += n
        self.ws = _words((self.batch.workspace_bytes + 7) // 8)
        self.batch.commit(self.sk, self.ws, (seed << 8) + 1000, (seed << 8) + 5000)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            self.batch.forward(stream=side)
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(self.graph):
            self.batch.forward()

    def run(self):
        self.graph.replay()
        return {"y0": self.y0, "y1": self.y1}


class _Online:
    """Alg. 3's online phase of a layer's forward product, the m^2 preprocessed shares in hand."""

    def __init__(self, c, seed):
        g = _gen(seed)
        self.ctx = he.Context(c["log_n"], c["limbs"], c["bits"], c["t"])
        self.sk = self.ctx.keygen(seed + 1)
        w, x, _ = _shapes(c)
        m = c["m"]
        self.w = _fixed(g, w, c["frac"])
        self.x1 = _uniform(g, x, c["t"])
        self.k = [int(v) for v in _uniform(g, (m,), c["t"]).cpu()]
        self.l = [int(v) for v in _uniform(g, (m,), c["t"]).cpu()]
        self.prod = prep.PrepProduct(self.ctx, self.sk, _layer(c), he.ROLE_FWD, m)
        self.prod.preprocess(_uniform(g, (m * w[0],) + tuple(w[1:]), c["t"]),
                             _uniform(g, (m * x[0],) + tuple(x[1:]), c["t"]), seed + 3, seed + 4)

    def run(self):
        ut, vt, z0, z1 = self.prod.online(self.w, self.x1, self.k, self.l)
        return {"ut": ut, "vt": vt, "z0": z0, "z1": z1}


class _Ntt:
    """In-place transforms of a batch of uniform polynomials."""

    def __init__(self, c, seed):
        g = _gen(seed)
        self.ctx = he.Context(c["log_n"], c["limbs"], c["bits"], 41 if c["bits"] > 41 else 20)
        primes, _ = self.ctx.primes()
        self.inverse = c["inverse"]
        self.polys = torch.empty((c["count"], c["limbs"], 1 << c["log_n"]), dtype=torch.int64, device="cuda")
        for j, q in enumerate(primes):
            self.polys[:, j] = torch.randint(0, q, (c["count"], 1 << c["log_n"]), generator=g, device="cuda",
                                             dtype=torch.int64)

    def run(self):
        he.pencil_ntt_batch(self.ctx, self.polys, self.inverse)
        return self.polys


# ------------------------------------------------------------------ the 3-layer network
def _cnn_inputs(c, seed, device):
    """Fixed-point weights N(0, 1/fan_in), images and the upstream gradient of the logits (float64, CPU draws)."""
    g = torch.Generator().manual_seed(seed)
    fc_in = c["c2"] * (c["hw"] // 2) ** 2

    def w(shape, fan):
        return torch.floor(torch.randn(shape, generator=g, dtype=torch.float64) / math.sqrt(fan) * 4096) / 4096
    p = {"w1": w((c["c1"], 3, 3, 3), 27), "b1": w((c["c1"],), 27), "w2": w((c["c2"], c["c1"], 3, 3), 9 * c["c1"]),
         "b2": w((c["c2"],), 9 * c["c1"]), "w3": w((c["classes"], fc_in), fc_in), "b3": w((c["classes"],), fc_in)}
    x = torch.floor(torch.randn((c["b"], 3, c["hw"], c["hw"]), generator=g, dtype=torch.float64).clamp_(-8, 8)
                    * 4096) / 4096
    gy = torch.randn((c["b"], c["classes"]), generator=g, dtype=torch.float64) * 8
    return {k: v.to(device) for k, v in p.items()}, x.to(device), gy.to(device)


class _Cnn:
    def __init__(self, c, seed):
        p, self.x, self.gy = _cnn_inputs(c, seed, "cuda")
        self.sess = autograd.HeSession(13, 3, 60, 41, seed=seed)
        self.model = autograd.SecureCNN(self.sess, c["b"], p, c["hw"], c["hw"])
        self.names = ("w1", "b1", "w2", "b2", "w3", "b3")

    def run(self):
        logits = self.model(self.x)
        grads = torch.autograd.grad(logits, [getattr(self.model, n) for n in self.names], self.gy)
        return {"logits": logits.detach(), **dict(zip(self.names, grads))}


def _cnn_exact(c, seed):
    """The same step on plaintext fixed-point values: every sum is an integer below 2^53, exact in float64."""
    p, x, gy = _cnn_inputs(c, seed, "cpu")
    f = float(1 << 12)
    conv = torch.nn.functional.conv2d

    def enc(v):
        return torch.floor(v * f)

    def dec(v, bits):
        return v / float(1 << bits)

    X1, W1, W2, W3 = enc(x), enc(p["w1"]), enc(p["w2"]), enc(p["w3"])
    b1, b2, b3 = (torch.floor(p[k] * f * f) for k in ("b1", "b2", "b3"))
    y1 = dec(conv(X1, W1, b1, padding=1), 24)
    on = y1 >= 0
    X2 = enc(torch.where(on, y1, torch.zeros_like(y1)))
    y2 = dec(conv(X2, W2, b2, padding=1), 24)
    X3 = enc(torch.nn.functional.avg_pool2d(y2, 2).reshape(c["b"], -1))
    logits = dec(X3 @ W3.T + b3, 24)
    G3 = torch.floor(gy * f + 0.5)
    g3 = dec(G3 @ W3, 24)
    g2 = (g3.reshape(c["b"], c["c2"], c["hw"] // 2, c["hw"] // 2) / 4).repeat_interleave(2, 2).repeat_interleave(2, 3)
    G2 = torch.floor(g2 * f + 0.5)
    w2 = torch.nn.grad.conv2d_weight(X2, W2.shape, G2, padding=1)
    g1 = dec(torch.nn.grad.conv2d_input(X2.shape, W2, G2, padding=1), 24)
    G1 = torch.floor(torch.where(on, g1, torch.zeros_like(g1)) * f + 0.5)
    w1 = torch.nn.grad.conv2d_weight(X1, W1.shape, G1, padding=1)
    return {"logits": logits, "w1": dec(w1, 24), "b1": dec(G1.sum((0, 2, 3)), 12), "w2": dec(w2, 24),
            "b2": dec(G2.sum((0, 2, 3)), 12), "w3": dec(G3.T @ X3, 24), "b3": dec(G3.sum(0), 12)}


# ------------------------------------------------------------------ entry points
_FAMILIES = {"linear": _Linear, "serve": _Serve, "train": _Train, "batch": _Batch, "online": _Online, "ntt": _Ntt,
             "cnn": _Cnn}


def prepare(case, seed):
    return _FAMILIES[case["family"]](case, seed)


def run(state):
    return state.run()


def exact(case, seed):
    # every other output is whole numbers, held bit for bit
    return _cnn_exact(case, seed) if case["family"] == "cnn" else None
