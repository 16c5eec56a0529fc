"""What this library is timed on: the block-CAT quantized linear layer as a program calls it.

A case is a dict of plain values.  ``op`` names what a pass does:

* ``layer``: one W4A4 layer forward, x -> y: the online transform with its per-token codes, then the
  integer GEMM with dequantization.  ``codes`` is the storage form: ``packed`` (4 bits a code, what
  decoding streams) or ``bytes`` (one E4M3 byte a code, what prefill multiplies).  ``sqnr`` adds the
  quality sums against a full-precision y.  ``graph`` replays the calls from a CUDA graph captured
  once, as a decode loop does; otherwise every pass issues them from Python.
* ``dp``: one layer forward at other bit widths (``bits_x``, ``bits_w``), the activations symmetric or
  asymmetric per token.
* ``calib``: the diagonal blocks of the calibration autocorrelation.
* ``weights``: the offline preparation of a layer from its weights and calibration tokens.

Activations have correlated bulk channels and a few outlier channels (or are SwiGLU products), the
weights rows of unequal energy; T is dense inside its blocks (Hadamard times a symmetric positive
matrix that evens out the channels), as block CAT makes it.  ``exact`` works the same inputs out in
float64 with plain torch.
"""
import math

import numpy as np
import torch

import paper_2603_04359_gb300 as cat

LARGEST = 8192 * 8192 * 28672        # multiply-adds of the largest layer listed


def listed():
    return [
        # one token through a fused QKV projection, issued call by call: latency and host cost
        dict(name="decode_1_qkv", op="layer", n=1, d_in=4096, d_out=6144, k=128, dtype="bf16", act="lowrank",
             codes="packed", sqnr=False, graph=False),
        # a small decode batch through an up projection, replayed from a graph
        dict(name="decode_16_up", op="layer", n=16, d_in=4096, d_out=14336, k=128, dtype="bf16", act="lowrank",
             codes="packed", sqnr=False, graph=True),
        # a ragged decode batch through a down projection: the long contraction, few outputs
        dict(name="decode_27_down", op="layer", n=27, d_in=14336, d_out=4096, k=128, dtype="bf16", act="swiglu",
             codes="packed", sqnr=False, graph=True),
        # a short prompt chunk of odd length, 64-wide blocks
        dict(name="chunk_201_qkv", op="layer", n=201, d_in=4096, d_out=6144, k=64, dtype="bf16", act="lowrank",
             codes="bytes", sqnr=False, graph=False),
        # an ordinary prompt, with the layer's quality measured on the way
        dict(name="prefill_2048_qkv", op="layer", n=2048, d_in=4096, d_out=6144, k=128, dtype="bf16", act="lowrank",
             codes="bytes", sqnr=True, graph=False),
        # an ordinary prompt batch through a down projection
        dict(name="prefill_4096_down", op="layer", n=4096, d_in=14336, d_out=4096, k=128, dtype="bf16", act="swiglu",
             codes="bytes", sqnr=False, graph=False),
        # the largest: a 70B gate/up projection, with its quality
        dict(name="prefill_8192_gateup", op="layer", n=8192, d_in=8192, d_out=28672, k=128, dtype="bf16", act="lowrank",
             codes="bytes", sqnr=True, graph=False),
        # a small float32 layer with packed codes: every launch counts
        dict(name="layer_512_f32", op="layer", n=512, d_in=256, d_out=256, k=32, dtype="f32", act="lowrank",
             codes="packed", sqnr=True, graph=False),
        # 4-bit weights under asymmetric 8-bit activations
        dict(name="w4a8_asym_2048_qkv", op="dp", n=2048, d_in=4096, d_out=6144, k=128, dtype="bf16", act="lowrank",
             bits_x=8, bits_w=4, asym=True),
        # 8 by 8 bits, a ragged batch through a down projection
        dict(name="w8a8_1000_down", op="dp", n=1000, d_in=14336, d_out=4096, k=128, dtype="bf16", act="swiglu",
             bits_x=8, bits_w=8, asym=False),
        # one batch of a calibration run (128 sequences of 2048 tokens come in batches like this)
        dict(name="calib_16384_qkv", op="calib", n=16384, d_in=4096, k=128, dtype="bf16", act="lowrank"),
        # a layer made ready: autocorrelation blocks, the transform, the weights' codes
        dict(name="weights_qkv", op="weights", n=512, d_in=4096, d_out=6144, k=128, dtype="bf16", act="lowrank"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["layer", "layer", "layer", "layer", "dp", "dp", "calib", "weights"])
    act = rng.choice(["lowrank", "swiglu"])
    dtype = "f32" if rng.random() < 0.15 else "bf16"
    k = rng.choice([32, 64, 128, 128, 128, 256])
    unit = max(k, 128)
    d_in = unit * max(1, round(_log_int(rng, 256, 14336) / unit))
    if op == "calib":
        return dict(op=op, n=_log_int(rng, 64, 4096 if dtype == "f32" else 16384), d_in=d_in, k=k, dtype=dtype, act=act)
    if op == "weights":
        k = rng.choice([32, 64, 128])
        d_in = k * max(2, round(_log_int(rng, 256, 4096) / k))
        return dict(op=op, n=512, d_in=d_in, d_out=max(2 * k, _log_int(rng, 256, 6144)), k=k, dtype="bf16", act="lowrank")
    if op == "dp":
        n, d_out = _log_int(rng, 1, 4096), _log_int(rng, 64, 14336)
        n = max(1, min(n, LARGEST // (16 * d_in * d_out)))
        bits_x, bits_w = rng.choice([(4, 4), (8, 4), (6, 6), (8, 8)])
        return dict(op=op, n=n, d_in=d_in, d_out=d_out, k=k, dtype=dtype, act=act, bits_x=bits_x, bits_w=bits_w,
                    asym=rng.random() < 0.5)
    n, d_out = _log_int(rng, 1, 8192), _log_int(rng, 64, 28672)
    if rng.random() < 0.6:
        d_out = 32 * max(2, d_out // 32)
    if dtype == "f32":
        n, d_in = min(n, 2048), min(d_in, 4096)
    n = max(1, min(n, LARGEST // (d_in * d_out)))
    return dict(op=op, n=n, d_in=d_in, d_out=d_out, k=k, dtype=dtype, act=act,
                codes="packed" if n <= 32 or rng.random() < 0.25 else "bytes", sqnr=rng.random() < 0.4,
                graph=n <= 32 and rng.random() < 0.6)


# ---------------------------------------------------------------------------------------------- inputs

DEV = "cuda"


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


class _Tokens:
    """Activations: 64 shared factors plus isotropic noise with 1 % of the channels a hundred times larger, or SiLU(g) u."""

    def __init__(self, case, g):
        self.d, self.act = case["d_in"], case["act"]
        self.dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
        self.F = _randn(g, 64, self.d) / 8.0 if self.act == "lowrank" else None
        self.scale = torch.ones(self.d, device=DEV)
        if self.act == "lowrank":
            self.scale[torch.randperm(self.d, generator=g, device=DEV)[: max(1, self.d // 100)]] = 100.0

    def draw(self, g, n):
        out = torch.empty((n, self.d), dtype=self.dtype, device=DEV)
        for i in range(0, n, 2048):
            m = min(2048, n - i)
            if self.act == "lowrank":
                x = (_randn(g, m, 64) @ self.F + math.sqrt(0.1) * _randn(g, m, self.d)) * self.scale
            else:
                a = _randn(g, m, self.d)
                x = a * torch.sigmoid(a) * _randn(g, m, self.d)
            out[i:i + m] = x.to(self.dtype)
        return out


def _hadamard(k):
    h = torch.ones((1, 1), dtype=torch.float64, device=DEV)
    while h.shape[0] < k:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
    return h / math.sqrt(k)


def _weight_rows(case, g, rows):
    w = 0.02 * _randn(g, rows, case["d_in"])
    if case["act"] == "lowrank":
        w *= torch.exp(0.5 * _randn(g, rows, 1))
    return w


def _transform(case, tokens, g):
    """T_b = H_k M_b with M_b = D^{1/2} (I + S) D^{1/2}: D the k = 1 optimum (E[x_i^2])^{-1/4} up to a common factor,
    S a small symmetric matrix.  float64 [d/k, k, k] and its inverse."""
    k, d = case["k"], case["d_in"]
    power = tokens.draw(g, 256).double().square().mean(0).clamp_min(1e-6)
    root = power.pow(-0.125).view(d // k, k)
    S = _randn(g, d // k, k, k).double() * (0.2 / math.sqrt(k))
    M = torch.eye(k, dtype=torch.float64, device=DEV) + 0.5 * (S + S.transpose(1, 2))
    M = root[:, :, None] * M * root[:, None, :]
    H = _hadamard(k)
    return (H @ M).float(), (torch.linalg.inv(M) @ H.T).float()


def _weight_codes(case, Tinv, g, qmax):
    """Codes int8 [d_out, d_in] of W T^{-1} on the symmetric grid and their steps, made in slices."""
    d_out, d_in, k = case["d_out"], case["d_in"], case["k"]
    q = torch.empty((d_out, d_in), dtype=torch.int8, device=DEV)
    s = torch.empty((d_out,), dtype=torch.float32, device=DEV)
    for i in range(0, d_out, 4096):
        m = min(4096, d_out - i)
        w = _weight_rows(case, g, m)
        wt = torch.bmm(w.view(m, d_in // k, k).transpose(0, 1), Tinv).transpose(0, 1).reshape(m, d_in)
        a = wt.abs().amax(1)
        q[i:i + m] = torch.round(wt * (qmax / a)[:, None]).clamp_(-qmax, qmax).to(torch.int8)
        s[i:i + m] = a / qmax
    return q, s


def _bytes(q):
    """One byte a code or digit, the E4M3 form of q 2^-9: the sign in bit 7, the magnitude below."""
    return ((q < 0).to(torch.uint8) << 7) | q.abs().to(torch.uint8)


def _packed(q):
    """The packed 4-bit form: 8 codes e0..e7 a word; byte i has e_i's magnitude and, in bit 7, sign, and
    e_{4+i}'s magnitude in bits 4-6; bit 3 has the sign of e_{4+(i+3)%4}."""
    rows, d = q.shape
    out = torch.empty((rows, d // 2), dtype=torch.uint8, device=DEV)
    for i in range(0, rows, 4096):
        e = q[i:i + 4096].view(-1, d // 8, 8)
        m, s = e.abs().to(torch.uint8), (e < 0).to(torch.uint8)
        high = torch.roll(s[..., 4:], 1, dims=-1)
        out[i:i + 4096] = (m[..., :4] | (s[..., :4] << 7) | (m[..., 4:] << 4) | (high << 3)).view(-1, d // 2)
    return out


def _digits(q, bits):
    """Digit planes of symmetric codes: d0 = ((q + 8) mod 16) - 8, d1 = (q - d0) / 16, a sign-magnitude byte each."""
    if bits <= 4:
        return _bytes(q)[None].contiguous()
    planes = torch.empty((2,) + tuple(q.shape), dtype=torch.uint8, device=DEV)
    for i in range(0, q.shape[0], 4096):
        v = q[i:i + 4096].to(torch.int16)
        d0 = torch.remainder(v + 8, 16) - 8
        planes[0, i:i + 4096] = _bytes(d0)
        planes[1, i:i + 4096] = _bytes(torch.div(v - d0, 16, rounding_mode="floor"))
    return planes


def _inputs(case, seed):
    """Everything that is an input, as plain tensors: the same for prepare() and exact()."""
    g = _generator(seed)
    tokens = _Tokens(case, g)
    i = {}
    if case["op"] == "calib":
        i["x"] = tokens.draw(g, case["n"])
        return i
    if case["op"] == "weights":
        i["x"] = tokens.draw(g, case["n"])
        i["W"] = _weight_rows(case, g, case["d_out"]).to(torch.bfloat16)
        return i
    qmax = 7 if case["op"] == "layer" else 2 ** (case["bits_w"] - 1) - 1
    i["T"], Tinv = _transform(case, tokens, g)
    i["qw"], i["sw"] = _weight_codes(case, Tinv, g, qmax)
    i["x"] = tokens.draw(g, case["n"])
    if case.get("sqnr"):
        # a full-precision y that the layer's own is near: the codes' product with noise of about -27 dB
        a = torch.bmm(i["x"].float().view(case["n"], -1, case["k"]).transpose(0, 1), i["T"].transpose(1, 2))
        a = a.transpose(0, 1).reshape(case["n"], -1).to(torch.bfloat16)
        y = torch.empty((case["n"], case["d_out"]), dtype=torch.float32, device=DEV)
        for r in range(0, case["d_out"], 4096):
            y[:, r:r + 4096] = (a @ i["qw"][r:r + 4096].to(torch.bfloat16).T).float() * i["sw"][r:r + 4096]
        i["y_ref"] = y
    return i


# ------------------------------------------------------------------------------------------ the passes

def prepare(case, seed):
    i = _inputs(case, seed)
    st = {"case": case, "x": i["x"]}
    if case["op"] == "weights":
        st["W"] = i["W"]
        return st
    if case["op"] == "calib":
        return st
    st["T"], st["sw"] = i["T"], i["sw"]
    if case["op"] == "dp":
        st["w"] = _digits(i["qw"], case["bits_w"])
        st["rowsum"] = i["qw"].sum(1, dtype=torch.int32)
        return st
    st["w"] = _packed(i["qw"]) if case["codes"] == "packed" else _bytes(i["qw"])
    st["planes"] = None
    if case["dtype"] == "bf16" and cat.cat_split_transform_bytes(case["d_in"], case["k"]) > 0:
        st["planes"] = cat.cat_split_transform(st["T"], case["k"])
    st["y_ref"] = i.get("y_ref")
    if case["graph"]:
        st["out"] = _layer(st)                       # loads what the capture will use
        torch.cuda.synchronize()
        st["replay"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(st["replay"]):
            st["out"] = _layer(st)
    return st


def _layer(st):
    case = st["case"]
    if case["codes"] == "packed":
        codes, sx = cat.cat_transform_quantize_act_split(st["x"], st["T"], st["planes"], case["k"])
        linear, linear_sqnr = cat.cat_w4a4_linear, cat.cat_w4a4_linear_sqnr
    else:
        codes, sx = cat.cat_transform_quantize_act_e8(st["x"], st["T"], st["planes"], case["k"])
        linear, linear_sqnr = cat.cat_w4a4_linear_e8, cat.cat_w4a4_linear_sqnr_e8
    if case["sqnr"]:
        y, sums = linear_sqnr(codes, sx, st["w"], st["sw"], st["y_ref"])
        return {"y": y, "sqnr": sums}
    return {"y": linear(codes, sx, st["w"], st["sw"])}


def run(st):
    case = st["case"]
    if case["op"] == "layer":
        if case["graph"]:
            st["replay"].replay()
            return st["out"]
        return _layer(st)
    if case["op"] == "dp":
        planes, sx, zx = cat.cat_transform_quantize_act_dp(st["x"], st["T"], case["k"], case["bits_x"], case["asym"])
        y = cat.cat_linear_dp(planes, case["bits_x"], sx, st["w"], case["bits_w"], st["sw"], x_zero=zx,
                              w_rowsum=st["rowsum"] if case["asym"] else None)
        return {"y": y, "x_scale": sx}
    if case["op"] == "calib":
        return {"sigma": cat.cat_calib_cov(st["x"], case["k"])}
    sigma = cat.cat_calib_cov(st["x"], case["k"])
    T, Wq, sw = cat.cat_quantize_weights(st["W"], case["k"], "cat", sigma_x=sigma, n_calib=case["n"])
    return {"T": T, "Wq": Wq, "w_scale": sw}


def work(case):
    n, d, k = case["n"], case["d_in"], case["k"]
    item = 4 if case["dtype"] == "f32" else 2
    if case["op"] == "calib":
        # the blocks are symmetric: k (k + 1) products a token and block, half of the full square
        return {"bytes": n * d * item + d * k * 8, "flops": n * d * (k + 1)}
    o = case["d_out"]
    if case["op"] == "weights":
        # both autocorrelations, the weights through the inverse blocks; tokens and weights read once
        return {"bytes": n * d * 2 + o * d * 2 + o * d // 2 + d * k * 4 + o * 4,
                "flops": (n + o) * d * (k + 1) + 2 * o * d * k}
    if case["op"] == "dp":
        # x, T, the weights' digit planes and steps in; y out (the activation codes need not leave the chip)
        planes = 1 if case["bits_w"] <= 4 else 2
        products = planes * (1 if case["bits_x"] <= 4 else 2)
        return {"bytes": n * d * item + d * k * 4 + planes * o * d + 4 * o + 4 * n * o,
                "flops": 2 * n * d * k + 2 * products * n * d * o}
    w = o * d // 2 if case["codes"] == "packed" else o * d
    return {"bytes": n * d * item + d * k * 4 + w + 4 * o + 4 * n * o * (2 if case["sqnr"] else 1),
            "flops": 2 * n * d * k + 2 * n * d * o}


def tolerance(case):
    if case["op"] == "calib":
        # float32 sums of exact bf16 products (2e-6 seen over 16384 tokens); float32 rows are summed in pairs of floats
        return {"rel": 1e-5 if case["dtype"] == "bf16" else 1e-10}
    if case["op"] == "weights":
        # T follows the float32 sums through two square roots; a code on a rounding boundary may go either way
        return {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
    # y is exact but for codes that lie on a rounding boundary: x' in float32 moves a 4-bit code in about one of
    # 10^6, an 8-bit code in about one of 10^5 (of a sixteenth of the weight).  Small calls have room for two codes.
    codes = case["n"] * case["d_in"]
    if case["op"] == "dp":
        finer = 7.0 / (2 ** (case["bits_x"] - 1) - 1)          # more codes on boundaries, each of less weight
        return {"rel": min(0.03, 1.5e-3 * math.sqrt(finer) + finer / math.sqrt(codes)), "max": 0.3}
    return {"rel": min(0.03, 1e-3 + 1.0 / math.sqrt(codes)), "max": 0.5}


# ------------------------------------------------------------------------------------------ in 64 bits

def _exact_codes(case, x, T):
    n, d, k = x.shape[0], case["d_in"], case["k"]
    v = torch.bmm(x.double().view(n, d // k, k).transpose(0, 1), T.double().transpose(1, 2))
    v = v.transpose(0, 1).reshape(n, d)
    if case["op"] == "layer" or not case["asym"]:
        qmax = 7 if case["op"] == "layer" else 2 ** (case["bits_x"] - 1) - 1
        a = v.abs().amax(1)
        q = torch.where(a[:, None] > 0, torch.round(qmax * v / a[:, None]), torch.zeros_like(v)).clamp_(-qmax, qmax)
        return q, a / qmax
    N = 2 ** case["bits_x"] - 1
    lo, hi = v.amin(1).clamp_max(0.0), v.amax(1).clamp_min(0.0)
    width = torch.where(hi > lo, hi - lo, torch.ones_like(hi))
    z = torch.round(N * (-lo) / width)
    q = (torch.round(N * v / width[:, None]) + z[:, None]).clamp_(0, N)
    return q - z[:, None], (hi - lo) / N


def _exact_weights(case, i):
    k, d, n = case["k"], case["d_in"], case["n"]

    def blocks(v):
        v = v.double().view(v.shape[0], d // k, k).transpose(0, 1)
        return (v.transpose(1, 2) @ v).cpu().numpy()

    def power(m, p):
        w, u = np.linalg.eigh(0.5 * (m + np.swapaxes(m, 1, 2)))
        return (u * (w ** p)[:, None, :]) @ np.swapaxes(u, 1, 2)

    sx, swt = blocks(i["x"]) / n, blocks(i["W"])
    r, ri = power(swt, 0.5), power(swt, -0.5)
    # Sigma_w # Sigma_x^{-1}, then its square root
    geo = r @ power(ri @ np.linalg.inv(sx) @ ri, 0.5) @ r
    M = torch.from_numpy(power(geo, 0.5)).to(DEV)
    H = _hadamard(k)
    T, Tinv = H @ M, torch.linalg.inv(M) @ H.T
    o = case["d_out"]
    wt = torch.bmm(i["W"].double().view(o, d // k, k).transpose(0, 1), Tinv).transpose(0, 1).reshape(o, d)
    return {"T": T, "Wq": None, "w_scale": wt.abs().amax(1) / 7}


def exact(case, seed):
    i = _inputs(case, seed)
    if case["op"] == "calib":
        n, d, k = case["n"], case["d_in"], case["k"]
        s = torch.zeros((d // k, k, k), dtype=torch.float64, device=DEV)
        for r in range(0, n, 4096):
            v = i["x"][r:r + 4096].double()
            v = v.view(v.shape[0], d // k, k).transpose(0, 1)
            s += v.transpose(1, 2) @ v
        return {"sigma": s}
    if case["op"] == "weights":
        return _exact_weights(case, i)
    n, d, o = case["n"], case["d_in"], case["d_out"]
    y = torch.empty((n, o), dtype=torch.float64, device=DEV)
    wide = torch.float32 if case["op"] == "layer" else torch.float64    # 49 d_in < 2^24: whole numbers are exact
    scales = torch.empty((n,), dtype=torch.float64, device=DEV)
    for t in range(0, n, 2048):
        q, s = _exact_codes(case, i["x"][t:t + 2048], i["T"])
        scales[t:t + 2048] = s
        q = q.to(wide)
        for r in range(0, o, 4096):
            acc = q @ i["qw"][r:r + 4096].to(wide).T
            y[t:t + 2048, r:r + 4096] = acc.double() * s[:, None] * i["sw"][r:r + 4096].double()
    if case["op"] == "dp":
        return {"y": y, "x_scale": scales}
    if not case["sqnr"]:
        return {"y": y}
    signal = noise = 0.0
    for t in range(0, n, 1024):
        ref = i["y_ref"][t:t + 1024].double()
        signal += float(ref.square().sum())
        noise += float((ref - y[t:t + 1024]).square().sum())
    return {"y": y, "sqnr": torch.tensor([signal, noise, 10 * math.log10(signal / noise)], dtype=torch.float64)}
