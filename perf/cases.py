"""The work that is timed when the performance of this library is looked at: calls of the public entry points
at the sizes of the benchmark's configurations, of the GPU tests, and at sizes of the same kind in between.

What a program holds before a call is made by `prepare`: a model's packed weights and scales (as they come
out of a checkpoint), calibrated static grids, a workspace, the activations.  A decode step is held in a CUDA
graph, as a serving loop holds it; longer calls are made eagerly.  `exact` restates the definition in 64-bit
torch; where the path defines a rounding (packed codes, bf16 gate, up, product and hidden state), it rounds there too.
"""
import math

import torch

from paper_2506_04985_b200 import binding as B

DEV = "cuda"
EPS = 1e-5


# ------------------------------------------------------------------------------------------------ cases
def listed():
    def layer(name, m, d, n_qkv, d_ff, parts="attn+mlp", sym=True, hadamard=False, f16=False, graph=False):
        return dict(name=name, kind="layer", parts=parts, m=m, d=d, n_qkv=n_qkv, d_ff=d_ff, sym=sym,
                    hadamard=hadamard, f16=f16, graph=graph)

    return [
        # one small linear called on its own, eagerly: the cost of a call
        dict(name="linear_128x1024", kind="linear", m=128, k=1024, n=1024, bits=4, dynamic=False, sym=True, f16=False,
             scale_input=False, post="none"),
        # a decoder layer's linears in a decode step: one user, a few, a ragged batch, a mixed batch of decode
        # tokens and a short prompt (sizes of the 8B-class model: hidden 4096, QKV 6144, MLP 14336)
        layer("layer_decode_1", 1, 4096, 6144, 14336, f16=True, graph=True),
        layer("layer_decode_8", 8, 4096, 6144, 14336, f16=True, graph=True),
        layer("layer_decode_37", 37, 4096, 6144, 14336, f16=True, graph=True),
        layer("layer_mixed_120", 120, 4096, 6144, 14336, graph=True),
        # the attention half for a prompt: a short ragged one with asymmetric grids, the headline size
        layer("attn_prompt_333_asym", 333, 4096, 6144, 0, parts="attn", sym=False),
        layer("attn_prompt_2048", 2048, 4096, 6144, 0, parts="attn"),
        # the SwiGLU block for a prompt, and with the online Hadamard at the down projection's input
        layer("mlp_prompt_4096", 4096, 4096, 0, 14336, parts="mlp"),
        layer("mlp_prompt_1003_hadamard", 1003, 4096, 0, 14336, parts="mlp", hadamard=True),
        # a 70B-class layer at the largest token count
        layer("layer_70b_8192", 8192, 8192, 10240, 28672),
        # the dynamic grid with 8-bit activation codes, a ragged prompt, plain-linear semantics
        dict(name="linear_a8_dynamic_777", kind="linear", m=777, k=4096, n=6144, bits=8, dynamic=True, sym=True, f16=False,
             scale_input=True, post="inverse"),
        # conversion of a checkpoint: range search and packing of one weight matrix
        dict(name="weights_lp_14336x4096", kind="weights", n=14336, k=4096, range="lp", f16=True),
    ]


def draw(rng):
    def near(lo, hi):                                   # spread over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def mult(lo, hi, of):
        return max(lo, near(lo, hi) // of * of)

    kind = rng.choice(["decode", "decode", "prompt", "prompt", "linear", "linear", "weights"])
    if kind == "weights":
        return dict(kind="weights", n=mult(64, 14336, 8), k=mult(256, 4096, 32), range=rng.choice(["lp", "lp", "minmax"]),
                    f16=rng.random() < 0.5)
    if kind == "linear":
        dynamic = rng.random() < 0.5
        bits = rng.choice([4, 8])
        return dict(kind="linear", m=near(1, 4096), k=mult(256, 8192, 128), n=mult(256, 14336, 8), bits=bits, dynamic=dynamic,
                    sym=dynamic or bits == 8 or rng.random() < 0.6, f16=rng.random() < 0.5, scale_input=rng.random() < 0.5,
                    post=rng.choice(["none", "inverse"]))
    decode = kind == "decode"
    d = mult(1024, 8192, 128)
    parts = rng.choice(["attn+mlp", "attn+mlp", "attn", "mlp"])
    hadamard = "mlp" in parts and rng.random() < 0.3
    d_ff = mult(2048, 28672, 128)
    if hadamard:                                        # groups of 256 .. 4096 channels
        d_ff = max(d_ff // 256, 8) * 256
        d_ff += 256 if d_ff % 8192 == 0 else 0
    return dict(kind="layer", parts=parts, m=near(1, 128) if decode else near(129, 8192), d=d,
                n_qkv=d + 256 * rng.randint(1, 8) if "attn" in parts else 0, d_ff=d_ff if "mlp" in parts else 0,
                sym=rng.random() < 0.7, hadamard=hadamard, f16=rng.random() < 0.5, graph=decode)


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV)


def _activations(g, m, k, gain):
    """Student-t(3) values, 0.5 % of the channels `gain` times larger, tokens of different norms, mean square near 1."""
    x = _randn(g, m, k) * (((_randn(g, m, k) ** 2 + _randn(g, m, k) ** 2 + _randn(g, m, k) ** 2) / 3.0).rsqrt())
    hot = torch.randperm(k, generator=g, device=DEV)[: max(1, k // 200)]
    x[:, hot] *= gain
    x *= torch.exp(0.25 * _randn(g, m, 1)) / math.sqrt(3.0 * (1.0 + gain * gain * max(1, k // 200) / k))
    return x.to(torch.bfloat16)


def _weight(g, n, k, f16):
    """Packed 4-bit codes of a Gaussian matrix on the min-max grid, per-row scales (unit gain; a few large rows), row sums."""
    codes = (_randn(g, n, k) * 1.9).round_().clamp_(-8, 7).to(torch.int8)
    sw = torch.exp(0.1 * _randn(g, n)) / (1.9 * math.sqrt(k))
    sw[torch.rand((n,), generator=g, device=DEV) < 0.002] *= 4.0
    wq = ((codes[:, 0::2] & 15) | (codes[:, 1::2] << 4)).view(torch.uint8)
    return dict(q=wq.contiguous(), sw=sw.to(torch.float16 if f16 else torch.float32), wsum=codes.sum(1, dtype=torch.int32))


def _grid(v, sym):
    """Static grid of a calibration slice v: least sum of |v - v^|^3 over scales up to the min-max one."""
    v = v[:64].double()
    z = 0 if sym else 8
    lo, hi = (-8, 7) if sym else (-z, 15 - z)
    best, scale = math.inf, 1.0
    for i in range(10, 101, 5):
        d = float(v.abs().max()) * i / 100.0 / 7.0
        err = float(((v / d).round().clamp(lo, hi) * d - v).abs().pow(3).sum())
        if err <= best:
            best, scale = err, d
    return B.QParams(4, sym, scale, z)


def _rms_inv(x):
    return 1.0 / torch.sqrt(x.double().square().mean(1, keepdim=True) + EPS)


def _layer_inputs(case, g):
    m, d, n_qkv, d_ff, sym, f16 = (case[k] for k in ("m", "d", "n_qkv", "d_ff", "sym", "f16"))
    s = dict(case=case, x=_activations(g, m, d, 50.0), s_prev=torch.exp(0.25 * _randn(g, m)))
    x = s["x"].double()
    if n_qkv:
        s["a"] = _activations(g, m, d, 10.0)            # what the caller's attention gives back
        s["wqkv"], s["wo"] = _weight(g, n_qkv, d, f16), _weight(g, d, d, f16)
        s["qp_in"] = _grid(x * _rms_inv(x), sym)
        s["qp_ap"] = _grid(s["a"].double() * _rms_inv(x) * s["s_prev"].double()[:, None], sym)
    if d_ff:
        s["wgu"], s["wd"] = _weight(g, 2 * d_ff, d, f16), _weight(g, d, d_ff, f16)
        s["qp_mlp"] = _grid(x * _rms_inv(x), True)
        s["qp_mid"] = B.QParams(4, True, 0.4, 0)
    return s


def _linear_inputs(case, g):
    s = dict(case=case, x=_activations(g, case["m"], case["k"], 40.0), w=_weight(g, case["n"], case["k"], case["f16"]),
             s_in=torch.exp(0.25 * _randn(g, case["m"])) if case["scale_input"] else None)
    v = s["x"].double() * _rms_inv(s["x"]) * (s["s_in"].double()[:, None] if case["scale_input"] else 1.0)
    s["qp"] = _grid(v, case["sym"])
    if case["bits"] == 8 and not case["dynamic"]:
        s["qp"] = B.QParams(8, True, s["qp"].scale / 16.0, 0)
    return s


def prepare(case, seed):
    g = _gen(seed)
    if case["kind"] == "weights":
        w = _randn(g, case["n"], case["k"]) * 0.02
        w[torch.rand((case["n"],), generator=g, device=DEV) < 0.002] *= 20.0
        return dict(case=case, w=w.to(torch.bfloat16))
    if case["kind"] == "linear":
        s = _linear_inputs(case, g)
        s["ws"] = B.new_workspace(B.OP_LINEAR_A8 if case["bits"] == 8 else B.OP_LINEAR, case["m"], case["n"], case["k"])
        return s
    s = _layer_inputs(case, g)
    m, d = case["m"], case["d"]
    if case["n_qkv"]:
        s["ws_attn"] = B.new_workspace(B.OP_LINEAR, m, case["n_qkv"], d)
    if case["d_ff"]:
        s["ws_mlp"] = B.new_workspace(B.OP_MLP_HADAMARD if case["hadamard"] else B.OP_MLP, m, case["d_ff"], d)
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _layer(s)
        torch.cuda.current_stream().wait_stream(side)
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            s["out"] = _layer(s)
    return s


# ------------------------------------------------------------------------------------------------ the call
def _layer(s):
    """The linears of a decoder layer around the caller's attention; both halves add the normalised residual."""
    case, out, x, s_n = s["case"], {}, s["x"], s["s_prev"]
    if case["n_qkv"]:
        w, o = s["wqkv"], s["wo"]
        sums = (None, None) if case["sym"] else (w["wsum"], o["wsum"])
        out["qkv"], s_n, r = B.fpt_decoder_attn_qkv(x, w["q"], w["sw"], s["qp_in"], eps=EPS, s_prev=s_n, wsum=sums[0],
                                                    ws=s["ws_attn"])
        x = B.fpt_decoder_attn_out(s["a"], o["q"], o["sw"], s["qp_ap"], s_n, X=x, r=r, wsum=sums[1], ws=s["ws_attn"])
        out["attn"], out["s_attn"], out["r"] = x, s_n, r
    if case["d_ff"]:
        w, dn = s["wgu"], s["wd"]
        out["mlp"], out["s_mlp"] = B.fpt_decoder_mlp(x, w["q"], w["sw"], dn["q"], dn["sw"], s["qp_mlp"], s["qp_mid"], eps=EPS,
                                                     s_prev=s_n, add_residual=True, mid_hadamard=case["hadamard"],
                                                     ws=s["ws_mlp"])
    return out


def run(s):
    case = s["case"]
    if case["kind"] == "weights":
        return B.fpt_quantize_weights(s["w"], range_mode=B.RANGE_LP if case["range"] == "lp" else B.RANGE_MINMAX, p=3.0,
                                      scale_dtype=torch.float16 if case["f16"] else torch.float32)
    if case["kind"] == "linear":
        w = s["w"]
        flags = B.RMSNORM | (B.SCALE_INPUT if case["scale_input"] else 0)
        post = B.POST_INVERSE_OF_PRE if case["post"] == "inverse" else B.POST_NONE
        if case["dynamic"]:
            return B.fpt_w4a4_linear_dynamic(s["x"], w["q"], w["sw"], bits=case["bits"], flags=flags, eps=EPS, s_in=s["s_in"],
                                             post_mode=post, ws=s["ws"])
        return B.fpt_w4a4_linear(s["x"], w["q"], w["sw"], s["qp"], flags=flags, eps=EPS, s_in=s["s_in"], post_mode=post,
                                 wsum=None if case["sym"] else w["wsum"], ws=s["ws"])
    if case["graph"]:
        s["graph"].replay()
        return s["out"]
    return _layer(s)


# ------------------------------------------------------------------------------------------------ what it costs at least
def work(case):
    wide = 2 if case["f16"] else 4

    def weight(n, k):
        return n * k // 2 + n * wide

    if case["kind"] == "weights":
        n, k = case["n"], case["k"]
        # one candidate costs an element a division, a rounding, two clamps, a product, a difference, a power and an addition
        return {"bytes": n * k * 2 + weight(n, k) + 4 * n, "flops": n * k * (8 * 81 if case["range"] == "lp" else 4)}
    if case["kind"] == "linear":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 2 * m * k + weight(n, k) + 2 * m * n + 4 * m * (2 if case["scale_input"] else 1), "flops": 2 * m * n * k}
    m, d, q, f = case["m"], case["d"], case["n_qkv"], case["d_ff"]
    by, fl = 2 * m * d + 4 * m, 0
    if q:
        by += weight(q, d) + weight(d, d) + 2 * m * (q + d + d) + 8 * m
        fl += 2 * m * d * (q + d)
    if f:
        by += weight(2 * f, d) + weight(d, f) + 2 * m * d + 4 * m
        fl += 6 * m * d * f
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """Whole numbers are defined to the bit.  For bf16 results, four times what the path differs from `exact`: 1.7e-3,
    the bf16 rounding; 6.9e-3 with the dynamic 4-bit grid, where ratios of bf16 values that fall on a tie change a code."""
    if case["kind"] == "weights":
        return "exact"
    return {"rel": 2.5e-2 if case.get("dynamic") and case["bits"] == 4 else 7e-3}


# ------------------------------------------------------------------------------------------------ the definition, in 64 bits
def _bf16(v):
    return v.to(torch.bfloat16).double()


def _codes(v, qp):
    """Codes minus the zero point of values on a static grid; the grid's step is the stored float32 one."""
    inv = float(1.0 / torch.tensor(qp.scale, dtype=torch.float32))
    z, lo, hi = (0, -(1 << (qp.bits - 1)), (1 << (qp.bits - 1)) - 1) if qp.symmetric else (qp.zero_point, 0, 15)
    return (v * inv).round().clamp(lo - z, hi - z)


def _times(c, w):
    """codes [m, k] x packed weight [n, k/2], times the weight's scales; rows in chunks."""
    parts = []
    for i in range(0, w["q"].shape[0], 8192):
        q = w["q"][i:i + 8192].view(torch.int8)
        q = torch.stack(((q << 4) >> 4, q >> 4), 2).flatten(1).double()
        parts.append((c @ q.T) * w["sw"][i:i + 8192].double())
    return torch.cat(parts, 1)


def _hadamard(v):
    m, k = v.shape
    b = k & -k
    h = v.view(m * k // b, b)
    dist = 1
    while dist < b:
        h = h.view(-1, b // (2 * dist), 2, dist)
        h = torch.stack((h[:, :, 0] + h[:, :, 1], h[:, :, 0] - h[:, :, 1]), 2)
        dist *= 2
    return h.reshape(m, k) / math.sqrt(b)


def _exact_layer(case, s):
    out, x, s_n = {}, s["x"].double(), s["s_prev"].double()[:, None]
    if case["n_qkv"]:
        r = _rms_inv(x)
        s_n = s_n * r
        out["qkv"] = _times(_codes(x * r, s["qp_in"]), s["wqkv"]) * s["qp_in"].scale
        y = _times(_codes(s["a"].double() * s_n, s["qp_ap"]), s["wo"]) * s["qp_ap"].scale + x * r
        out["attn"], out["s_attn"], out["r"], x = y, s_n[:, 0], r[:, 0], _bf16(y)
    if case["d_ff"]:
        r = _rms_inv(x)
        s_n = s_n * r
        gu = _bf16(_times(_codes(x * r, s["qp_mlp"]), s["wgu"]) * s["qp_mlp"].scale).view(case["m"], -1, 2, 64)
        mid = _bf16(gu[:, :, 0] * torch.sigmoid(gu[:, :, 0]) * gu[:, :, 1]).flatten(1)
        mid = _hadamard(mid) if case["hadamard"] else mid
        out["mlp"] = _times(_codes(mid * s_n, s["qp_mid"]), s["wd"]) * s["qp_mid"].scale + x * r
        out["s_mlp"] = s_n[:, 0]
    return out


def _exact_weights(case, w):
    def grid(frac):
        d = a * frac / 7.0
        d = d.to(torch.float16).float() if case["f16"] else d
        return torch.where((a == 0) | (d == 0), torch.ones_like(d), d)

    a = w.abs().amax(1).float()
    delta, best = grid(1.0), torch.full_like(a, math.inf, dtype=torch.float64)
    if case["range"] == "lp":
        v = w.double()
        for i in range(20, 101):
            d = grid(torch.tensor(i, dtype=torch.float32, device=DEV) / 100.0)
            q = (w.float() / d[:, None]).round().clamp(-8, 7).double()
            err = (q * d.double()[:, None] - v).abs().pow(3).sum(1)
            take = err <= best
            best, delta = torch.where(take, err, best), torch.where(take, d, delta)
    return None, delta.double(), None


def exact(case, seed):
    g = _gen(seed)
    if case["kind"] == "weights":
        return _exact_weights(case, prepare(case, seed)["w"])
    if case["kind"] == "layer":
        return _exact_layer(case, _layer_inputs(case, g))
    s = _linear_inputs(case, g)
    x = s["x"].double()
    r = _rms_inv(x)
    p = r * s["s_in"].double()[:, None] if case["scale_input"] else r
    if case["dynamic"]:
        hi = (1 << (case["bits"] - 1)) - 1
        step = (x * p).abs().amax(1, keepdim=True) / hi
        codes = (x * p / step).round().clamp(-hi - 1, hi)
    else:
        step, codes = s["qp"].scale, _codes(x * p, s["qp"])
    y = _times(codes, s["w"]) * step
    return (y / p if case["post"] == "inverse" else y), p[:, 0]
