"""GPU parity of the quantise kernels against the oracle: packed codes, scales and row
sums must match bit for bit."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import quantizers as OQ
from paper_2506_04985_b200 import binding as B, synth
from helpers import dev, host, oqp, bf16_host

pytestmark = pytest.mark.gpu


def _acts(M, K, seed, law="student_t3"):
    return synth.activations(M, K, seed, f"x{M}x{K}", law=law, outlier_frac=0.005, outlier_gain=50.0,
                             token_log_std=0.7)


@pytest.mark.parametrize("M,K", [(128, 1024), (37, 4096), (5, 14336), (3, 28672), (130, 128), (2, 32), (9, 8192),
                                 (4, 2048), (1, 65536 - 32)])
@pytest.mark.parametrize("mode", ["norm", "norm_sin", "scale", "norm_scale", "asym"])
def test_act_quant_codes_bit_exact(M, K, mode):
    x = _acts(M, K, 3)
    s_in = synth.per_token_scale(M, 3, "s_in")
    flags = {"norm": B.RMSNORM, "norm_sin": B.RMSNORM, "scale": B.SCALE_INPUT,
             "norm_scale": B.RMSNORM | B.SCALE_INPUT, "asym": B.RMSNORM}[mode]
    use_s = mode in ("norm_sin", "scale", "norm_scale")
    qp = B.QParams(4, mode != "asym", 0.37 if flags & B.RMSNORM else 1.9, 7)
    xq, s_out = B.fpt_act_quant(dev(x), qp, flags, 1e-5, s_in=dev(s_in) if use_s else None)
    codes, so, _, _ = OQ.act_quant(synth.f32(x), oqp(qp), bool(flags & B.RMSNORM), bool(flags & B.SCALE_INPUT),
                                   1e-5, s_in.numpy() if use_s else None)
    assert np.array_equal(host(xq), OQ.pack_int4(codes))
    assert np.array_equal(host(s_out).view(np.uint32), so.view(np.uint32))
    assert len(np.unique(codes)) >= 8 or K < 64        # the grid is actually exercised


@pytest.mark.parametrize("M,K,ld", [(600, 768, 768), (513, 544, 552), (600, 1024, 1024), (1500, 4096, 4096), (777, 8192, 8200), (513, 16384, 16384)])
@pytest.mark.parametrize("mode", ["norm", "scale", "asym"])
def test_act_quant_many_tokens_streaming_kernel(M, K, ld, mode):
    """Enough tokens for the persistent double-buffered kernel: every warp walks over several rows,
    some rows carry Inf / NaN / zeros, rows may be strided."""
    x = torch.zeros((M, ld), dtype=torch.bfloat16)
    x[:, :K] = _acts(M, K, 8)
    x[:, K:] = -777.0
    x[3, :K] = 0.0
    x[M // 2, 11] = float("nan")
    x[M - 1, K - 1] = float("inf")
    s_in = synth.per_token_scale(M, 8, "s_in")
    flags = B.SCALE_INPUT if mode == "scale" else B.RMSNORM
    qp = B.QParams(4, mode != "asym", 0.37 if flags & B.RMSNORM else 1.9, 9)
    xq, s_out = B.fpt_act_quant(dev(x), qp, flags, 1e-5, s_in=dev(s_in), K=K)
    with np.errstate(all="ignore"):
        codes, so, _, _ = OQ.act_quant(synth.f32(x)[:, :K], oqp(qp), bool(flags & B.RMSNORM),
                                       bool(flags & B.SCALE_INPUT), 1e-5, s_in.numpy())
    assert np.array_equal(host(xq), OQ.pack_int4(codes))
    assert np.array_equal(host(s_out), so, equal_nan=True)


def test_act_quant_strided_rows_and_edge_values():
    M, K, ld = 6, 256, 384
    x = torch.zeros((M, ld), dtype=torch.bfloat16)
    x[:, :K] = _acts(M, K, 4)
    x[:, K:] = 1000.0                                # must be ignored
    x[1, :K] = 0.0                                   # zero row: r = 1/sqrt(eps)
    x[2, 5] = float("nan")
    x[3, 7] = float("inf")
    x[4, :K] = 3.0e38                                # squares overflow float32
    x[5, 9] = 3.0e38                                 # finite, but far beyond the exact range of the rounding trick
    x[5, 10] = -3.0e38
    qp = B.QParams(4, True, 0.41, 0)
    xq, s_out = B.fpt_act_quant(dev(x), qp, B.RMSNORM, 1e-6, K=K)
    with np.errstate(all="ignore"):
        codes, so, _, _ = OQ.act_quant(synth.f32(x)[:, :K], oqp(qp), True, False, 1e-6)
    assert np.array_equal(host(xq), OQ.pack_int4(codes))
    assert np.array_equal(host(s_out), so, equal_nan=True)           # NaN payloads may differ
    assert np.isnan(so[2]) and so[3] == 0.0 and so[4] == 0.0


@pytest.mark.parametrize("M,K", [(64, 1024), (7, 14336), (3, 256)])
@pytest.mark.parametrize("inter", [False, True])
def test_silu_mul_quant_bit_exact(M, K, inter):
    g = synth.activations(M, K, 5, "g", law="normal", outlier_frac=0.01, outlier_gain=6.0)
    u = synth.activations(M, K, 5, "u", law="student_t3", outlier_frac=0.0)
    g.view(-1)[:256] = torch.linspace(-90, 90, 256).to(torch.bfloat16)   # exp2 range reduction edges
    s_n = synth.per_token_scale(M, 5, "s_n")
    qp = B.QParams(4, True, 0.23, 0)
    if inter:
        gu = torch.empty((M, 2 * K), dtype=torch.bfloat16)
        gu.view(M, K // 64, 2, 64)[:, :, 0, :] = g.view(M, K // 64, 64)
        gu.view(M, K // 64, 2, 64)[:, :, 1, :] = u.view(M, K // 64, 64)
        xq, _ = B.fpt_act_quant(dev(gu), qp, B.SILU_MUL | B.GU_INTERLEAVED | B.SCALE_INPUT, 0.0, s_in=dev(s_n))
    else:
        xq, _ = B.fpt_act_quant(dev(g), qp, B.SILU_MUL | B.SCALE_INPUT, 0.0, X2=dev(u), s_in=dev(s_n))
    codes, _ = OQ.silu_mul_quant(synth.f32(g), synth.f32(u), oqp(qp), s_n.numpy())
    assert np.array_equal(host(xq), OQ.pack_int4(codes))


# Without the norm a CTA takes several short rows or a part of a long one, with one chunk a thread or more: ragged rows
# a CTA, last CTAs that are nearly empty, rows that end inside a part.
@pytest.mark.parametrize("M,K", [(1, 32), (63, 32), (65, 32), (90001, 32), (25, 96), (30001, 96), (5, 1024), (10007, 1056),
                                 (3, 4064), (3300, 768), (801, 4128), (777, 8192), (301, 8256), (2, 65536), (70, 65536)])
@pytest.mark.parametrize("form", ["plain", "scale_asym", "silu", "gate_up"])
def test_act_quant_without_norm_short_and_long_rows(M, K, form):
    if form == "gate_up" and K % 64:
        pytest.skip("64-column groups")
    g = torch.Generator(device="cuda").manual_seed(M + K)
    x, x2 = (torch.randn((M, K), device="cuda", generator=g).to(torch.bfloat16) for _ in range(2))
    x[M // 2, K // 3], x[M - 1, K - 1] = float("nan"), float("inf")
    s_in = torch.rand((M,), device="cuda", generator=g) + 0.5
    qp = B.QParams(4, form != "scale_asym", 0.31, 7)
    if form == "plain":
        xq, s_out = B.fpt_act_quant(x, qp, 0, s_in=s_in)
    elif form == "scale_asym":
        xq, s_out = B.fpt_act_quant(x, qp, B.SCALE_INPUT, s_in=s_in)
    elif form == "silu":
        xq, s_out = B.fpt_act_quant(x, qp, B.SILU_MUL | B.SCALE_INPUT, X2=x2, s_in=s_in)
    else:
        gu = torch.stack((x.view(M, K // 64, 64), x2.view(M, K // 64, 64)), 2).reshape(M, 2 * K)
        xq, s_out = B.fpt_act_quant(gu, qp, B.SILU_MUL | B.GU_INTERLEAVED | B.SCALE_INPUT, s_in=s_in)
    rows = np.unique(np.r_[0:min(M, 70), M // 2, max(0, M - 70):M])          # the oracle on the first, a middle and the last rows
    xr, x2r, sr = synth.f32(x.cpu()[rows]), synth.f32(x2.cpu()[rows]), host(s_in)[rows]
    with np.errstate(all="ignore"):
        if form in ("silu", "gate_up"):
            codes, _ = OQ.silu_mul_quant(xr, x2r, oqp(qp), sr)
        else:
            codes, _, _, _ = OQ.act_quant(xr, oqp(qp), rmsnorm=False, scale_input=form != "plain", s_in=sr)
    assert np.array_equal(host(xq)[rows], OQ.pack_int4(codes))
    assert torch.equal(s_out, s_in)
    if form in ("plain", "scale_asym"):                                      # every row against torch's own operations
        v = (x.float() * s_in[:, None] if form == "scale_asym" else x.float()) * float(np.float32(1.0) / np.float32(qp.scale))
        lo, hi, z = (0, 15, 7) if form == "scale_asym" else (-8, 7, 0)
        q = torch.where(v.isnan(), torch.full_like(v, lo), (v.round() + z).clamp(lo, hi)).to(torch.int32) & 15
        assert torch.equal(xq.to(torch.int32), q[:, 0::2] | (q[:, 1::2] << 4))


@pytest.mark.parametrize("N,K", [(64, 1024), (33, 4096), (8, 14336), (300, 128)])
@pytest.mark.parametrize("mode", ["minmax32", "minmax16", "lp32", "lp16_f32in"])
def test_weight_quant_bit_exact(N, K, mode):
    w = synth.weights(N, K, 0.02, 6, f"w{N}x{K}", outlier_row_frac=0.02, outlier_row_gain=20.0)
    if N > 2:
        w[2] = 0.0                                    # all-zero row: scale 1
    wf = synth.f32(w)
    sd = torch.float16 if "16" in mode else torch.float32
    rm = B.RANGE_LP if mode.startswith("lp") else B.RANGE_MINMAX
    wd = dev(w).float() if mode.endswith("f32in") else dev(w)
    wq, sw, wsum = B.fpt_quantize_weights(wd, None, rm, 3.0, sd)
    codes, d, ws = OQ.quantize_weights(wf, range_mode=OQ.RANGE_LP if rm else OQ.RANGE_MINMAX, p=3.0,
                                       scale_dtype="fp16" if sd == torch.float16 else "fp32")
    assert np.array_equal(host(sw.float()).view(np.uint32), d.view(np.uint32))
    assert np.array_equal(host(wq), OQ.pack_int4(codes))
    assert np.array_equal(host(wsum), ws)


@pytest.mark.parametrize("K", [32, 1024, 1056, 2080, 4128, 8224])       # either side of each thread count and of a second pass
def test_weight_quant_range_search_at_ties_and_odd_rows(K):
    rng = np.random.default_rng(K)
    w = rng.standard_normal((12, K)).astype(np.float32) * 0.02
    w[0] = rng.integers(-14, 15, K) * 0.5                # quotients that are k + 1/2 on the min-max grid
    w[0, 0] = 7.0
    w[1] = rng.integers(-14, 15, K) * np.float32(0.35)   # ... and on the candidate at 70 %, up to rounding
    w[1, 0] = 7.0
    w[2] *= 1e-6                                         # float16 scales that underflow
    w[3] *= 1e7                                          # ... that overflow
    w[4] *= 1e-37                                        # reciprocals out of range
    w[5, 3] = np.inf
    w[6, 5] = np.nan
    for dt in (torch.bfloat16, torch.float32):
        wd = torch.from_numpy(w).to(dt)
        for sd, name in ((torch.float16, "fp16"), (torch.float32, "fp32")):
            with np.errstate(all="ignore"):
                codes, d, sums = OQ.quantize_weights(wd.float().numpy()[:5], range_mode=OQ.RANGE_LP, p=3.0, scale_dtype=name)
            wq, sw, wsum = B.fpt_quantize_weights(dev(wd), None, B.RANGE_LP, 3.0, sd)
            assert np.array_equal(host(sw.float())[:5].view(np.uint32), d.view(np.uint32))
            assert np.array_equal(host(wq)[:5], OQ.pack_int4(codes))
            assert np.array_equal(host(wsum)[:5], sums)
            # an infinite row has no finite candidate, a NaN compares with none: both keep the min-max step
            assert np.isinf(host(sw.float())[5])
            finite = wd.float().numpy()[6]
            want = np.float32(np.nanmax(np.abs(finite))) / np.float32(7.0)
            assert host(sw.float())[6] == (np.float32(np.float16(want)) if name == "fp16" else want)
            assert host(wq)[6, 2] >> 4 == 8              # a NaN takes the lowest code


@pytest.mark.parametrize("K", [992, 1216, 1248, 2080, 4096, 14336])     # either side of the rows whose magnitudes are counted
def test_weight_quant_range_search_keeps_the_least_error(K):
    """Rows on which the float32 screening of the candidates could go wrong: many equal errors, one sign, magnitudes at
    the ends of what is counted, scales at the end of float16."""
    rng = np.random.default_rng(K + 1)
    w = rng.standard_normal((16, K)) * 0.02
    w[0] = rng.choice([-1.0, 1.0], K)                    # one magnitude: the errors of many candidates are nearly alike
    w[1] = np.abs(w[1])
    w[2] = -np.abs(w[2])
    w[3] = rng.integers(-8, 9, K) * 0.125                # a grid point of several candidates, both ends in use
    w[4] = np.exp2(rng.uniform(-9, 0, K)) * rng.choice([-1.0, 1.0], K)      # every octave down to where all codes are 0
    w[5], w[5, 7] = 0.0, 1.0                             # zeros but for one value
    w[6, 11] = 40.0                                      # everything else far below the least step
    w[7] = rng.uniform(-1, 1, K)
    w[8] = -0.0 * w[8]
    w[9] *= 0.004 / 0.08                                 # float16 scales around the least ordinary one
    w[10] *= 1e-5
    w[11] = rng.choice([-1.0, 1.0], K) * (1.0 + rng.integers(0, 128, K) / 128)      # one octave
    w[12] = rng.integers(-14, 15, K) * 0.5
    for dt in (torch.bfloat16, torch.float32):
        wd = torch.from_numpy(w.astype(np.float32)).to(dt)
        for sd, name in ((torch.float16, "fp16"), (torch.float32, "fp32")):
            codes, d, sums = OQ.quantize_weights(wd.float().numpy(), range_mode=OQ.RANGE_LP, p=3.0, scale_dtype=name)
            wq, sw, wsum = B.fpt_quantize_weights(dev(wd), None, B.RANGE_LP, 3.0, sd)
            assert np.array_equal(host(sw.float()).view(np.uint32), d.view(np.uint32))
            assert np.array_equal(host(wq), OQ.pack_int4(codes))
            assert np.array_equal(host(wsum), sums)


def test_weight_quant_range_search_of_a_row_without_end():
    """A row of 33 million values, a pattern of 1024 over and over, with two candidates whose errors differ by 1e-10: float32
    sums from chunk to chunk are 5e-4 off, each in its own way, and the screening dropped the right one."""
    pattern = np.random.default_rng(2).standard_normal(1024) * 0.02
    pattern[:64] *= 1.463646882039535
    pattern[100] = 0.08
    pattern = pattern.astype(np.float32)
    codes, d, sums = OQ.quantize_weights(pattern[None], range_mode=OQ.RANGE_LP, p=3.0)
    times = 1 << 15
    wq, sw, wsum = B.fpt_quantize_weights(dev(pattern).repeat(times)[None], None, B.RANGE_LP, 3.0)
    assert np.array_equal(host(sw), d.astype(np.float32)) and int(host(wsum)[0]) == int(sums[0]) * times
    assert torch.equal(wq.view(times, 512), dev(OQ.pack_int4(codes)).expand(times, 512))


@pytest.mark.parametrize("K", [32, 64, 96, 160, 1056, 4096, 4128, 8224])       # 1 to 33 values a thread, remainders
@pytest.mark.parametrize("p", [2.0, 2.4, 0.7])
def test_weight_quant_range_search_with_a_general_power(K, p):
    rng = np.random.default_rng(K)
    w = (rng.standard_normal((9, K)) * 0.02).astype(np.float32)
    w[0] = rng.integers(-14, 15, K) * 0.5                # ties
    w[1] = 0.0
    w[2] *= 1e7                                          # float16 scales that overflow
    w[3, 0] = 3.0                                        # one large value
    for dt in (torch.bfloat16, torch.float32):
        wd = torch.from_numpy(w).to(dt)
        for sd, name in ((torch.float16, "fp16"), (torch.float32, "fp32")):
            with np.errstate(all="ignore"):
                codes, d, sums = OQ.quantize_weights(wd.float().numpy(), range_mode=OQ.RANGE_LP, p=p, scale_dtype=name)
            wq, sw, wsum = B.fpt_quantize_weights(dev(wd), None, B.RANGE_LP, p, sd)
            assert np.array_equal(host(sw.float()).view(np.uint32), d.view(np.uint32))
            assert np.array_equal(host(wq), OQ.pack_int4(codes))
            assert np.array_equal(host(wsum), sums)


@pytest.mark.parametrize("M", [1, 37, 600])
@pytest.mark.parametrize("K", [96, 256, 1024, 1536, 4096, 8192, 14336, 32768])
def test_per_token_scale_in_place(M, K):
    """s_out == s_in: every thread of a token has to see the scale as it was before the call."""
    g = torch.Generator(device="cuda").manual_seed(K + M)
    x = torch.randn((M, K), device="cuda", generator=g).to(torch.bfloat16)
    s_in = torch.exp(torch.randn((M,), device="cuda", generator=g))
    qp, q8, both = B.QParams(4, True, 0.3, 0), B.QParams(8, True, 0.02, 0), B.RMSNORM | B.SCALE_INPUT
    ref = [B.fpt_act_quant(x, qp, both, s_in=s_in), B.fpt_act_quant(x, qp, B.SCALE_INPUT, s_in=s_in),
           B.fpt_act_quant(x, q8, both, s_in=s_in), B.fpt_act_quant_dynamic(x, 4, both, s_in=s_in)]
    L, delta = B.lib(), torch.empty((M,), device="cuda")
    for _ in range(5):
        for i, (codes, s_out) in enumerate(r[:2] for r in ref):
            s, out = s_in.clone(), torch.empty_like(codes)
            if i < 3:
                rc = L.fpt_act_quant(B._stream(), B._ptr(x), M, K, K, ctypes.byref((qp, qp, q8)[i]), (both, B.SCALE_INPUT, both)[i],
                                     1e-5, None, B._ptr(s), B._ptr(out), B._ptr(s))
            else:
                rc = L.fpt_act_quant_dynamic(B._stream(), B._ptr(x), M, K, K, 4, both, 1e-5, B._ptr(s), B._ptr(out), B._ptr(s),
                                             B._ptr(delta))
            assert rc == B.OK
            assert torch.equal(s, s_out) and torch.equal(out, codes)


def test_interleave_gate_up_layout():
    d_ff, K = 384, 256
    rng = np.random.default_rng(0)
    g = torch.from_numpy(rng.integers(0, 256, (d_ff, K // 2), dtype=np.uint8))
    u = torch.from_numpy(rng.integers(0, 256, (d_ff, K // 2), dtype=np.uint8))
    sg = torch.from_numpy(rng.standard_normal(d_ff).astype(np.float32))
    su = torch.from_numpy(rng.standard_normal(d_ff).astype(np.float32))
    wgu, sw = B.fpt_interleave_gate_up(dev(g), dev(u), dev(sg), dev(su))
    wgu, sw = host(wgu), host(sw)
    for r in range(d_ff // 64):
        assert np.array_equal(wgu[128 * r:128 * r + 64], g[64 * r:64 * r + 64].numpy())
        assert np.array_equal(wgu[128 * r + 64:128 * r + 128], u[64 * r:64 * r + 64].numpy())
        assert np.array_equal(sw[128 * r:128 * r + 64], sg[64 * r:64 * r + 64].numpy())
        assert np.array_equal(sw[128 * r + 64:128 * r + 128], su[64 * r:64 * r + 64].numpy())


def _rows_with_products_that_round_to_a_tie(scale, n_rows, K, seed):
    """Per-token multipliers p and bf16 inputs for which (x * p) * (1/D) is exactly k + 1/2 after its
    two roundings while the unrounded product is not: a kernel that contracts the second multiply
    with anything that follows takes the other code there.  Found by search over all bf16 values."""
    rng = np.random.default_rng(seed)
    F = np.float32
    inv = F(1.0) / F(scale)
    vals = np.arange(0x3C00, 0x4300, dtype=np.uint32)                       # bf16 patterns of about 0.008 .. 128
    xs = (vals << 16).view(F)
    rows, ps, hits = [], [], 0
    while len(rows) < n_rows:
        cand = np.exp(rng.uniform(-3.0, 0.5, 4096)).astype(F)                # many multipliers at once
        v = (xs[None, :] * cand[:, None]).astype(F)
        u = (v * inv).astype(F)
        tie = (np.abs(u) < 8) & (u - np.floor(u) == F(0.5))
        off = v.astype(np.float64) * np.float64(inv) != u.astype(np.float64)
        good = tie & off
        for i in np.nonzero(good.any(axis=1))[0]:
            if len(rows) == n_rows:
                break
            sel = xs[good[i]]
            row = rng.choice(xs, K).astype(F) * rng.choice([-1, 1], K).astype(F)
            row[:sel.size] = sel
            row[sel.size:2 * sel.size] = -sel
            hits += 2 * sel.size
            rows.append(row)
            ps.append(cand[i])
    return np.stack(rows), np.array(ps, dtype=F), hits


@pytest.mark.parametrize("K", [256, 4096])
def test_act_quant_products_that_round_to_a_tie(K):
    scale = 0.62
    x, p, hits = _rows_with_products_that_round_to_a_tie(scale, 60, K, 9)
    assert hits >= 100
    x, p = np.tile(x, (10, 1)), np.tile(p, 10)           # 600 tokens: enough for the many-token kernels
    xb = synth.to_bf16(x)
    qp = B.QParams(4, True, scale, 0)
    for M in (600, 24):                                  # the many-token and the few-token kernels
        xq, _ = B.fpt_act_quant(dev(xb[:M]), qp, B.SCALE_INPUT, 0.0, s_in=dev(torch.from_numpy(p[:M])))
        codes, _, _, _ = OQ.act_quant(synth.f32(xb[:M]), oqp(qp), False, True, 0.0, p[:M])
        assert np.array_equal(host(xq), OQ.pack_int4(codes))
