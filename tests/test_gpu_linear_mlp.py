"""GPU parity of the composed entry points (one W4A4 linear; one SwiGLU MLP block) against
the oracle, on the paper-shaped synthetic configurations."""
import numpy as np
import pytest
import torch

from oracle import quantizers as OQ, linear as OL
from oracle.int_matmul import int_matmul
from oracle.epilogue import dequant_epilogue
from paper_2506_04985_b200 import binding as B, fold, synth
from helpers import dev, host, oqp, bf16_host, assert_bf16_close
from tile_rules import wt_ahead, wt_cut

pytestmark = pytest.mark.gpu


def _calibrated_scale(calib, eps=1e-5):
    """Static activation scale from a calibration batch (L_3 range setting), harness side."""
    c = synth.f32(calib)
    r = OQ.rms_reciprocal(c, eps)
    return float(OQ.calibrate_static_scale(c * r[:, None], OQ.QParams()))


def test_config1_single_linear_full_parity():
    """128 tokens x 1024 -> 1024, 1 % outlier channels x40, static scale from a seeded
    256-token batch, RMSNorm-derived per-token scale undone after the matmul."""
    M, K, N = 128, 1024, 1024
    x = synth.activations(M, K, 0, "cfg1/x", law="normal", outlier_frac=0.01, outlier_gain=40.0)
    calib = synth.activations(256, K, 0, "cfg1/calib", law="normal", outlier_frac=0.01, outlier_gain=40.0)
    # both batches share their outlier channels: same seed and a name-independent channel draw is not
    # needed for parity, the scale is an input to both sides
    w = synth.weights(N, K, 0.02, 0, "cfg1/w")
    qp = B.QParams(4, True, _calibrated_scale(calib), 0)
    wq, sw, _ = B.fpt_quantize_weights(dev(w))
    cw, d, _ = OQ.quantize_weights(synth.f32(w))
    assert np.array_equal(host(wq), OQ.pack_int4(cw)) and np.array_equal(host(sw), d)
    Y, s_out = B.fpt_w4a4_linear(dev(x), wq, sw, qp, B.RMSNORM, 1e-5, post_mode=B.POST_INVERSE_OF_PRE)
    ref = OL.w4a4_linear(synth.f32(x), cw, d, oqp(qp), True, False, 1e-5, None, OL.POST_INVERSE_OF_PRE)
    assert np.array_equal(host(s_out), ref["s_out"])
    assert assert_bf16_close(bf16_host(Y), ref["y"], "cfg1 Y") == 0
    # and the result is a usable approximation of the unquantised linear
    fp = synth.f32(x).astype(np.float64) @ synth.f32(w).astype(np.float64).T
    assert np.linalg.norm(bf16_host(Y) - fp) / np.linalg.norm(fp) < 0.5


@pytest.mark.parametrize("post_mode", [B.POST_NONE, B.POST_VECTOR])
@pytest.mark.parametrize("flags", [B.RMSNORM, B.SCALE_INPUT, B.RMSNORM | B.SCALE_INPUT])
def test_linear_flag_and_post_combinations(flags, post_mode):
    M, K, N = 70, 512, 264
    x = synth.activations(M, K, 1, "lin/x", law="student_t3", outlier_frac=0.01, outlier_gain=30.0)
    w = synth.weights(N, K, 0.02, 1, "lin/w")
    s_in = synth.per_token_scale(M, 1, "lin/s")
    post = synth.per_token_scale(M, 1, "lin/post")
    qp = B.QParams(4, False, 0.5 if flags & B.RMSNORM else 2.5, 8)
    wq, sw, wsum = B.fpt_quantize_weights(dev(w), scale_dtype=torch.float16)
    cw, d, _ = OQ.quantize_weights(synth.f32(w), scale_dtype="fp16")
    Y, s_out = B.fpt_w4a4_linear(dev(x), wq, sw, qp, flags, 1e-5, s_in=dev(s_in), post_mode=post_mode,
                                 post=dev(post), wsum=wsum)
    ref = OL.w4a4_linear(synth.f32(x), cw, d, oqp(qp), bool(flags & B.RMSNORM), bool(flags & B.SCALE_INPUT), 1e-5,
                         s_in.numpy(), post_mode, post.numpy())
    assert np.array_equal(host(s_out), ref["s_out"])
    assert assert_bf16_close(bf16_host(Y), ref["y"], "Y") == 0


def _mlp_case(M, d, d_ff, seed, with_prev, residual, f16=False):
    x = synth.activations(M, d, seed, "mlp/x", law="student_t3", outlier_frac=0.005, outlier_gain=50.0)
    wg = synth.weights(d_ff, d, 0.02, seed, "mlp/wg")
    wu = synth.weights(d_ff, d, 0.02, seed, "mlp/wu")
    wd = synth.weights(d, d_ff, 0.02, seed, "mlp/wd")
    s_prev = synth.per_token_scale(M, seed, "mlp/s") if with_prev else None
    xf = synth.f32(x)
    (cg, sg, _), (cu, su, _), (cd, sd, _) = (OQ.quantize_weights(synth.f32(w), scale_dtype="fp16" if f16 else "fp32")
                                             for w in (wg, wu, wd))
    # static scales from the data itself (harness side, float64)
    r = OQ.rms_reciprocal(xf, 1e-5)
    d_in = float(OQ.calibrate_static_scale(xf[:64] * r[:64, None], OQ.QParams()))
    qp_in = B.QParams(4, True, d_in, 0)
    pre = OL.decoder_mlp(xf[:32], cg, sg, cu, su, cd, sd, oqp(qp_in), OQ.QParams(4, True, 1.0), 1e-5,
                         None if s_prev is None else s_prev.numpy()[:32])
    sn = pre["s_out"]
    d_mid = float(OQ.calibrate_static_scale(pre["m"] * sn[:, None], OQ.QParams()))
    qp_mid = B.QParams(4, True, d_mid, 0)
    (gq, gs, _), (uq, us, _), (dq, ds, _) = (B.fpt_quantize_weights(dev(w), scale_dtype=torch.float16 if f16 else torch.float32)
                                             for w in (wg, wu, wd))
    wgu, swgu = B.fpt_interleave_gate_up(gq, uq, gs, us)
    Y, s_out = B.fpt_decoder_mlp(dev(x), wgu, swgu, dq, ds, qp_in, qp_mid, 1e-5,
                                 None if s_prev is None else dev(s_prev), residual)
    ref = OL.decoder_mlp(xf, cg, sg, cu, su, cd, sd, oqp(qp_in), oqp(qp_mid), 1e-5,
                         None if s_prev is None else s_prev.numpy(), residual)
    return Y, s_out, ref


@pytest.mark.parametrize("M,d,d_ff,with_prev,residual", [(96, 256, 512, True, True), (130, 512, 1408, False, False),
                                                         (33, 1024, 3584, True, False), (300, 1024, 3584, True, True),
                                                         (513, 256, 640, False, True)])
def test_decoder_mlp_parity(M, d, d_ff, with_prev, residual):
    Y, s_out, ref = _mlp_case(M, d, d_ff, 2, with_prev, residual)
    assert np.array_equal(host(s_out), ref["s_out"])
    assert len(np.unique(ref["mq"])) >= 8
    assert assert_bf16_close(bf16_host(Y), ref["y"], "mlp Y") == 0


# At most 16 tokens: 8 or 16 token columns, many warps a strip below 600 strips (d_ff < 4800); one k-block (d = 128).
@pytest.mark.parametrize("M,d,d_ff", [(1, 128, 128), (1, 1024, 3584), (2, 128, 4864), (7, 256, 4864), (8, 512, 1408),
                                      (9, 256, 4864), (16, 1024, 3584)])
@pytest.mark.parametrize("f16", [False, True])
def test_decoder_mlp_parity_of_a_few_tokens(M, d, d_ff, f16):
    Y, s_out, ref = _mlp_case(M, d, d_ff, 2, True, f16, f16)
    assert np.array_equal(host(s_out), ref["s_out"])
    assert len(np.unique(ref["mq"])) >= 8
    assert assert_bf16_close(bf16_host(Y), ref["y"], "mlp Y") == 0


@pytest.mark.parametrize("M", [1, 7, 8, 9, 16, 33, 130])
@pytest.mark.parametrize("d_ff,hadamard", [(640, False), (4864, False), (4864, True)])
def test_decoder_mlp_equals_its_parts_with_infinities_and_nans(M, d_ff, hadamard):
    """Whichever kernel forms the products: the codes are those of the separate gate||up matmul and SwiGLU quantiser,
    also where weight scales, per-token scales or activations are infinite, NaN, zero or at the ends of the range."""
    d = 256
    g = torch.Generator(device="cuda").manual_seed(M + d_ff)
    wgu, wd = (torch.randint(0, 256, s, dtype=torch.uint8, device="cuda", generator=g) for s in ((2 * d_ff, d // 2), (d, d_ff // 2)))
    sgu, sd = (torch.rand((n,), device="cuda", generator=g) * 0.05 for n in (2 * d_ff, d))
    odd = torch.tensor([float("inf"), float("nan"), 0.0, 3e38, 1e-40, -0.02], device="cuda")
    s_prev = torch.rand((M,), device="cuda", generator=g) + 0.5
    x = torch.randn((M, d), device="cuda", generator=g).to(torch.bfloat16)
    for special in (False, True):
        if special:
            sgu[5::97] = odd.repeat(2 * d_ff)[: sgu[5::97].numel()]
            s_prev[M // 2:] = odd.repeat(M)[: M - M // 2]
            x[M // 3, 3], x[M - 1, 5] = float("inf"), float("nan")
        qi, qm = B.QParams(4, True, 0.4, 0), B.QParams(4, True, 0.7, 0)
        Y, s_out = B.fpt_decoder_mlp(x, wgu, sgu, wd, sd, qi, qm, 1e-5, s_prev, mid_hadamard=hadamard)
        xq, s_n = B.fpt_act_quant(x, qi, B.RMSNORM, 1e-5, s_in=s_prev)
        gu, _ = B.fpt_w4a4_gemm(xq, wgu, sgu, qi.scale)
        form = B.SILU_MUL | B.GU_INTERLEAVED | B.SCALE_INPUT
        mq = B.fpt_hadamard_quant(gu, qm, form, s_in=s_n) if hadamard else B.fpt_act_quant(gu, qm, form, s_in=s_n)[0]
        ref, _ = B.fpt_w4a4_gemm(mq, wd, sd, qm.scale)
        assert torch.equal(s_out.view(torch.int32), s_n.view(torch.int32))
        assert torch.equal(Y.view(torch.int16), ref.view(torch.int16))
        assert special or mq.unique().numel() >= 16


@pytest.mark.parametrize("M", [1, 8, 16, 37, 64, 100, 300])
def test_weights_written_by_the_kernel_in_front(M):
    """The composed calls may request weights before they wait for the kernel in front of them: not before the kernel that
    writes those weights, just before the call on the same stream, has finished."""
    d, d_ff = 2048, 8192
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((M, d), device="cuda", generator=g).to(torch.bfloat16)
    wgu, wd = (torch.randint(0, 256, s, dtype=torch.uint8, device="cuda", generator=g) for s in ((2 * d_ff, d // 2), (d, d_ff // 2)))
    sgu, sd = torch.full((2 * d_ff,), 0.01, device="cuda"), torch.full((d,), 0.01, device="cuda")
    qi, qm = B.QParams(4, True, 0.4, 0), B.QParams(4, True, 0.05, 0)
    ws, wl = B.new_workspace(B.OP_MLP, M, d_ff, d), B.new_workspace(B.OP_LINEAR, M, 2 * d_ff, d)

    outs = [(torch.empty((M, d), dtype=torch.bfloat16, device="cuda"), torch.empty((M, 2 * d_ff), dtype=torch.bfloat16, device="cuda"))
            for _ in range(22)]
    for i, (mlp, linear) in enumerate(outs):
        wait = torch.cuda.synchronize if i < 2 else (lambda: None)       # the first two: what comes out with nothing running
        for step in (lambda: wd.bitwise_xor_(0xA5), lambda: wgu.bitwise_xor_(0x5A),
                     lambda: B.fpt_decoder_mlp(x, wgu, sgu, wd, sd, qi, qm, want_s_out=False, ws=ws, Y=mlp),
                     lambda: wgu.bitwise_xor_(0x0F),
                     lambda: B.fpt_w4a4_linear(x, wgu, sgu, qi, want_s_out=False, ws=wl, Y=linear),
                     lambda: wgu.bitwise_xor_(0x0F)):
            step()
            wait()
    torch.cuda.synchronize()
    assert not any(torch.equal(a, b) for a, b in zip(*outs[:2]))
    for i, out in enumerate(outs):
        assert all(torch.equal(y, w) for y, w in zip(out, outs[i % 2])), i


def test_config2_attention_projections_sampled():
    """Llama-3-8B-shaped projections at 2048 tokens: full launch on the GPU, the oracle
    checks sampled rows (first/last rows of several tiles) over all columns."""
    M, K = 2048, 4096
    x = synth.activations(M, K, 0, "cfg2/x", law="student_t3", outlier_frac=0.005, outlier_gain=50.0)
    rows = np.array([0, 1, 127, 128, 129, 1023, 1024, 1919, 1920, 2047])
    xf = synth.f32(x)
    r = OQ.rms_reciprocal(xf[:256], 1e-5)
    qp = B.QParams(4, True, float(OQ.calibrate_static_scale(xf[:256] * r[:, None], OQ.QParams())), 0)
    xd = dev(x)
    # the mergeable transforms are folded into the weights offline, in float64, before quantisation
    raw = {n: synth.f32(synth.weights(N, K, 0.02, 0, "cfg2/w" + n)).astype(np.float64)
           for n, N in (("q", 4096), ("k", 1024), ("v", 1024), ("o", 4096))}
    phi, s = synth.tk_params(8, 128, 0, "cfg2/tk")
    fq, fk = fold.fold_pre_rope(raw["q"], raw["k"], phi, s, 8, 128, "half")
    fv, fo = fold.fold_value(raw["v"], raw["o"], synth.tv_params(8, 128, 0, "cfg2/tv"), 8, 128)
    folded = {"q": fq, "k": fk, "v": fv, "o": fo}
    for name, N in (("q", 4096), ("k", 1024), ("v", 1024)):
        w = synth.to_bf16(folded[name])
        wq, sw, _ = B.fpt_quantize_weights(dev(w))
        cw, d, _ = OQ.quantize_weights(synth.f32(w))
        Y, s_out = B.fpt_w4a4_linear(xd, wq, sw, qp, B.RMSNORM, 1e-5)
        ref = OL.w4a4_linear(xf[rows], cw, d, oqp(qp), True, False, 1e-5)
        assert np.array_equal(host(s_out)[rows], ref["s_out"])
        assert assert_bf16_close(bf16_host(Y)[rows], ref["y"], "cfg2 " + name) == 0
    # output projection: its input is the attention output, scaled per token by S_n before the grid
    ao = synth.activations(M, K, 0, "cfg2/ao", law="student_t3", outlier_frac=0.005, outlier_gain=50.0)
    s_in = synth.per_token_scale(M, 0, "cfg2/s_in")
    aof = synth.f32(ao)
    qp_o = B.QParams(4, True, 0.75, 0)       # a grid fine enough that all 16 codes occur (the L_3 grid of
                                             # these outlier-heavy activations uses only three of them)
    w = synth.to_bf16(folded["o"])
    wq, sw, _ = B.fpt_quantize_weights(dev(w))
    cw, d, _ = OQ.quantize_weights(synth.f32(w))
    Y, s_out = B.fpt_w4a4_linear(dev(ao), wq, sw, qp_o, B.SCALE_INPUT, 1e-5, s_in=dev(s_in))
    ref = OL.w4a4_linear(aof[rows], cw, d, oqp(qp_o), False, True, 1e-5, s_in.numpy()[rows])
    assert len(np.unique(ref["codes"])) >= 8
    assert assert_bf16_close(bf16_host(Y)[rows], ref["y"], "cfg2 o") == 0


@pytest.mark.parametrize("M,d,n_q,n_kv,with_prev,residual,symmetric",
                         [(96, 256, 256, 64, True, True, True), (300, 1024, 1024, 256, True, True, True),
                          (33, 512, 512, 128, False, False, True), (513, 256, 256, 128, True, True, False),
                          (1, 1024, 1024, 256, True, True, False), (8, 1024, 1024, 256, True, True, True),
                          (9, 512, 512, 128, False, False, True), (16, 512, 512, 128, True, True, False)])
def test_decoder_attention_projections_parity(M, d, n_q, n_kv, with_prev, residual, symmetric):
    """fpt_decoder_attn_qkv -> (an attention stand-in on the host) -> fpt_decoder_attn_out against the
    oracle's two halves on the same values: codes-derived outputs, S_n and r bit-exact."""
    seed = 5
    x = synth.activations(M, d, seed, "attn/x", law="student_t3", outlier_frac=0.005, outlier_gain=50.0)
    wqkv = synth.weights(n_q + 2 * n_kv, d, 0.02, seed, "attn/wqkv")
    wo = synth.weights(d, n_q, 0.02, seed, "attn/wo")
    s_prev = synth.per_token_scale(M, seed, "attn/s") if with_prev else None
    xf = synth.f32(x)
    cqkv, sqkv, wsum_qkv = OQ.quantize_weights(synth.f32(wqkv))
    co, so, wsum_o = OQ.quantize_weights(synth.f32(wo))
    r = OQ.rms_reciprocal(xf, 1e-5)
    if symmetric:
        qp_in = B.QParams(4, True, float(OQ.calibrate_static_scale(xf[:64] * r[:64, None], OQ.QParams())), 0)
    else:
        qp_in = B.QParams(4, False, 0.3, 7)
    wq_d, sw_d, ws_d = B.fpt_quantize_weights(dev(wqkv), want_wsum=not symmetric)
    wo_d, swo_d, wso_d = B.fpt_quantize_weights(dev(wo), want_wsum=not symmetric)
    xd = dev(x)
    QKV, s_n, r_out = B.fpt_decoder_attn_qkv(xd, wq_d, sw_d, qp_in, 1e-5, None if s_prev is None else dev(s_prev),
                                             wsum=ws_d)
    ref1 = OL.decoder_attn_qkv(xf, cqkv, sqkv, oqp(qp_in), 1e-5, None if s_prev is None else s_prev.numpy())
    assert np.array_equal(host(s_n), ref1["s_out"]) and np.array_equal(host(r_out), ref1["r"])
    assert len(np.unique(ref1["xq"])) >= 8
    assert assert_bf16_close(bf16_host(QKV), ref1["qkv"], "attn QKV") == 0
    # stand-in for the caller's attention: any bf16 [M, n_q] tensor computed from QKV will do for parity;
    # a causal running mean of the value heads keeps it data-dependent
    qkv = bf16_host(QKV)
    v = qkv[:, n_q + n_kv:]
    run = np.cumsum(v.astype(np.float64), axis=0) / np.arange(1, M + 1)[:, None]
    a = synth.to_bf16(np.tile(run, (1, n_q // n_kv)) + 0.25 * qkv[:, :n_q])
    af = synth.f32(a)
    if symmetric:
        qp_ap = B.QParams(4, True, float(OQ.calibrate_static_scale(af[:64] * ref1["s_out"][:64, None], OQ.QParams())), 0)
    else:
        qp_ap = B.QParams(4, False, float(np.abs(af * ref1["s_out"][:, None]).max() / 7.5), 8)
    Y = B.fpt_decoder_attn_out(dev(a), wo_d, swo_d, qp_ap, s_n, xd if residual else None, r_out if residual else None,
                               wsum=wso_d)
    ref2 = OL.decoder_attn_out(af, co, so, oqp(qp_ap), ref1["s_out"], xf if residual else None,
                               ref1["r"] if residual else None)
    assert len(np.unique(ref2["aq"])) >= 6
    assert assert_bf16_close(bf16_host(Y), ref2["y"], "attn Y") == 0


@pytest.mark.parametrize("M", [65, 96, 97, 129, 161, 250, 333, 900])     # tiles of 32 to 160 tokens, the last one ragged
@pytest.mark.parametrize("K,N", [(128, 264), (384, 1032), (1024, 4096), (4224, 520)])     # half a weight stage, odd k-blocks, two pairs a tile
@pytest.mark.parametrize("sym", [True, False])
def test_linear_with_widened_codes_equals_the_one_with_packed_codes(M, K, N, sym):
    """A workspace of FPT_OP_LINEAR bytes has room for widened codes, one without that room takes the packed route: the same
    exact integers, so the same bits.  Guard bands around every buffer (helpers) catch a store outside."""
    g = torch.Generator(device="cuda").manual_seed(M + K + N)
    x = torch.randn((M, K), device="cuda", generator=g).to(torch.bfloat16)
    w = torch.randint(0, 256, (N, K // 2), device="cuda", generator=g, dtype=torch.uint8)
    sw = (torch.rand((N,), device="cuda", generator=g) + 0.5).to(torch.float16)
    codes = torch.stack(((w.view(torch.int8) << 4) >> 4, w.view(torch.int8) >> 4), 2)
    wsum = codes.sum((1, 2), dtype=torch.int32)
    qp = B.QParams(4, sym, 0.4, 0 if sym else 7)
    wide = B.new_workspace(B.OP_LINEAR, M, N, K)
    packed = 8192 + (M * K // 2 + 255) // 256 * 256 + (M * 4 + 255) // 256 * 256
    assert wide.numel() > packed
    out = []
    for ws in (wide, wide[:packed].clone()):
        assert B.lib().fpt_reset_status(B._stream(), B._ptr(ws)) == B.OK
        out.append(B.fpt_w4a4_linear(x, w, sw, qp, B.RMSNORM, 1e-5, post_mode=B.POST_INVERSE_OF_PRE, wsum=wsum, ws=ws))
        assert B.fpt_check_status(ws) == B.OK
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


def _signed(q):
    return torch.stack(((q.view(torch.int8) << 4) >> 4, q.view(torch.int8) >> 4), 2).flatten(1)


def _room(M, N, K, wide):
    """A workspace of a linear with room for codes of one byte each, or for packed ones only."""
    ws = B.new_workspace(B.OP_LINEAR, M, N, K)
    if not wide:
        ws = ws[:8192 + (M * K // 2 + 255) // 256 * 256 + (M * 4 + 255) // 256 * 256].clone()
    return ws


# tokens of a tile; whether two CTA pairs share a tile, a pair has one tile or several; every last tile is ragged
@pytest.mark.parametrize("M,N,K,tokens,tiles", [
    (65, 264, 384, 32, "one"), (65, 264, 4096, 32, "shared"), (100, 512, 4096, 32, "shared"), (130, 10248, 384, 64, "many"),
    (517, 264, 4096, 64, "shared"), (65, 10248, 384, 96, "one"), (65, 20488, 384, 96, "many"), (517, 6152, 384, 128, "many"),
    (97, 5128, 4096, 128, "shared"), (130, 14344, 384, 160, "one"), (130, 6152, 4096, 160, "shared"), (777, 6144, 4096, 160, "many"),
    (333, 6152, 2176, 192, "one"), (517, 10248, 2048, 192, "many"), (400, 8200, 2048, 224, "one"), (400, 14344, 2048, 224, "many"),
    (700, 5128, 4096, 256, "one"), (500, 14344, 4096, 256, "many"),
    (70, 8, 1024, None, None), (300, 64, 2048, None, None), (1000, 128, 4096, None, None)])          # few outputs
def test_every_tile_of_one_byte_codes_equals_the_packed_route(M, N, K, tokens, tiles):
    """Both grids with a per-token factor, the dynamic grid, and the output projection with its residual, which the tiles of
    a launch fetch and hand on to one another in the slabs that they leave through."""
    cut = wt_cut(M, N, K)
    assert all(wt_ahead(M, N, K, extras) for extras in (0, 1, 2))
    assert tokens is None or (cut.tokens, "shared" if cut.shared else "one" if cut.tiles <= 74 else "many") == (tokens, tiles)
    g = torch.Generator(device="cuda").manual_seed(M + K + N)
    x = torch.randn((M, K), device="cuda", generator=g).to(torch.bfloat16)
    res = torch.randn((M, N), device="cuda", generator=g).to(torch.bfloat16)
    s_n, r = (torch.rand((M,), device="cuda", generator=g) + 0.5 for _ in range(2))
    w = torch.randint(0, 256, (N, K // 2), device="cuda", generator=g, dtype=torch.uint8)
    sw = torch.rand((N,), device="cuda", generator=g) * 0.01 + 0.005
    wsum = _signed(w).sum(1, dtype=torch.int32)
    for qp in (B.QParams(4, True, 0.4, 0), B.QParams(4, False, 0.4, 7)):
        z = None if qp.symmetric else wsum
        out = []
        for wide in (True, False):
            ws = _room(M, N, K, wide)
            calls = [lambda: B.fpt_w4a4_linear(x, w, sw, qp, B.RMSNORM, 1e-5, post_mode=B.POST_INVERSE_OF_PRE, wsum=z, ws=ws)[0],
                     lambda: B.fpt_w4a4_linear(x, w, sw, qp, B.RMSNORM, 1e-5, wsum=z, ws=ws)[0],
                     lambda: B.fpt_decoder_attn_out(x, w, sw, qp, s_n, X=res, r=r, wsum=z, ws=ws)]
            if qp.symmetric:
                calls.append(lambda: B.fpt_w4a4_linear_dynamic(x, w, sw, 4, B.RMSNORM, 1e-5, ws=ws)[0])
            out.append([c() for c in calls])
            assert B.fpt_check_status(ws) == B.OK
        assert all(torch.equal(a, b) for a, b in zip(*out))
        assert all(float(y.float().abs().max()) > 0.01 for y in out[0])


@pytest.mark.parametrize("M,N,K", [(66, 264, 34944), (66, 264, 35072), (66, 264, 65408), (130, 264, 35072), (130, 264, 65408),
                                   (300, 14344, 35072)])         # the last: several tiles a pair, one accumulator
def test_one_byte_codes_at_the_accumulator_bound(M, N, K):
    """Code - z = +-15 against weights of -8 and 7: from K = 34953 on |acc| passes 2^22, where the conversion to float needs
    another form; on the symmetric grid -8 and 7 against them stay below 2^22 up to the longest rows."""
    assert wt_ahead(M, N, K, 1)
    w = torch.full((N, K // 2), 0x88, dtype=torch.uint8, device="cuda")
    w[1::2] = 0x77
    qw = np.where(np.arange(N) % 2, 7, -8).astype(np.int64)
    sw = (2.0 ** -20 * (1.0 + (np.arange(N) % 61) / 64.0)).astype(np.float32)
    one = torch.ones((M,), device="cuda")
    sign = np.where(np.arange(M) % 3, 1, -1)
    x = torch.from_numpy(np.tile(1000.0 * sign[:, None], (1, K)).astype(np.float32)).to(torch.bfloat16).cuda()
    for z in (None, 0, 15):
        qp = B.QParams(4, z is None, 1.0, z or 0)
        ws = _room(M, N, K, True)
        Y, _ = B.fpt_w4a4_linear(x, w, dev(sw), qp, B.SCALE_INPUT, 0.0, s_in=one,
                                 wsum=None if z is None else dev((qw * K).astype(np.int32)), ws=ws)
        assert B.fpt_check_status(ws) == B.OK
        code = np.where(sign > 0, 7, -8) if z is None else np.where(sign > 0, 15, 0) - z
        acc = code[:, None] * (qw * K)[None]
        assert assert_bf16_close(bf16_host(Y), dequant_epilogue(acc.astype(np.int32), sw, np.float32(1.0)), "Y") == 0


@pytest.mark.parametrize("M", [17, 33, 48, 49, 128])
def test_large_block_of_17_to_128_tokens_equals_its_parts(M):
    """From 32 Mi weights a matrix on, the products of 17 tokens and more are quantised in the epilogue of gate||up."""
    d, d_ff = 4096, 8192
    g = torch.Generator(device="cuda").manual_seed(M)
    x = torch.randn((M, d), device="cuda", generator=g).to(torch.bfloat16)
    wgu, wd = (torch.randint(0, 256, s, dtype=torch.uint8, device="cuda", generator=g) for s in ((2 * d_ff, d // 2), (d, d_ff // 2)))
    sgu, sd = (torch.rand((n,), device="cuda", generator=g) * 0.01 for n in (2 * d_ff, d))
    s_prev = torch.rand((M,), device="cuda", generator=g) + 0.5
    qi, qm = B.QParams(4, True, 0.4, 0), B.QParams(4, True, 0.3, 0)
    Y, s_out = B.fpt_decoder_mlp(x, wgu, sgu, wd, sd, qi, qm, 1e-5, s_prev, True)
    xq, s_n = B.fpt_act_quant(x, qi, B.RMSNORM, 1e-5, s_in=s_prev)
    _, r = B.fpt_act_quant(x, qi, B.RMSNORM, 1e-5)
    gu = ((_signed(xq).double() @ _signed(wgu).double().T).float() * sgu * torch.tensor(0.4)).to(torch.bfloat16)
    mq, _ = B.fpt_act_quant(gu, qm, B.SILU_MUL | B.GU_INTERLEAVED | B.SCALE_INPUT, s_in=s_n)
    y = (_signed(mq).double() @ _signed(wd).double().T).float() * sd * torch.tensor(0.3) + x.float() * r[:, None]
    assert torch.equal(s_out, s_n) and mq.unique().numel() >= 64
    assert torch.equal(Y, y.to(torch.bfloat16))


@pytest.mark.parametrize("M", [49, 64, 65, 100, 129, 300])
def test_mlp_block_that_writes_over_its_input_equals_the_one_that_does_not(M):
    """With Y apart from X the codes of the input may lie in Y until the down projection; with Y = X they may not."""
    d, dff = 512, 1152
    g = torch.Generator(device="cuda").manual_seed(M)
    x = torch.randn((M, d), device="cuda", generator=g).to(torch.bfloat16)
    wgu = torch.randint(0, 256, (2 * dff, d // 2), device="cuda", generator=g, dtype=torch.uint8)
    wd = torch.randint(0, 256, (d, dff // 2), device="cuda", generator=g, dtype=torch.uint8)
    sg, sd = torch.rand((2 * dff,), device="cuda", generator=g) * 0.02, torch.rand((d,), device="cuda", generator=g) * 0.02
    qi, qm = B.QParams(4, True, 0.4, 0), B.QParams(4, True, 0.3, 0)
    y, s = B.fpt_decoder_mlp(x, wgu, sg, wd, sd, qi, qm, 1e-5, None, True)
    over = x.clone()
    y2, s2 = B.fpt_decoder_mlp(over, wgu, sg, wd, sd, qi, qm, 1e-5, None, True, Y=over)
    assert torch.equal(y, y2) and torch.equal(s, s2)
