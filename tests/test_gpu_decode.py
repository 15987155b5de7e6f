"""GPU parity of the decode-size matmul (at most 64 tokens; weights streamed once, work split
evenly over the SMs, partial sums added as integers) against the oracle: int32 accumulators
bit-exact, bf16 outputs identical."""
import numpy as np
import pytest
import torch

from oracle.int_matmul import int_matmul
from oracle.epilogue import dequant_epilogue
from paper_2506_04985_b200 import binding as B
from helpers import dev, host, bf16_host, random_codes, packed_dev, assert_bf16_close

pytestmark = pytest.mark.gpu


def _run(M, N, K, symmetric=True, z=0, seed=0, post=False, residual=False, f16=True, ws=None, reps=1):
    rng = np.random.default_rng(seed + 7 * M + N + K)
    qa = random_codes(rng, (M, K), symmetric)
    qw = random_codes(rng, (N, K), True)
    sw = (np.exp(rng.standard_normal(N)) * 0.01).astype(np.float16 if f16 else np.float32)
    act_scale = np.float32(0.311)
    pv = np.exp(rng.standard_normal(M)).astype(np.float32) if post else None
    res = rs = None
    if residual:
        res = torch.from_numpy(rng.standard_normal((M, N)).astype(np.float32)).to(torch.bfloat16)
        rs = np.exp(rng.standard_normal(M)).astype(np.float32)
    wsum = qw.astype(np.int64).sum(axis=1).astype(np.int32)
    ref_acc = int_matmul(qa, qw, z)
    rres = (res.float().numpy() * rs[:, None]).astype(np.float32) if residual else None
    ref_y = dequant_epilogue(ref_acc, sw.astype(np.float32), act_scale, pv, rres)
    xa, xw, xs = packed_dev(qa), packed_dev(qw), dev(sw)
    for _ in range(reps):          # the same workspace again: its tile counters must be back at zero
        Y, acc = B.fpt_w4a4_gemm(xa, xw, xs, float(act_scale), wsum=None if symmetric else dev(wsum),
                                 act_symmetric=symmetric, act_zero_point=z, post=None if pv is None else dev(pv),
                                 residual=None if res is None else dev(res), res_scale=None if rs is None else dev(rs),
                                 want_acc=True, ws=ws)
        assert np.array_equal(host(acc), ref_acc), f"int32 accumulators differ {M}x{N}x{K}"
        assert assert_bf16_close(bf16_host(Y), ref_y, f"Y {M}x{N}x{K}") == 0
    if ws is not None:
        assert B.fpt_check_status(ws) == B.OK


@pytest.mark.parametrize("M", [1, 2, 8, 16, 17, 32, 33, 64])
@pytest.mark.parametrize("N,K", [(128, 128), (264, 512), (1024, 2048), (72, 384)])
def test_decode_shapes(M, N, K):
    _run(M, N, K)


@pytest.mark.parametrize("M", [1, 8, 32, 64])
@pytest.mark.parametrize("N,K", [(14336, 4096), (4096, 14336)])
def test_decode_llama_mlp_shapes_full_size(M, N, K):
    """Decode configuration: every output of the full-size launch is checked."""
    _run(M, N, K, seed=3)


@pytest.mark.parametrize("M,N,K", [(8, 520, 1024), (64, 4096, 1024), (40, 1032, 256)])
@pytest.mark.parametrize("z", [8, 15])
def test_decode_asymmetric_activations(M, N, K, z):
    _run(M, N, K, symmetric=False, z=z)


def test_decode_post_residual_and_f32_scales():
    _run(24, 1024, 1024, post=True)
    _run(64, 2048, 512, post=True, residual=True, f16=False)
    _run(3, 136, 256, residual=True)


def test_decode_same_workspace_many_launches():
    M, N, K = 64, 4096, 2048
    ws = B.new_workspace(B.OP_GEMM, M, N, K)
    _run(M, N, K, ws=ws, reps=5)
    _run(9, 8192, 1024, ws=B.new_workspace(B.OP_GEMM, 9, 8192, 1024), reps=3)


def test_decode_extreme_codes_and_long_k():
    M, N, K = 64, 264, 28672
    qa = np.full((M, K), -8, dtype=np.int8)
    qw = np.full((N, K), -8, dtype=np.int8)
    qw[1::2] = 7
    sw = np.full(N, 2.0 ** -10, dtype=np.float32)
    _, acc = B.fpt_w4a4_gemm(packed_dev(qa), packed_dev(qw), dev(sw), 1.0, want_acc=True, want_y=False)
    acc = host(acc)
    assert np.all(acc[:, 0::2] == 64 * K) and np.all(acc[:, 1::2] == -56 * K)


def test_decode_few_tokens_and_many_rows():
    """The kernel for up to 16 tokens, which has no tiles to count, at 4000 strips of sixteen rows."""
    _run(8, 64000, 128, seed=11)


@pytest.mark.parametrize("M,N,K", [(20, 64000, 512), (33, 64000, 768), (17, 254080, 128)])
def test_decode_counters_of_many_tiles(M, N, K):
    """500 tiles whose ranges are cut (a counter byte per tile and lane quadrant), twice on one workspace; 1985 tiles,
    more than there are counters."""
    _run(M, N, K, seed=12, ws=B.new_workspace(B.OP_GEMM, M, N, K), reps=2)


@pytest.mark.parametrize("M,K,residual", [(17, 384, True), (37, 384, False), (64, 128, False), (40, 256, True)])
def test_decode_more_tiles_than_counters(M, K, residual):
    """Ranges of whole tiles, the last one shorter (1993 tiles in 143 ranges of 14), the last tile ragged."""
    N = 255016
    _run(M, N, K, symmetric=residual, z=0 if residual else 9, seed=13, post=True, residual=residual,
         ws=B.new_workspace(B.OP_GEMM, M, N, K))


@pytest.mark.parametrize("M,N,K,what", [
    (40, 8192, 2048, "64 tiles cut in 2: clusters of two CTAs"),
    (33, 2048, 4096, "16 tiles cut in 8: clusters of eight CTAs"),
    (64, 4096, 2048, "32 tiles cut in 4, asymmetric grid and residual below"),
    (64, 1024, 8192, "8 tiles cut in 16 ranges: no cluster that size, partial sums through the scratch slots"),
    (20, 1152, 1280, "9 tiles, 5 k-blocks: ranges that do not end on tile boundaries")])
def test_decode_split_tiles_cluster_and_slot_paths(M, N, K, what):
    """Few tiles and long rows: every tile is cut into ranges whose partial sums are exchanged through a
    cluster's shared memory (2, 4, 8 CTAs) or through scratch slots; twice on one workspace."""
    ws = B.new_workspace(B.OP_GEMM, M, N, K)
    _run(M, N, K, seed=21, ws=ws, reps=2)
    _run(M, N, K, symmetric=False, z=9, seed=22, post=True, residual=True, f16=False, ws=ws, reps=2)


@pytest.mark.parametrize("M", [65, 80, 113, 128])
@pytest.mark.parametrize("N,K", [(1024, 8192), (4096, 14336)])
def test_decode_65_to_128_tokens_in_two_launches(M, N, K):
    """Few outputs and long rows: 64 tokens and the rest, the second launch on offset operands."""
    _run(M, N, K, seed=31, f16=False)
    _run(M, N, K, symmetric=False, z=9, seed=32, post=True, residual=True)


def _every_output_every_time(calls, outs, want, nbytes):
    """`calls[i]` writes outs[i] from operands of its own; all of them in a graph, whose replays find nothing they need
    in L2 (the operands are larger than twice that, `nbytes` in all): tiles arrive late and out of order."""
    assert nbytes >= 2 * torch.cuda.get_device_properties(0).L2_cache_size
    for c in calls:
        c()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for c in calls:
            c()
    for _ in range(30):
        for y in outs:
            y.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(y, w) for y, w in zip(outs, want))


def _sets_for(weight_bytes):
    return max(9, 2 * torch.cuda.get_device_properties(0).L2_cache_size // weight_bytes + 1)


def _signed(q):
    return torch.stack(((q.view(torch.int8) << 4) >> 4, q.view(torch.int8) >> 4), 2).flatten(1).double()


@pytest.mark.parametrize("M,N,K,form", [
    (37, 4096, 14336, "sym"), (64, 14336, 4096, "sym"), (37, 28672, 4096, "sym"), (120, 4096, 14336, "sym"),
    (2048, 6144, 4096, "sym"), (37, 6144, 4096, "asym"), (333, 6144, 4096, "asym"), (200, 6144, 4096, "a8"),
    (777, 6144, 4096, "a8")])
def test_launches_in_a_row_give_every_output_every_time(M, N, K, form):
    """One launch by itself, with a slow epilogue, hides a converter that runs ahead."""
    g = torch.Generator(device="cuda").manual_seed(5)
    calls, outs, want, states = [], [], [], []
    n = _sets_for(N * K // 2)
    for _ in range(n):
        xw = torch.randint(0, 256, (N, K // 2), dtype=torch.uint8, device="cuda", generator=g)
        sw = torch.rand((N,), device="cuda", generator=g)
        y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
        w = _signed(xw)
        ws = B.new_workspace(B.OP_GEMM_A8 if form == "a8" else B.OP_GEMM, M, N, K)
        if form == "a8":
            xa = torch.randint(-128, 128, (M, K), dtype=torch.int8, device="cuda", generator=g)
            a = xa.double()
            calls.append(lambda xa=xa, xw=xw, sw=sw, ws=ws, y=y: B.fpt_w4a8_gemm(xa, xw, sw, 0.3, ws=ws, Y=y))
        else:
            xa = torch.randint(0, 256, (M, K // 2), dtype=torch.uint8, device="cuda", generator=g)
            sym = form == "sym"
            a = _signed(xa) if sym else torch.stack((xa & 15, xa >> 4), 2).flatten(1).double() - 8
            wsum = None if sym else w.sum(1).to(torch.int32)
            calls.append(lambda xa=xa, xw=xw, sw=sw, ws=ws, y=y, sym=sym, wsum=wsum: B.fpt_w4a4_gemm(
                xa, xw, sw, 0.3, wsum=wsum, act_symmetric=sym, act_zero_point=0 if sym else 8, ws=ws, Y=y))
        outs.append(y)
        want.append(((a @ w.T).float() * sw * torch.tensor(0.3)).to(torch.bfloat16))
        states.append(ws)
    _every_output_every_time(calls, outs, want, n * N * K // 2)
    assert all(B.fpt_check_status(ws) == B.OK for ws in states)


@pytest.mark.parametrize("M,N,K,sym", [(120, 4096, 4096, True), (333, 6144, 4096, False), (777, 6144, 4096, True), (777, 6144, 4096, False)])
def test_output_projections_in_a_row_give_every_output_every_time(M, N, K, sym):
    """The same for composed calls on one-byte codes with a residual: two pairs a tile, one tile a pair, several."""
    g = torch.Generator(device="cuda").manual_seed(8)
    calls, outs, want = [], [], []
    n = _sets_for(N * K // 2)
    qp = B.QParams(4, sym, 0.4, 0 if sym else 8)
    ws = B.new_workspace(B.OP_LINEAR, M, N, K)
    for _ in range(n):
        a, x = (torch.randn((M, k), device="cuda", generator=g).to(torch.bfloat16) for k in (K, N))
        s_n, r = (torch.rand((M,), device="cuda", generator=g) + 0.5 for _ in range(2))
        xw = torch.randint(0, 256, (N, K // 2), dtype=torch.uint8, device="cuda", generator=g)
        sw = torch.rand((N,), device="cuda", generator=g) * 0.01
        y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
        w, aq = _signed(xw), B.fpt_act_quant(a, qp, B.SCALE_INPUT, s_in=s_n)[0]
        codes = _signed(aq) if sym else torch.stack((aq & 15, aq >> 4), 2).flatten(1).double() - 8
        want.append(((codes @ w.T).float() * sw * torch.tensor(0.4) + x.float() * r[:, None]).to(torch.bfloat16))
        wsum = None if sym else w.sum(1).to(torch.int32)
        calls.append(lambda a=a, x=x, s_n=s_n, r=r, xw=xw, sw=sw, y=y, wsum=wsum: B.fpt_decoder_attn_out(
            a, xw, sw, qp, s_n, X=x, r=r, wsum=wsum, ws=ws, Y=y))
        outs.append(y)
    _every_output_every_time(calls, outs, want, n * N * K // 2)
    assert B.fpt_check_status(ws) == B.OK


@pytest.mark.parametrize("M,d,d_ff,hadamard", [(16, 4096, 3584, False), (520, 4096, 3584, False), (520, 4096, 3584, True)])
def test_blocks_in_a_row_give_every_output_every_time(M, d, d_ff, hadamard):
    """The same for the MLP block, whose gate||up matmul has the SwiGLU epilogues; against its parts, one by one."""
    g = torch.Generator(device="cuda").manual_seed(6)
    calls, outs, want, states = [], [], [], []
    n = _sets_for(3 * d * d_ff // 2)
    qi, qm = B.QParams(4, True, 0.4, 0), B.QParams(4, True, 0.3, 0)
    for _ in range(n):
        x = torch.randn((M, d), device="cuda", generator=g).to(torch.bfloat16)
        wgu, wd = (torch.randint(0, 256, s, dtype=torch.uint8, device="cuda", generator=g) for s in ((2 * d_ff, d // 2), (d, d_ff // 2)))
        sgu, sd = (torch.rand((k,), device="cuda", generator=g) * 0.01 for k in (2 * d_ff, d))
        y = torch.empty((M, d), dtype=torch.bfloat16, device="cuda")
        ws = B.new_workspace(B.OP_MLP_HADAMARD if hadamard else B.OP_MLP, M, d_ff, d)
        xq, s_n = B.fpt_act_quant(x, qi, B.RMSNORM)
        torch.cuda.synchronize()
        gu = ((_signed(xq) @ _signed(wgu).T).float() * sgu * torch.tensor(0.4)).to(torch.bfloat16)
        form = B.SILU_MUL | B.GU_INTERLEAVED | B.SCALE_INPUT
        mq = B.fpt_hadamard_quant(gu, qm, form, s_in=s_n) if hadamard else B.fpt_act_quant(gu, qm, form, s_in=s_n)[0]
        torch.cuda.synchronize()
        want.append(((_signed(mq) @ _signed(wd).T).float() * sd * torch.tensor(0.3)).to(torch.bfloat16))
        assert mq.unique().numel() >= 64
        calls.append(lambda x=x, wgu=wgu, sgu=sgu, wd=wd, sd=sd, ws=ws, y=y: B.fpt_decoder_mlp(
            x, wgu, sgu, wd, sd, qi, qm, want_s_out=False, ws=ws, Y=y, mid_hadamard=hadamard))
        outs.append(y)
        states.append(ws)
    _every_output_every_time(calls, outs, want, n * 3 * d * d_ff // 2)
    assert all(B.fpt_check_status(ws) == B.OK for ws in states)
