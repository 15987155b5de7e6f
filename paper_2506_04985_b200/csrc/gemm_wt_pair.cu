// Steps (2)+(3) of the path where the activation codes come one byte each: widened 4-bit codes (code * 16, the order of
// `widen_word`) that the quantiser in front left that way, or 8-bit codes.  Packed-INT4 weights x int8 activations with an
// exact INT32 accumulator (App. J "Setup") and the floating-point scale factors applied after it (App. B "Static
// quantization"), on CTA pairs.
//
// Why this shape: what bounds the kernel that widens both operands (gemm_w4a4_2cta.cu) is the converters' chain and the
// shared-memory pipe: per k-block of 128 codes and CTA 16 KB of packed tiles in, 16 KB out to the converters, 16 KB of
// int8 weights in again and 16 KB to the tensor core, 512 transfers of 128 bytes for 512 cycles of MMA.  Here the sides
// are swapped: the 256 WEIGHT rows of a tile are the M side, widened in registers and written to TENSOR memory, and the
// tokens are the N side, brought by TMA as the swizzled K-major tile the tensor core reads, without passing through any
// thread: 8 KB of packed weights and 16 KB of activations in, 8 KB to the converters, 16 KB to the tensor core = 384
// transfers, half of the conversion work, and one hand-over per k-block in place of two.
//   * the token side of a tile is any multiple of 32 up to 256 (the host picks it), the last tile of a column takes only
//     the tokens there are, and with up to 128 tokens there are two accumulators and more stages;
//   * a k-block (tokens in shared memory, widened weights in tensor memory) has one place and one set of barriers, the
//     MMA's commit frees both; the packed weights have a ring of their own, which runs ahead;
//   * where there are few tiles, two pairs (a cluster of four CTAs) share one, half of the k-blocks each, and exchange
//     partial sums through their shared memory, each finishing half of the tokens.
//
// Roles per CTA (24 warps):
//   warps 0, 2, 3 TMA producers of the weights and of the tokens (two that take the k-blocks in turns: the loop of one took
//                 330 cycles a k-block, and that was the pace of tiles up to 128 tokens)
//   warp 1        tensor-memory owner; in the leader CTA of a pair also the MMA issuer
//   warps 4..15   weight converters, three groups of four warps that take the k-blocks in turns (one row per thread)
//   warps 16..23  epilogue: the accumulator holds a weight row per lane and a token per column; tcgen05.ld in the
//                 16x256b form gives a warp 8 x 8 fragments, which stmatrix.trans stores as rows of a token; the tile
//                 leaves by TMA store, a residual tile arrives by TMA in the same slabs (ldmatrix.trans reads it back).
//                 SwiGLU forms: the gate and up values of a token lie in the two slabs, a thread takes eight at a time.
#include <cuda.h>

#include "fpt_internal.cuh"
#include "quant_math.cuh"

namespace fpt {
namespace wt {

constexpr int RT = kWtRows;                // weight rows of a CTA pair's tile
constexpr int HR = 128;                    // weight rows of a CTA
constexpr int TOK = kWtTokens;             // tokens of a tile at most
constexpr int BK = 128;                    // codes per k-block
constexpr int WK = kWtStage;               // codes per weight stage: rows of 128 packed bytes (see Layout)
constexpr int W_ROW = WK / 2;
constexpr int kWStageCols = BK / 4;        // 32 tensor-memory columns hold 128 int8 per lane
constexpr int kTmemCols = 512;
constexpr int kMaxStages = 12, kMaxW = 6;
constexpr int kGroups = 3;                 // converter groups of four warps
constexpr int kTokProducers = 2;           // warps that ask for tokens
constexpr int kConvWarp0 = 4, kEpiWarp0 = kConvWarp0 + 4 * kGroups, kEpiWarps = 8;
constexpr int kThreads = 32 * (kEpiWarp0 + kEpiWarps);
// Registers per thread: what the CTA is launched with, and what the roles trade it into (warps 0-3, the converter groups,
// epilogue).  A CTA can only redistribute what it owns: an increase that the decreases do not cover would never return.
constexpr int kRegsLaunch = 80, kRegsCtl = 40, kRegsConv = 40, kRegsEpi = 160;
static_assert(kThreads * kRegsLaunch <= 65536, "launch allocation exceeds the register file");
static_assert(128 * (kRegsCtl + kGroups * kRegsConv) + 32 * kEpiWarps * kRegsEpi <= kThreads * kRegsLaunch,
              "the warpgroups ask for more registers than the CTA was launched with: setmaxnreg.inc would never return");

// What a launch makes of a CTA's shared and tensor memory: a ring of k-blocks (tokens in shared memory, widened weights in
// tensor memory) and a ring of packed weights in steps of two k-blocks (rows of 128 bytes).
// A barrier's wait tells one phase from the next by its parity only, so whoever waits for a phase must know that the one
// before it is over: with lengths that are multiples of the number of converter groups a place in either ring belongs to
// the same group (two groups) every time, and these have themselves waited for the phase before.
struct Layout {
  int tn;                                  // tokens of a tile, a multiple of 32
  int nbuf;                                // accumulators of tn tensor-memory columns
  int ns;                                  // k-blocks in flight
  int nw;                                  // weight stages in flight
  static constexpr int kWStage = HR * W_ROW;                        // 16 KB
  // fixed part at the head: per-token factors of two tiles, barriers, tensor-memory base and abort flag
  static constexpr int kVecOff = 0;
  static constexpr int kBarOff = kVecOff + 2 * 2 * TOK * 4;
  static constexpr int kNumBars = 3 * kMaxStages + 2 * kMaxW + 4 + 5 * 2;
  static constexpr int kMiscOff = kBarOff + kNumBars * 8;
  static constexpr int kXOff = 5 * 1024;
  static_assert(kMiscOff + 16 <= kXOff, "the fixed part overlaps the stages");
  __host__ __device__ constexpr int x_stage() const { return tn / 2 * BK; }    // the CTA's half of the tokens, 128-byte rows
  __host__ __device__ constexpr int slab() const { return tn * 128; }          // output: 2 slabs of tn tokens x 64 features, bf16
  __host__ __device__ constexpr int w_off() const { return kXOff + ns * x_stage(); }
  __host__ __device__ constexpr int stg_off() const { return w_off() + nw * kWStage; }
  __host__ __device__ constexpr int alloc() const { return stg_off() + 2 * slab() + 1024; }    // (slack to align the base to 1024)
  __host__ __device__ constexpr int acc_col(int b) const { return b * tn; }
  __host__ __device__ constexpr int w_col(int s) const { return kTmemCols - (ns - s) * kWStageCols; }
};
__host__ __device__ constexpr Layout layout_of(int tn) {
  return tn > 192 ? Layout{tn, 1, 6, 3} : tn > kWtDouble ? Layout{tn, 1, 6, 6} : tn > 64 ? Layout{tn, 2, 6, 6} : Layout{tn, 2, 12, 6};
}
constexpr bool layouts_fit() {
  for (int tn = 32; tn <= TOK; tn += 32) {
    const Layout l = layout_of(tn);
    if (l.ns > kMaxStages || l.ns % kGroups || l.ns % kTokProducers || l.nw > kMaxW || l.nw % kGroups || l.acc_col(l.nbuf) > l.w_col(0) ||
        l.alloc() > 232448) return false;
  }
  return true;
}
constexpr int most_shared() {
  int n = 0;
  for (int tn = 32; tn <= TOK; tn += 32) n = layout_of(tn).alloc() > n ? layout_of(tn).alloc() : n;
  return n;
}
static_assert(umma_i8_pair_width(32) && umma_i8_pair_width(TOK), "a tile takes any multiple of 32 tokens up to TOK");
static_assert(WK == 2 * BK && layout_of(kWtDouble).nbuf == 2 && layout_of(kWtDouble + 32).nbuf == 1, "what wt_cut takes for granted");
static_assert(layouts_fit(), "rings and accumulators must fit; a place in a ring must keep its converter groups and its producer");

// 32 tensor-memory lanes x 32 columns in the 16x256b form: v[16 * h + 4 * j + 2 * r + e] is lane 16 h + 8 r + lane / 4,
// column 8 j + 2 (lane % 4) + e.  (Loads and their wait in one statement, see tmem_ld_32x32.)
__device__ __forceinline__ void tmem_ld_frag32(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr), "r"(taddr + (16u << 16))
      : "memory");
}
// Four 8 x 8 matrices of 16-bit values, each stored (loaded) transposed: lane 8 i + q gives the address of row q of matrix i.
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, const uint32_t (&r)[4]) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};"
               ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// The four instructions of a k-block (128 codes: 8 tensor-memory columns and 32 bytes of a row each) over a CTA pair, the
// commit that frees its place, and, in front of them so that its latency is theirs, a look at the two barriers of the next
// k-block: returns whether both are ready.  One thread.
__device__ __forceinline__ uint32_t umma_kblock_pair(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate,
                                                     uint32_t commit_bar, uint16_t mask, uint32_t next_w, uint32_t next_x,
                                                     uint32_t next_parity) {
  uint32_t ready;
  asm volatile(
      "{\n\t.reg .pred p, q, r, t;\n\t.reg .b32 a1, a2, a3;\n\t.reg .b64 b1, b2, b3;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 q, [%8], %10;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 r, [%9], %10;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "setp.eq.b32 t, %5, %5;\n\t"
      "add.u32 a1, %2, 8;\n\tadd.u32 a2, %2, 16;\n\tadd.u32 a3, %2, 24;\n\t"
      "add.u64 b1, %3, 2;\n\tadd.u64 b2, %3, 4;\n\tadd.u64 b3, %3, 6;\n\t"
      "tcgen05.mma.cta_group::2.kind::i8 [%1], [%2], %3, %4, p;\n\t"
      "tcgen05.mma.cta_group::2.kind::i8 [%1], [a1], b1, %4, t;\n\t"
      "tcgen05.mma.cta_group::2.kind::i8 [%1], [a2], b2, %4, t;\n\t"
      "tcgen05.mma.cta_group::2.kind::i8 [%1], [a3], b3, %4, t;\n\t"
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%6], %7;\n\t"
      "and.pred q, q, r;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(ready)
      : "r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(commit_bar), "h"(mask), "r"(next_w), "r"(next_x), "r"(next_parity)
      : "memory");
  return ready;
}
// 2-D tiled TMA load whose completion counts on a barrier of the pair's leader CTA (address from map_to_cta).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const void* tmap, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(tmap), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
// Two barriers at once: the latencies of the two looks overlap (a look that succeeds takes 120 cycles).
__device__ __forceinline__ uint32_t mbar_try_two(uint32_t bar_a, uint32_t par_a, uint32_t bar_b, uint32_t par_b) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 q, [%3], %4;\n\t"
      "and.pred p, p, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(bar_a), "r"(par_a), "r"(bar_b), "r"(par_b)
      : "memory");
  return done;
}
__device__ __forceinline__ void st_shared_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// kFuse: 0 plain scale-factor epilogue; 1 SwiGLU product + quantiser (codes out); 2 SwiGLU product (bf16 out).
// kNat: the activations are 8-bit codes in their natural order (the weights are put into it too); otherwise widened
// 4-bit codes.  kAsym: unsigned codes with a zero point.  kWide: accumulators may leave the range of the exponent trick
// (see `magic_ok`).  kHold: a tile's only accumulator goes to registers as a whole, for the next tile's MMAs to start (more
// than 128 tokens and several tiles a pair); otherwise 32 columns at a time, a quarter of the code, which the last tile of a
// launch enters cold.  (Both in one kernel: 1 to 2 KB of spills.)  kAcc: the accumulators leave too, a debugging aid of
// fpt_w4a8_gemm, in a form of its own: tested for in the plain one it cost every call without it (8-bit codes, us, with the
// test / without: 777x3072x1024 10.3 / 8.9, 2048x8192x1024 32.1 / 25.0, 8192x4096x128 53.0 / 39.2).
template <int kFuse, bool kNat, bool kAsym, bool kWide, bool kHold, bool kAcc = false>
__global__ void __launch_bounds__(kThreads, 1)
gemm_wt_pair_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                    const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmR,
                    const GemmParams P) {
  using L = Layout;
  extern __shared__ uint8_t smem_raw[];
  // (aligned by an offset on the array itself: a round trip through an integer would leave generic pointers)
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + L::kBarOff;
  auto x_full = [&](int s) { return bar0 + 8u * s; };                          // the tokens of a k-block have arrived in both CTAs; used in the leader CTA
  auto op_full = [&](int s) { return bar0 + 8u * (kMaxStages + s); };          // ... and its weights are widened; waited on in the leader CTA
  auto empty = [&](int s) { return bar0 + 8u * (2 * kMaxStages + s); };        // the k-block's MMAs are done
  auto w_full = [&](int w) { return bar0 + 8u * (3 * kMaxStages + w); };       // packed weights of two k-blocks have arrived
  auto w_empty = [&](int w) { return bar0 + 8u * (3 * kMaxStages + kMaxW + w); };
  constexpr int kBar1 = 3 * kMaxStages + 2 * kMaxW;
  auto acc_full = [&](int b) { return bar0 + 8u * (kBar1 + b); };
  auto acc_empty = [&](int b) { return bar0 + 8u * (kBar1 + 2 + b); };        // waited on in the leader CTA
  auto vec_full = [&](int h) { return bar0 + 8u * (kBar1 + 4 + h); };         // per-token factors of a half are in shared memory
  auto stg_full = [&](int h) { return bar0 + 8u * (kBar1 + 6 + h); };         // a half of the tile is staged
  auto stg_empty = [&](int h) { return bar0 + 8u * (kBar1 + 8 + h); };        // ... and has been read
  auto res_full = [&](int h) { return bar0 + 8u * (kBar1 + 10 + h); };        // the residual of a half has arrived in the slabs
  auto prod_full = [&](int h) { return bar0 + 8u * (kBar1 + 12 + h); };       // the products of a half are staged (kFuse 2)
  volatile uint32_t* misc = reinterpret_cast<volatile uint32_t*>(smem + L::kMiscOff);
  volatile uint32_t* abort_flag = misc + 1;

  uint32_t* const status_w = P.status;
  const int ksplit = kHold ? 1 : P.ksplit;                         // 1, or 2: two pairs of a cluster share a tile, half of the k-blocks each
  const int num_tiles = P.num_tiles, tiles_m = P.tiles_m, tn = P.tn;
  const Layout lay = layout_of(tn);
  const int ns = lay.ns, nw = lay.nw, nbuf = kHold ? 1 : lay.nbuf;
  const uint32_t x_smem = sbase + L::kXOff, w_smem = sbase + lay.w_off(), x_stage = lay.x_stage(), slab = lay.slab();
  const int n_cols = P.N, m_rows = P.M;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t crank = cluster_ctarank(), rank = crank & 1u;         // rank 0 = leader of its pair
  const uint32_t leader = crank & ~1u;
  const int part = (int)(crank >> 1);                  // which half of the k-blocks
  const int wb_all = (P.K + WK - 1) / WK, wb_first = part * (wb_all / ksplit);
  const int wblocks = part + 1 == ksplit ? wb_all - wb_first : wb_all / ksplit;        // weight stages of a tile
  const int kblocks = 2 * wblocks;                     // (half a stage at the end of a row reads zeros, as do its tokens)
  const int pair_id = ksplit == 2 ? blockIdx.x >> 2 : blockIdx.x >> 1;
  const int num_pairs = ksplit == 2 ? gridDim.x >> 2 : gridDim.x >> 1;
  // tokens of the tile that starts at token m0, a multiple of 32
  auto tile_tokens = [&](int m0) { const int left = (m_rows - m0 + 31) & ~31; return left < tn ? left : tn; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < ns; ++s) { mbar_init(x_full(s), 1); mbar_init(op_full(s), 8); mbar_init(empty(s), 1); }
    for (int w = 0; w < nw; ++w) { mbar_init(w_full(w), 1); mbar_init(w_empty(w), 8); }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full(b), 1);
      mbar_init(acc_empty(b), 2 * kEpiWarps);
      mbar_init(vec_full(b), 4);
      mbar_init(stg_full(b), 4);
      mbar_init(stg_empty(b), kFuse == 1 ? 4 : 1);
      mbar_init(res_full(b), 1);
      mbar_init(prod_full(b), 4);
    }
    misc[1] = 0;
    fence_mbar_init();
    prefetch_tmap(&tmW);
    prefetch_tmap(&tmX);
    if (kFuse != 1 && P.Y) prefetch_tmap(&tmY);
  }
  if (warp == 1) {
    tmem_alloc_pair(sbase + L::kMiscOff, kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync_all();                                  // barriers of all CTAs exist before any remote arrive
  tc_fence_after();
  const uint32_t tmem_base = misc[0];
  // Everything above touched only the cluster's own shared and tensor memory.  In the composed calls the weights of the
  // first k-blocks are requested too before the wait for the kernel in front, which writes none.
  const int pre = P.early_weights && pair_id < num_tiles ? (wblocks < nw ? wblocks : nw) : 0;
  if (warp == 0 && elect_one()) {
    const int n0 = (pair_id / tiles_m) * RT + (int)rank * HR;
    for (int w = 0; w < pre; ++w) {
      mbar_arrive_expect_tx(w_full(w), L::kWStage);
      tma_load_2d(w_smem + w * L::kWStage, &tmW, w_full(w), (wb_first + w) * W_ROW, n0);
    }
  }
  pdl_wait();
  pdl_launch_dependents();

  if (warp < kConvWarp0) {
    reg_dec<kRegsCtl>();
    if (warp == 0) {
      // ---------------------------------------------------------------- TMA producer: weights
      if (elect_one()) {
        int asked = pre;                                 // stages that are on their way already
        int s = 0; uint32_t ph = 0;
        uint32_t armed = 0, armed_par = 0;
        bool ok = true;
        for (int tile = pair_id; ok && tile < num_tiles; tile += num_pairs) {
          const int n0 = (tile / tiles_m) * RT + (int)rank * HR;
          for (int wb = 0; wb < wblocks; ++wb) {
            if (asked > 0) {
              --asked;
            } else {
              if (!mbar_wait(w_empty(s), ph ^ 1u, abort_flag, status_w, 1)) { ok = false; break; }
              mbar_arrive_expect_tx(w_full(s), L::kWStage);
              tma_load_2d(w_smem + s * L::kWStage, &tmW, w_full(s), (wb_first + wb) * W_ROW, n0);
            }
            armed |= 1u << s;
            armed_par = (armed_par & ~(1u << s)) | (ph << s);
            if (++s == nw) { s = 0; ph ^= 1u; }
          }
        }
        if (!ok) {
          // bounded wait for the copies still in flight before this CTA's shared memory goes away
          const uint64_t t0 = globaltimer_ns();
          for (int q = 0; q < nw; ++q)
            if (armed & (1u << q))
              while (!mbar_try_wait(w_full(q), (armed_par >> q) & 1u) && globaltimer_ns() - t0 < 2000000ull) {}
        }
      }
    } else if (warp != 1) {
      // ---------------------------------------------------------------- TMA producers: tokens, every second k-block each
      if (elect_one()) {
        const uint32_t x_full_leader = map_to_cta(x_full(0), leader);
        const int first = warp - 2;
        int s = first; uint32_t ph = 0;
        bool ok = true;
        for (int tile = pair_id; ok && tile < num_tiles; tile += num_pairs) {
          const int m0 = (tile % tiles_m) * tn;
          const int y = m0 + (int)rank * (tile_tokens(m0) >> 1);
          for (int kb = first; kb < kblocks; kb += kTokProducers) {
            if (!mbar_wait(empty(s), ph ^ 1u, abort_flag, status_w, 1)) { ok = false; break; }
            if (rank == 0) mbar_arrive_expect_tx(x_full(s), 2 * x_stage);
            tma_load_2d_pair(x_smem + s * x_stage, &tmX, x_full_leader + 8u * s, (2 * wb_first + kb) * BK, y);
            s += kTokProducers;
            if (s >= ns) { s -= ns; ph ^= 1u; }
          }
        }
        if (!ok) {
          // Copies may still be in flight, and the barriers that count them are the leader's: time for them to land
          // before this CTA's shared memory goes away.
          const uint64_t t0 = globaltimer_ns();
          while (globaltimer_ns() - t0 < 2000000ull) {}
        }
      }
    } else if (warp == 1) {
      // ---------------------------------------------------------------- MMA issuer (leader CTA only, one elected thread)
      if (rank == 0 && elect_one()) {
        const uint16_t pair_mask = (uint16_t)(3u << leader);
        const uint64_t bdesc0 = umma_desc_kmajor_sw128(x_smem);
        const uint32_t a_tmem0 = tmem_base + lay.w_col(0);
        int s = 0; uint32_t ph = 0; int it = 0;
        uint32_t ready = 0;                              // the k-block is known to be ready
        for (int tile = pair_id; tile < num_tiles; tile += num_pairs, ++it) {
          const uint32_t idesc = umma_idesc_i8(RT, tile_tokens((tile % tiles_m) * tn), true, !kAsym);
          const int b = nbuf == 2 ? it & 1 : 0; const uint32_t bph = (nbuf == 2 ? it >> 1 : it) & 1;
          if (!mbar_wait_cluster(acc_empty(b), bph ^ 1u, abort_flag, status_w, 2)) break;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + lay.acc_col(b);
          bool ok = true;
          for (int kb = 0; kb < kblocks; ++kb) {
            if (!ready && (!mbar_wait_cluster(op_full(s), ph, abort_flag, status_w, 3) ||
                           !mbar_wait_cluster(x_full(s), ph, abort_flag, status_w, 2))) { ok = false; break; }
            tc_fence_after();
            const int s0 = s;
            if (++s == ns) { s = 0; ph ^= 1u; }
            ready = umma_kblock_pair(d_tmem, a_tmem0 + s0 * kWStageCols, bdesc0 + (uint32_t)(s0 * x_stage >> 4), idesc, kb != 0,
                                     empty(s0), pair_mask, op_full(s), x_full(s), ph);
          }
          if (!ok) break;
          umma_commit_pair(acc_full(b), pair_mask);
        }
      }
    }
    if (ksplit == 2) { __syncwarp(); cluster_sync_all(); }               // (the exchange of the epilogue warps)
  } else if (warp < kEpiWarp0) {
    // ------------------------------------------------------------------ weight converters
    // A group takes every third k-block: the CTA's 128 weight rows, one per thread (warp % 4 selects the tensor-memory
    // lanes the warp may touch).
    reg_dec<kRegsConv>();
    const int grp = (warp - kConvWarp0) >> 2;
    const int quad = warp & 3;
    const int r = quad * 32 + lane;
    const uint32_t swz = (uint32_t)(r & 7);              // SWIZZLE_128B: 16-byte chunk index ^= row % 8
    const uint32_t op_full_leader = map_to_cta(op_full(0), leader);
    const int my_tiles = pair_id < num_tiles ? (num_tiles - 1 - pair_id) / num_pairs + 1 : 0;
    const long long total = (long long)my_tiles * kblocks;               // k-blocks of this pair
    int s = grp, wk = grp; uint32_t ph = 0, wph = 0;     // place in the ring of k-blocks; k-block in the ring of weights
    for (long long kc = grp; kc < total; kc += kGroups) {
      const int w = wk >> 1;
      if (!__all_sync(0xffffffffu, mbar_try_two(empty(s), ph ^ 1u, w_full(w), wph))) {
        if (!mbar_wait_warp(empty(s), ph ^ 1u, abort_flag, status_w, 5)) break;
        if (!mbar_wait_warp(w_full(w), wph, abort_flag, status_w, 6)) break;
      }
      tc_fence_after();
      const uint8_t* src = smem + lay.w_off() + w * L::kWStage + r * W_ROW;
      const uint32_t half = (uint32_t)(wk & 1) * 4u;
      const uint32_t a_tmem = tmem_base + ((uint32_t)(quad * 32) << 16) + lay.w_col(s);
      // the row's 128 codes: all loads first, then two halves of 64 (16 tensor-memory columns each)
      uint4 c[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) c[j] = *reinterpret_cast<const uint4*>(src + (((half + (uint32_t)j) ^ swz) << 4));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint4 &c0 = c[2 * h], &c1 = c[2 * h + 1];
        const uint32_t p[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
        uint32_t v[16];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint2 w = widen_word(p[j]);
          v[2 * j] = kNat ? __byte_perm(w.x, w.y, 0x5140) : w.x;
          v[2 * j + 1] = kNat ? __byte_perm(w.x, w.y, 0x7362) : w.y;
        }
        tmem_st_32x16(a_tmem + 16 * h, v);
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      // (the packed rows have been read: what went to tensor memory depends on them)
      if (lane == 0) { mbar_arrive_cluster(op_full_leader + 8u * s); mbar_arrive(w_empty(w)); }
      s += kGroups;
      if (s >= ns) { s -= ns; ph ^= 1u; }
      wk += kGroups;
      if (wk >= 2 * nw) { wk -= 2 * nw; wph ^= 1u; }
    }
    if (ksplit == 2) { __syncwarp(); cluster_sync_all(); }
  } else {
    // ------------------------------------------------------------------ epilogue
    reg_inc<kRegsEpi>();
    const int quad = warp & 3;                           // TMEM lane quadrant this warp may read
    const int half = (warp - kEpiWarp0) >> 2;            // tokens [half * tn / 2, (half + 1) * tn / 2) of the tile
    const int htok = tn >> 1;
    const int t_own = quad * 32 + lane;                  // the token of the half whose factors this thread fetches
    const uint32_t acc_empty_leader = map_to_cta(acc_empty(0), leader);
    float* const vec = reinterpret_cast<float*>(smem + L::kVecOff);
    constexpr int kShift = kNat ? 4 : 8;                 // the weights carry a factor 16, widened 4-bit activations too
    // |acc| < 2^22: int -> float by the exponent trick.  With symmetric 4-bit activation codes that holds for every
    // K the entry points accept (64 * 65408 < 2^22); on an asymmetric grid |code - z| reaches 15 and 120 K passes 2^22
    // from K = 34953 on, where the host launches the kWide form.
    const bool magic_ok = kNat ? P.K < 4096 : !kWide;
    const bool issuer = quad == 0 && lane == 0;          // issues the TMA stores (and residual loads) of its half
    const bool finish = ksplit == 1 || half == part;     // two pairs: each finishes one half of the tokens
    bool met = ksplit == 1;                              // the pairs' exchange is over
    const bool use_res = kFuse == 0 && P.residual != nullptr && P.Y != nullptr;
    const bool use_y = kFuse != 0 || P.Y != nullptr;
    const bool has_vec = kFuse == 0 && (P.post != nullptr || P.res_scale != nullptr);
    int it = 0;
    int res_armed = 0, res_seen = 0;                     // residual loads issued / seen to arrive
    for (int tile = pair_id; tile < num_tiles; tile += num_pairs, ++it) {
      const int m0 = (tile % tiles_m) * tn;
      const int n0 = (tile / tiles_m) * RT + (int)rank * HR;             // first weight row (feature) of this CTA
      const int left = tile_tokens(m0) - half * htok;
      const int cols = left < 0 ? 0 : left < htok ? left : htok;         // accumulator columns of this half: a multiple of 16
      const int mh = m0 + half * htok;                                   // first token of the half
      const int b = nbuf == 2 ? it & 1 : 0; const uint32_t bph = (nbuf == 2 ? it >> 1 : it) & 1;
      // this thread's four features (fragment rows) and their constants
      const int nf = n0 + quad * 32 + (lane >> 2);
      float sw[4]; int zw[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int n = nf + 8 * i;
        sw[i] = n < n_cols ? load_scale(P.sw, P.scale_dtype, n) : 0.0f;
        zw[i] = (kAsym && n < n_cols) ? P.zero_point * __ldg(P.wsum + n) : 0;
      }
      float* const c_s = vec + (it & 1) * 2 * TOK + half * (TOK / 2);
      float* const rs_s = c_s + TOK;
      const int tok = mh + t_own;
      const bool tok_ok = t_own < cols && tok < m_rows;
      if (has_vec) {
        c_s[t_own] = (tok_ok && P.post) ? __fmul_rn(P.act_scale, __ldg(P.post + tok)) : P.act_scale;
        rs_s[t_own] = (tok_ok && P.res_scale) ? __ldg(P.res_scale + tok) : 1.0f;
        __syncwarp();
        if (lane == 0) mbar_arrive(vec_full(half));
        if (!mbar_wait_warp(vec_full(half), it & 1, abort_flag, status_w, 9)) break;
      }
      // the slabs' half must have been read by whatever took the previous tile from it
      if (use_y && !mbar_wait_warp(stg_empty(half), (it & 1) ^ 1u, abort_flag, status_w, 10)) break;
      const uint32_t stg = sbase + lay.stg_off() + (uint32_t)(half * htok) * 128u;       // in slab 0; slab 1 follows it
      if constexpr (kFuse == 0) {
        if (use_res && issuer && finish && cols > 0) {   // travels while the matmul of the tile still runs
          mbar_arrive_expect_tx(res_full(half), 2u * (uint32_t)htok * 128u);
          tma_load_2d(stg, &tmR, res_full(half), n0, mh);
          tma_load_2d(stg + slab, &tmR, res_full(half), n0 + 64, mh);
          ++res_armed;
        }
      }
      if (!mbar_wait_warp(acc_full(b), bph, abort_flag, status_w, 4)) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + lay.acc_col(b) + half * htok;
      if (ksplit == 2) {
        // The half that the other pair finishes goes to this CTA's own rings, which are free (all k-blocks have been
        // used, and there is no second tile), and the cluster meets.
        const uint32_t mine = x_smem + (uint32_t)(quad * TOK / 2 * 32 + lane) * 4u;
        if (!finish) {
#pragma unroll 1
          for (int c0 = 0; c0 < cols; c0 += 32) {
            uint32_t v[32];
            tmem_ld_frag32(taddr + c0, v);
#pragma unroll
            for (int e = 0; e < 32; ++e) st_shared_u32(mine + (uint32_t)(c0 + e) * 128u, v[e]);
          }
        }
        __syncwarp();
        cluster_sync_all();
        met = true;
        if (!finish) break;
      }
      if (use_res && cols > 0) {
        if (!mbar_wait_warp(res_full(half), res_seen & 1, abort_flag, status_w, 12)) break;
        ++res_seen;
      }
      // where lane 8 i + q stores (and finds the residual of) row q of fragment column i: token 8 j + q, features 8 i ..
      const uint32_t frag0 = stg + (uint32_t)(quad >> 1) * slab + (uint32_t)(lane & 7) * 128u +
                             ((uint32_t)(((quad & 1) * 4 + (lane >> 3)) ^ (lane & 7)) << 4);
      // 32 columns (tokens) of the accumulator
      auto finish_32 = [&](const uint32_t* v, int c0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int col = c0 + j * 8;
          if (col < cols) {
            const int t2 = col + 2 * (lane & 3);         // this thread's two tokens
            float2 c = make_float2(P.act_scale, P.act_scale), rs = make_float2(1.0f, 1.0f);
            if (has_vec) {
              c = *reinterpret_cast<const float2*>(c_s + t2);
              if (use_res) rs = *reinterpret_cast<const float2*>(rs_s + t2);
            }
            uint32_t rw[4];
            if (use_res) ldmatrix_x4_trans(frag0 + (uint32_t)col * 128u, rw);
            uint32_t o[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int a0 = (((int)v[16 * (i >> 1) + 4 * j + 2 * (i & 1)]) >> kShift) - zw[i];
              const int a1 = (((int)v[16 * (i >> 1) + 4 * j + 2 * (i & 1) + 1]) >> kShift) - zw[i];
              if constexpr (kAcc) {
                if (nf + 8 * i < n_cols) {
                  int32_t* const out = P.acc_out + (size_t)(mh + t2) * n_cols + nf + 8 * i;
                  if (mh + t2 < m_rows) out[0] = a0;
                  if (mh + t2 + 1 < m_rows) out[n_cols] = a1;
                }
              }
              // exact int -> float: 1.5 * 2^23 + a has a in its low mantissa bits
              const float f0 = magic_ok ? __fsub_rn(__int_as_float(0x4B400000 + a0), 12582912.0f) : (float)a0;
              const float f1 = magic_ok ? __fsub_rn(__int_as_float(0x4B400000 + a1), 12582912.0f) : (float)a1;
              float y0 = __fmul_rn(__fmul_rn(f0, sw[i]), c.x), y1 = __fmul_rn(__fmul_rn(f1, sw[i]), c.y);
              if (use_res) {                             // rows and columns outside the matrix arrive as zeros
                y0 = __fadd_rn(y0, __fmul_rn(bf16lo_to_f32(rw[i]), rs.x));
                y1 = __fadd_rn(y1, __fmul_rn(bf16hi_to_f32(rw[i]), rs.y));
              }
              o[i] = f32x2_to_bf16x2_bits(y0, y1);
            }
            if (use_y) stmatrix_x4_trans(frag0 + (uint32_t)col * 128u, o);
          }
        }
      };
      if constexpr (kHold) {
        uint32_t v[4][32];
#pragma unroll
        for (int ch = 0; ch < 4; ++ch)
          if (ch * 32 < cols) tmem_ld_frag32(taddr + 32 * ch, v[ch]);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acc_empty_leader + 8u * b);
#pragma unroll
        for (int ch = 0; ch < 4; ++ch)
          if (ch * 32 < cols) finish_32(v[ch], 32 * ch);
      } else {
        const uint32_t other = map_to_cta(x_smem + (uint32_t)(quad * TOK / 2 * 32 + lane) * 4u, crank ^ (ksplit == 2 ? 2u : 0u));
#pragma unroll 1
        for (int c0 = 0; c0 < cols; c0 += 32) {
          uint32_t v[32];
          tmem_ld_frag32(taddr + c0, v);
          if (ksplit == 2) {
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] += ld_shared_cluster_u32(other + (uint32_t)(c0 + e) * 128u);
          }
          finish_32(v, c0);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acc_empty_leader + 8u * b);
      }
      if (use_y) {
        if (kFuse == 0) fence_proxy_async_smem();        // staged tile -> visible to the TMA engine
        __syncwarp();
        if (lane == 0) mbar_arrive(stg_full(half));
        bool staged = true;
        if constexpr (kFuse != 0) {
          // 64 gate values of a token in slab 0, the matching 64 up values in slab 1: a thread takes eight of a token at
          // a time (a token each left most threads idle in narrow tiles: 17 tokens x 4096x14336 59 us, now 33.5).
          if (!mbar_wait_warp(stg_full(half), it & 1, abort_flag, status_w, 14)) break;
          const int f0 = n0 >> 1;                        // first of the 64 features
#pragma unroll 1
          for (int i = t_own; i < cols * 8; i += 128) {
            const int t = i >> 3, q = i & 7, tok = mh + t;
            uint4* const gp = reinterpret_cast<uint4*>(smem + lay.stg_off() + (half * htok + t) * 128 + ((q ^ (t & 7)) << 4));
            const uint4 g = *gp, u = *reinterpret_cast<const uint4*>(reinterpret_cast<const uint8_t*>(gp) + slab);
            const uint4 m = make_uint4(silu_mul_pair(g.x, u.x), silu_mul_pair(g.y, u.y), silu_mul_pair(g.z, u.z),
                                       silu_mul_pair(g.w, u.w));
            if constexpr (kFuse == 2) {
              *gp = m;
            } else if (tok < m_rows && n0 < n_cols) {
              const QuantConsts qc = quant_consts(__ldg(P.mid_scale + tok), P.mid_inv_delta, P.mid_qmax_minus_z, P.mid_flip);
              const uint32_t w = quant_word(m, qc);
              if (P.mq_wide) *reinterpret_cast<uint2*>(P.Mq + (size_t)tok * (size_t)(n_cols >> 1) + f0 + 8 * q) = widen_word(w);
              else *reinterpret_cast<uint32_t*>(P.Mq + (size_t)tok * (size_t)(n_cols >> 2) + (f0 >> 1) + 4 * q) = w;
            }
          }
          if constexpr (kFuse == 1) {
            __syncwarp();
            if (lane == 0) mbar_arrive(stg_empty(half));
          } else {
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(prod_full(half));
            if (issuer) staged = mbar_wait(prod_full(half), it & 1, abort_flag, status_w, 11);
          }
        } else {
          if (issuer) staged = mbar_wait(stg_full(half), it & 1, abort_flag, status_w, 11);
        }
        if constexpr (kFuse != 1) {
          if (issuer && staged) {
            const int x0 = kFuse == 2 ? n0 >> 1 : n0;    // first output column; a store starts inside the matrix only
            const int x_end = kFuse == 2 ? n_cols >> 1 : n_cols;
            if (mh < m_rows && cols > 0) {
              if (x0 < x_end) tma_store_2d(&tmY, stg, x0, mh);
              if (kFuse == 0 && x0 + 64 < x_end) tma_store_2d(&tmY, stg + slab, x0 + 64, mh);
            }
            tma_store_commit();
            tma_store_wait_read();
            mbar_arrive(stg_empty(half));
          }
        }
        if (!__all_sync(0xffffffffu, staged)) break;     // the warp leaves as one
      }
    }
    if (!met) { __syncwarp(); cluster_sync_all(); }
    if (issuer) tma_store_wait_read();
    if (issuer && res_armed > res_seen) {
      // left the loop on a timeout with a residual load still in flight: bounded wait before the shared memory it
      // writes to goes away
      const uint64_t t0 = globaltimer_ns();
      while (!mbar_try_wait(res_full(half), (uint32_t)(res_armed - 1) & 1u) && globaltimer_ns() - t0 < 2000000ull) {}
    }
  }

  // ------------------------------------------------------------------ teardown
  // No CTA may leave (or free tensor memory) while a peer can still arrive on its barriers or read its shared
  // memory, or the pair's MMAs can still read its shared / tensor memory.
  __syncwarp();
  tc_fence_before();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

// ------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------
static bool make_map(CUtensorMap* m, CUtensorMapDataType type, const void* base, size_t cols, size_t rows, size_t pitch, int box_cols,
                     int box_rows, CUtensorMapSwizzle swz, CUtensorMapL2promotion promo) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch};
  const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, type, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz, promo,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int kFuse, bool kNat, bool kAsym, bool kWide, bool kHold, bool kAcc = false>
static int launch_cut(cudaStream_t st, const int8_t* X8, const uint8_t* Wq, GemmParams P, int max_pairs) {
  auto kern = gemm_wt_pair_kernel<kFuse, kNat, kAsym, kWide, kHold, kAcc>;
  const size_t k = (size_t)P.K, out_cols = (size_t)(kFuse == 2 ? P.N / 2 : P.N);
  CUtensorMap tmW, tmX, tmY, tmR;
  if (!make_map(&tmW, CU_TENSOR_MAP_DATA_TYPE_UINT8, Wq, k / 2, P.N, k / 2, W_ROW, HR, CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B) ||
      !make_map(&tmX, CU_TENSOR_MAP_DATA_TYPE_UINT8, X8, k, P.M, k, BK, P.tn / 2, CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B))
    return FPT_ERR_CUDA;
  tmY = tmX;
  if (kFuse != 1 && P.Y && !make_map(&tmY, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, P.Y, out_cols, P.M, out_cols * 2, 64, P.tn / 2,
                                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE))
    return FPT_ERR_CUDA;
  tmR = tmY;
  if (kFuse == 0 && P.Y && P.residual &&
      !make_map(&tmR, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, P.residual, out_cols, P.M, out_cols * 2, 64, P.tn / 2,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE))
    return FPT_ERR_CUDA;
  const int grid = P.ksplit == 2 ? 4 * P.num_tiles : 2 * (P.num_tiles < max_pairs ? P.num_tiles : max_pairs);
  return launch_kernel_cluster(kern, dim3(grid), dim3(kThreads), layout_of(P.tn).alloc(), st, true, 2 * P.ksplit, tmW, tmX, tmY, tmR,
                               P) == cudaSuccess
             ? FPT_OK
             : FPT_ERR_CUDA;
}

template <int kFuse, bool kNat = false, bool kAsym = false, bool kWide = false>
static int launch(cudaStream_t st, const int8_t* X8, const uint8_t* Wq, GemmParams P) {
  // Once a device: the kernels' attribute, and the clusters of 2 and of 4 CTAs that are resident at once (one look-up a
  // call: each costs 0.1 us, which a small eager call notices).
  static PerDeviceInt prepared;
  const int found = prepared.get([] {
    auto kern = gemm_wt_pair_kernel<kFuse, kNat, kAsym, kWide, false>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most_shared()) != cudaSuccess ||
        cudaFuncSetAttribute(gemm_wt_pair_kernel<kFuse, kNat, kAsym, kWide, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             most_shared()) != cudaSuccess)
      return 0;
    int clusters[2];
    for (int i = 0; i < 2; ++i) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(2 << i, 1, 1);
      cfg.blockDim = dim3(kThreads, 1, 1);
      cfg.dynamicSmemBytes = most_shared();
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 2 << i; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr; cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&clusters[i], kern, &cfg) != cudaSuccess) { cudaGetLastError(); clusters[i] = 0; }
    }
    if (clusters[0] <= 0) clusters[0] = device_pairs();      // (not known)
    return (clusters[0] & 0x7FFF) | (clusters[1] > 0 ? clusters[1] & 0x7FFF : 0) << 15;
  });
  if (found <= 0) return FPT_ERR_CUDA;
  if constexpr (kNat) {
    static PerDeviceInt acc_attr;
    if (P.acc_out && !ensure_smem_attr(acc_attr, gemm_wt_pair_kernel<kFuse, kNat, kAsym, kWide, false, true>, most_shared()))
      return FPT_ERR_CUDA;
  }
  const int max_pairs = found & 0x7FFF;
  const WtCut cut = wt_cut(P.M, P.N, P.K, max_pairs, found >> 15, kFuse == 0);
  P.tn = cut.tn; P.ksplit = cut.ksplit;
  P.tiles_m = (P.M + P.tn - 1) / P.tn;
  P.num_tiles = P.tiles_m * ((P.N + RT - 1) / RT);
  if constexpr (kNat)
    if (P.acc_out) return launch_cut<kFuse, kNat, kAsym, kWide, false, true>(st, X8, Wq, P, max_pairs);
  if (layout_of(P.tn).nbuf == 1 && P.ksplit == 1 && P.num_tiles > max_pairs)
    return launch_cut<kFuse, kNat, kAsym, kWide, true>(st, X8, Wq, P, max_pairs);
  return launch_cut<kFuse, kNat, kAsym, kWide, false>(st, X8, Wq, P, max_pairs);
}

}  // namespace wt

bool gemm_wt_serves(int M, int N, int K, int extras) { return wt_ahead(M, N, K, device_pairs(), extras); }
bool gemm_wt_serves_swiglu(int M, int N, int K) { return wt_ahead_swiglu(M, N, K, device_pairs()); }

int gemm_wt_launch(cudaStream_t st, const int8_t* X8, const uint8_t* Wq, const GemmParams& P) {
  if (P.Mq) return wt::launch<1>(st, X8, Wq, P);
  if (P.swiglu_bf16) return wt::launch<2>(st, X8, Wq, P);
  if (P.a_bits == 8) return wt::launch<0, true>(st, X8, Wq, P);
  if (P.a_unsigned && 15ll * 8 * P.K >= (1 << 22)) return wt::launch<0, false, true, true>(st, X8, Wq, P);
  if (P.a_unsigned) return wt::launch<0, false, true>(st, X8, Wq, P);
  return wt::launch<0>(st, X8, Wq, P);
}

}  // namespace fpt
