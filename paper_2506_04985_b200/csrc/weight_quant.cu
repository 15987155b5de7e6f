// Offline weight quantiser: per-output-channel symmetric INT4 grid, round-to-nearest,
// min-max or L_p range setting (Sec. 4 "Quantization Setup"; App. D "Quantizer range
// setting"), packed two codes per byte (App. J).  One CTA per row.
//
// The L_p search is bound by arithmetic: 81 candidate scales x K values, each a division, a rounding and a
// float64 power.  A thread keeps sixteen values in registers (float32 and float64) and walks over the candidates,
// so that sixteen independent chains hide the float64 latency (nine candidates per value instead: 7.0 ms on the
// shape below, with half the warps); the division is a multiply that is redone as a division only where the
// quotient lies so close to a tie that the two could round differently, one branch for the sixteen values; |e|^3
// (the method's p) is two float64 multiplies; sums meet once per warp and candidate.
// 14336 x 4096, p = 3, f16 scales: 38.6 -> 2.63 ms; min-max 72 -> 53 us (the row is read once, 16 bytes a load).
// With the candidates screened in float32 first (below; the method's p only): bf16 488 us, f32 1.20 ms (2.48 without);
// 4096 x 14336 bf16 3.29 ms -> 257 us, 4096 x 2048 f32 368 -> 183 us.  What it takes now is instruction issue: 1216 x 81
// terms of five instructions a row, about 0.25 ms, then the float64 sums of what is left and the histogram.
#include <type_traits>

#include "fpt_common.cuh"
#include "fpt_host.cuh"
#include "quant_math.cuh"

namespace fpt {

constexpr int kWqThreads = 256;
constexpr int kLpFirst = 20, kLpCount = 81;                        // candidate scales a * i / 100, i = 20 .. 100
constexpr int kLpHold = 16;                                        // values a thread holds during the search

// eight consecutive weights as float
__device__ __forceinline__ void wload8(const __nv_bfloat16* p, float* w) {
  const uint4 v = *reinterpret_cast<const uint4*>(p);
  w[0] = bf16lo_to_f32(v.x); w[1] = bf16hi_to_f32(v.x); w[2] = bf16lo_to_f32(v.y); w[3] = bf16hi_to_f32(v.y);
  w[4] = bf16lo_to_f32(v.z); w[5] = bf16hi_to_f32(v.z); w[6] = bf16lo_to_f32(v.w); w[7] = bf16hi_to_f32(v.w);
}
__device__ __forceinline__ void wload8(const float* p, float* w) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
}

__device__ __forceinline__ float store_round(float d, int scale_dtype) {
  return scale_dtype == FPT_DTYPE_F16 ? __half2float(__float2half_rn(d)) : d;
}

// A grid step with what the multiply-instead-of-divide form needs.  `inv` is 0 where that form is not used: a
// step whose reciprocal is not an ordinary number.
struct Step {
  float d, inv;
};
__device__ __forceinline__ Step make_step(float d) {
  Step s;
  s.d = d;
  s.inv = (d > 0x1p-100f && d < 0x1p100f) ? __fdiv_rn(1.0f, d) : 0.0f;
  return s;
}

// clamp(rne(w / d), -8, 7) + 8, w / d rounded to float32 (IEEE division); a NaN gives 0.
__device__ __forceinline__ int biased_div(float w, float d) {
  return (int)fminf(fmaxf(rintf(__fdiv_rn(w, d)), -8.0f), 7.0f) + 8;
}
// The same through w * (1/d), for quotients below 2^22.  `far` returns how far the product is from its rounded
// value: the product is within 2^-23 of the quotient, relatively, and the float32 quotient within 2^-24, so for
// |quotient| < 9 the two are closer than 2e-6 and round alike unless they lie that close to k + 1/2, i.e. unless
// `far` is above kTieClose (beyond 9 both clamp alike).  A NaN must not come here.
constexpr float kTieClose = 0.5f - 4e-6f;
__device__ __forceinline__ int biased_mul(float w, float inv, float& far) {
  const float t = __fmul_rn(w, inv);
  const float r = __fadd_rn(t, 12582912.0f);                       // 1.5 * 2^23 + rne(t)
  far = fabsf(__fsub_rn(t, __fsub_rn(r, 12582912.0f)));
  return __viaddmin_s32_relu(__float_as_int(r), -0x4B400000 + 8, 15);
}
__device__ __forceinline__ int quant_code(float w, const Step& s, bool fast) {
  float far = 0.0f;
  int u = fast ? biased_mul(w, s.inv, far) : 0;
  if (!fast || far > kTieClose) u = biased_div(w, s.d);
  return u - 8;
}

// Sum (or maximum) over the CTA, the same in every thread.
template <int NT, typename V>
__device__ __forceinline__ V block_reduce(V v, V* scratch, bool is_max) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const V other = __shfl_xor_sync(0xffffffffu, v, o);
    v = is_max ? (other > v ? other : v) : v + other;
  }
  __syncthreads();                                // scratch may still be read from the last call
  if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
  __syncthreads();
  V r = scratch[0];
  for (int w = 1; w < NT / 32; ++w) r = is_max ? (scratch[w] > r ? scratch[w] : r) : r + scratch[w];
  return r;
}

// Sums of |w - D q|^p per candidate and warp over the values `from` .. `n` of a row, for a p that is not 3.  A power costs
// hundreds of instructions, so no thread takes one for a value that is not there: the values (in L1) are dealt out one by
// one, four at a time where a thread has that many.  p = 2, sixteen values held by each thread as below instead: 14336 x 96
// 10.4 ms, now 1.14; 64 x 256 560 us, now 62; 4096 x 1056 5.9 ms, now 2.9.
__device__ __forceinline__ float wload(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ float wload(const float* p) { return *p; }
template <typename T, int NT>
__device__ __forceinline__ void power_sums(const T* row, int from, int n, const Step* step, double (*part)[NT / 32], bool no_nan, double p) {
  const int tid = threadIdx.x;
  for (int i = 0; i < kLpCount; ++i) {
    const Step s = step[i];
    const bool fast = no_nan && s.inv != 0.0f;
    auto error = [&](int k) {
      const float w = wload(row + k);
      return pow(fabs((double)w - (double)s.d * (double)quant_code(w, s, fast)), p);
    };
    double sum = 0.0;
    int k = from + tid;
    for (; k + 3 * NT < n; k += 4 * NT) sum += (error(k) + error(k + NT)) + (error(k + 2 * NT) + error(k + 3 * NT));
    for (; k < n; k += NT) sum += error(k);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((tid & 31) == 0) part[i][tid >> 5] += sum;
  }
}

// Screening of the candidates of an L_3 search in float32.  A candidate's sum there is within `kScreenEps` of the exact
// one, relatively: a code can differ only where the quotient lies within 1e-6 of a tie, where both neighbours leave the
// same |e| to 4e-6, so a term |e|^3 is right to 2e-5, and the additions (a chain of at most 203 terms; from chunk to chunk in
// float64, a row has no end: in float32 33 million values lost 5e-4, and the answer with them) add less than 3e-5.  So a candidate beyond (1 + 4 kScreenEps) times the least sum cannot be the answer; the ones that
// are left (one to three of 81, as a rule) go through the float64 sums below, which decide as they always did.
// The row is scaled by a power of two so that its largest magnitude lies in [1, 2): |e|^3 then underflows only below
// 2^-42, which the absolute slack covers.
//   * bf16 rows longer than kBins: what counts is how often a magnitude occurs.  Bins by bit pattern below the row's
//     largest, 128 an octave: kTop for each sign (the grid's ends differ, -8 and 7), kBoth for the two together (no
//     candidate clamps there, 0.19 a < 7.4 D), and from seven octaves down every candidate has the code 0 (a / 128 <
//     0.49 D), the same error for all.  1216 magnitudes with a count each in place of K values.
//   * otherwise the values themselves, kChunk at a time.
// A thread takes a candidate and a third of the entries, which a warp then reads as broadcasts: nothing is reduced per
// candidate but three numbers.  Two entries an instruction where the packed forms allow.
constexpr float kScreenEps = 1e-4f;
constexpr int kTop = 320, kBoth = 576, kBins = 2 * kTop + kBoth, kChunk = 1024, kThirds = 3;
static_assert(kTop % 4 == 0 && kBoth % 4 == 0 && kChunk <= kBins, "four entries a load");

__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// Two entries: adds count * |D q - v|^3.  kClamp: 0 no code is clamped, 1 magnitudes, codes up to `hi`, 2 signed values.
template <int kClamp>
__device__ __forceinline__ uint64_t screen2(float v0, float v1, uint64_t count, uint64_t inv2, uint64_t neg_d2, float hi, uint64_t acc) {
  constexpr float kMagic = 12582912.0f;                            // 1.5 * 2^23
  const uint64_t v = pack_f32x2(v0, v1);
  uint64_t q = fma_f32x2(v, inv2, pack_f32x2(kMagic, kMagic));
  if constexpr (kClamp != 0) {
    float r0, r1;
    unpack_f32x2(q, r0, r1);
    if constexpr (kClamp == 2) { r0 = fmaxf(r0, kMagic - 8.0f); r1 = fmaxf(r1, kMagic - 8.0f); }
    q = pack_f32x2(fminf(r0, kMagic + hi), fminf(r1, kMagic + hi));
  }
  const uint64_t e = fma_f32x2(neg_d2, add_f32x2(q, pack_f32x2(-kMagic, -kMagic)), v);
  float e0, e1, s0, s1;
  unpack_f32x2(e, e0, e1);
  unpack_f32x2(mul_f32x2(e, e), s0, s1);
  return fma_f32x2(pack_f32x2(s0 * fabsf(e0), s1 * fabsf(e1)), count, acc);
}

// Finds the candidates that can be the answer: list[0 .. count), in ascending order.  False: not applicable, all can.
template <typename T, int NT>
__device__ bool lp_screen(const T* row, int chunks, float a, bool no_nan, const Step* step, unsigned char* list, int* count) {
  __shared__ __align__(16) float val[kBins];
  __shared__ __align__(16) union { unsigned n[kBins]; float f[kBins]; } cnt;   // (both read four at a time)
  __shared__ float part[kThirds][kLpCount];
  constexpr bool kBf16 = sizeof(T) == 2;
  constexpr int kTasks = kThirds * kLpCount, kPer = (kTasks + NT - 1) / NT;
  const int tid = threadIdx.x, lane = tid & 31;
  const float d_min = step[0].d;
  // (steps grow with the candidate; a step of 0 has been replaced by 1, one beyond float16 has no reciprocal)
  if (!no_nan || !(a > 0x1p-90f && a < 0x1p90f) || !(d_min < a * 0.03f) || step[0].inv == 0.0f || step[kLpCount - 1].inv == 0.0f) return false;
  const int exponent = (int)(__float_as_uint(a) >> 23);
  const float unit = __uint_as_float((uint32_t)(254 - exponent) << 23);       // a * unit in [1, 2)
  const bool bins = kBf16 && 8 * chunks > kBins && 0.19f * a < 7.4f * d_min && a * (1.0f / 128) < 0.49f * d_min;
  double acc[kPer];
#pragma unroll
  for (double& v : acc) v = 0.0;
  auto both = [](uint64_t v) {
    float lo, hi;
    unpack_f32x2(v, lo, hi);
    return (double)lo + (double)hi;
  };
  if (bins) {
    const int top = (int)(__float_as_uint(a) >> 16);               // pattern of the largest magnitude
    for (int i = tid; i < kBins; i += NT) cnt.n[i] = 0;
    __syncthreads();
    for (int c = tid; c < chunks; c += NT) {
      const uint4 x = *reinterpret_cast<const uint4*>(row + 8 * (size_t)c);
      const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t p = (w[j >> 1] >> (16 * (j & 1))) & 0xFFFFu;
        const int idx = top - (int)(p & 0x7FFFu);
        const int at = idx < kTop ? idx + ((p & 0x8000u) ? kTop : 0) : kTop + idx;
        if (idx < kTop + kBoth) atomicAdd(&cnt.n[at], 1u);
      }
    }
    __syncthreads();
    for (int i = tid; i < kBins; i += NT) {
      cnt.f[i] = (float)cnt.n[i];
      val[i] = __uint_as_float((uint32_t)(top - (i < kTop ? i : i - kTop)) << 16) * unit;
    }
    __syncthreads();
    int k = 0;
    for (int task = tid; task < kTasks; task += NT, ++k) {
      const int third = task / kLpCount;
      const float d = step[task % kLpCount].d * unit, inv = __fdiv_rn(1.0f, d);
      const uint64_t inv2 = pack_f32x2(inv, inv), nd2 = pack_f32x2(-d, -d);
      uint64_t sum = 0;
      auto run = [&](auto clamp, int from, int to, float hi) {
#pragma unroll 4
        for (int i = from + 4 * third; i < to; i += 4 * kThirds) {
          const float4 v = *reinterpret_cast<const float4*>(val + i), n = *reinterpret_cast<const float4*>(cnt.f + i);
          sum = screen2<decltype(clamp)::value>(v.x, v.y, pack_f32x2(n.x, n.y), inv2, nd2, hi, sum);
          sum = screen2<decltype(clamp)::value>(v.z, v.w, pack_f32x2(n.z, n.w), inv2, nd2, hi, sum);
        }
      };
      run(std::integral_constant<int, 1>(), 0, kTop, 7.0f);
      run(std::integral_constant<int, 1>(), kTop, 2 * kTop, 8.0f);
      run(std::integral_constant<int, 0>(), 2 * kTop, kBins, 0.0f);
#pragma unroll
      for (int q = 0; q < kPer; ++q) if (q == k) acc[q] = both(sum);
    }
  } else {
    for (int c0 = 0; c0 < chunks; c0 += kChunk / 8) {
      __syncthreads();
      for (int c = tid; c < kChunk / 8; c += NT) {
        float x[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};        // a zero costs no error on any grid
        if (c0 + c < chunks) wload8(row + 8 * (size_t)(c0 + c), x);
#pragma unroll
        for (int j = 0; j < 8; ++j) val[8 * c + j] = x[j] * unit;
      }
      __syncthreads();
      const int n = min(kChunk, 8 * (chunks - c0));
      int k = 0;
      for (int task = tid; task < kTasks; task += NT, ++k) {
        const float d = step[task % kLpCount].d * unit, inv = __fdiv_rn(1.0f, d);
        const uint64_t inv2 = pack_f32x2(inv, inv), nd2 = pack_f32x2(-d, -d), one = pack_f32x2(1.0f, 1.0f);
        uint64_t sum = 0;
#pragma unroll 4
        for (int i = 4 * (task / kLpCount); i < n; i += 4 * kThirds) {
          const float4 v = *reinterpret_cast<const float4*>(val + i);
          sum = screen2<2>(v.x, v.y, one, inv2, nd2, 7.0f, sum);
          sum = screen2<2>(v.z, v.w, one, inv2, nd2, 7.0f, sum);
        }
#pragma unroll
        for (int q = 0; q < kPer; ++q) if (q == k) acc[q] += both(sum);
      }
    }
  }
  int k = 0;
  for (int task = tid; task < kTasks; task += NT, ++k) {
    double sum = 0.0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) if (q == k) sum = acc[q];
    part[task / kLpCount][task % kLpCount] = (float)sum;
  }
  __syncthreads();
  if (tid < 32) {
    float e[(kLpCount + 31) / 32], least = 3.4e38f;
#pragma unroll
    for (int j = 0; j < (kLpCount + 31) / 32; ++j) {
      const int i = 32 * j + lane;
      e[j] = i < kLpCount ? (part[0][i] + part[1][i]) + part[2][i] : 3.4e38f;
      least = fminf(least, e[j]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) least = fminf(least, __shfl_xor_sync(0xffffffffu, least, o));
    const float limit = least * (1.0f + 4.0f * kScreenEps) + 0x1p-110f;
    int n = 0;
#pragma unroll
    for (int j = 0; j < (kLpCount + 31) / 32; ++j) {
      const bool keep = 32 * j + lane < kLpCount && e[j] <= limit;
      const unsigned mask = __ballot_sync(0xffffffffu, keep);
      if (keep) list[n + __popc(mask & ((1u << lane) - 1u))] = (unsigned char)(32 * j + lane);
      n += __popc(mask);
    }
    if (lane == 0) *count = n;
  }
  __syncthreads();
  return true;
}

// The search: the candidate with the least sum_k |w - D q|^p, equal sums to the larger scale, sums that are not
// numbers left out; `fallback` where none is left.  Every thread returns the same step.
template <typename T, int NT, int kRange>
__device__ float lp_search(const T* row, int chunks, float a, bool no_nan, float p, int scale_dtype, float fallback) {
  __shared__ Step step[kLpCount];
  __shared__ double part[kLpCount][NT / 32];
  __shared__ float found;
  __shared__ unsigned char list[kLpCount];               // the candidates the float64 sums are taken for, ascending
  __shared__ int count;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < kLpCount; i += NT) {
    float d = store_round(__fdiv_rn(__fmul_rn(a, __fdiv_rn((float)(kLpFirst + i), 100.0f)), 7.0f), scale_dtype);
    if (a == 0.0f || d == 0.0f) d = 1.0f;
    step[i] = make_step(d);
  }
  for (int i = tid; i < kLpCount * (NT / 32); i += NT) (&part[0][0])[i] = 0.0;
  __syncthreads();
  bool screened = false;
  if constexpr (kRange == 2) screened = lp_screen<T, NT>(row, chunks, a, no_nan, step, list, &count);
  const int cands = screened ? count : kLpCount;
  constexpr int kPass = NT * (kLpHold / 8);
  int c0 = 0;
  for (; kRange == 2 ? c0 < chunks : kRange == 3 && c0 + kPass <= chunks; c0 += kPass) {
    float w[kLpHold];
    double w64[kLpHold];
#pragma unroll
    for (int h = 0; h < kLpHold / 8; ++h) {
      const int c = c0 + h * NT + tid;
      if (c < chunks) wload8(row + 8 * (size_t)c, w + 8 * h);
      else
#pragma unroll
        for (int j = 0; j < 8; ++j) w[8 * h + j] = 0.0f;   // a zero costs no error on any grid
    }
#pragma unroll
    for (int j = 0; j < kLpHold; ++j) w64[j] = (double)w[j];
    for (int n = 0; n < cands; ++n) {
      const int i = screened ? list[n] : n;
      const Step s = step[i];
      const double neg_d = -(double)s.d;
      const bool fast = no_nan && s.inv != 0.0f;
      int u[kLpHold];
      float close = 0.0f;
#pragma unroll
      for (int j = 0; j < kLpHold; ++j) {
        float far;
        u[j] = biased_mul(w[j], s.inv, far);
        close = fmaxf(close, far);
      }
      if (!fast || close > kTieClose) {                    // rare
#pragma unroll
        for (int j = 0; j < kLpHold; ++j) u[j] = biased_div(w[j], s.d);
      }
      double err[2] = {0.0, 0.0};
#pragma unroll
      for (int j = 0; j < kLpHold; ++j) {
        // 2^52 + u as float64 by its bit pattern, then q = u - 8: one exact add instead of a conversion
        const double q = __hiloint2double(0x43300000, u[j]) - (4503599627370496.0 + 8.0);
        // |w - D q|: the product of a 24-bit and a 4-bit number is exact in float64
        const double e = fabs(fma(neg_d, q, w64[j]));
        err[j & 1] = kRange == 2 ? fma(__dmul_rn(e, e), e, err[j & 1]) : err[j & 1] + pow(e, (double)p);
      }
      double sum = err[0] + err[1];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (lane == 0) part[i][warp] += sum;
    }
  }
  if constexpr (kRange != 2) power_sums<T, NT>(row, 8 * c0, 8 * chunks, step, part, no_nan, (double)p);
  __syncthreads();
  if (warp == 0) {
    double best = 1.0 / 0.0;
    int at = -1;
    for (int n = lane; n < cands; n += 32) {
      const int i = screened ? list[n] : n;
      double e = 0.0;
      for (int v = 0; v < NT / 32; ++v) e += part[i][v];
      if (e <= best) { best = e; at = i; }                 // i grows with n: ties to the larger scale
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double e2 = __shfl_xor_sync(0xffffffffu, best, o);
      const int a2 = __shfl_xor_sync(0xffffffffu, at, o);
      if (a2 >= 0 && (at < 0 || e2 < best || (e2 == best && a2 > at))) { best = e2; at = a2; }
    }
    if (lane == 0) found = at >= 0 ? step[at].d : fallback;
  }
  __syncthreads();
  return found;
}

// NT threads; V > 0: the row (at most NT * 8 * V values) is held in registers; V = 0: it is read again (from L1 or
// L2) in each pass.  kRange: 0 min-max, 1 L_p, 2 L_3, 3 L_p with sixteen values held by a thread; separate kernels, the
// searches need twice the registers of the rest.
template <typename T, int NT, int V, int kRange>
__global__ void __launch_bounds__(NT, kRange == 2 ? 768 / NT : 1) weight_quant_kernel(const T* __restrict__ W, int K, float p, int scale_dtype,
                                                          uint8_t* __restrict__ Wq, void* __restrict__ sw,
                                                          int32_t* __restrict__ wsum) {
  __shared__ float scratch_f[NT / 32];
  __shared__ int scratch_i[NT / 32];
  const int n = blockIdx.x, tid = threadIdx.x;
  const T* row = W + (size_t)n * (size_t)K;
  const int chunks = K >> 3;
  constexpr int R = V > 0 ? V : 1;
  float w[R][8];
  if constexpr (V > 0) {
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int c = i * NT + tid;
      if (c < chunks) wload8(row + 8 * c, w[i]);
      else
#pragma unroll
        for (int j = 0; j < 8; ++j) w[i][j] = 0.0f;      // a zero costs no error on any grid
    }
  }
  // f(values of a chunk, chunk index) over this thread's part of the row
  auto each_chunk = [&](auto f) {
    if constexpr (V > 0) {
#pragma unroll
      for (int i = 0; i < V; ++i) f(w[i], i * NT + tid);
    } else {
#pragma unroll (kRange == 0 ? 2 : 1)
      for (int c = tid; c < chunks; c += NT) {             // (two: 148 x 65536 in 22 instead of 26 us)
        float x[8];
        wload8(row + 8 * c, x);
        f(x, c);
      }
    }
  };

  float a = 0.0f;
  bool nan = false;
  each_chunk([&](const float (&x)[8], int) {
#pragma unroll
    for (int j = 0; j < 8; ++j) { a = fmaxf(a, fabsf(x[j])); nan = nan || x[j] != x[j]; }
  });
  const bool no_nan = __syncthreads_or(nan) == 0;
  a = block_reduce<NT>(a, scratch_f, true);

  float delta = store_round(__fdiv_rn(a, 7.0f), scale_dtype);
  if (a == 0.0f || delta == 0.0f) delta = 1.0f;
  if constexpr (kRange != 0) delta = lp_search<T, NT, kRange>(row, chunks, a, no_nan, p, scale_dtype, delta);
  if (tid == 0) {
    if (scale_dtype == FPT_DTYPE_F16) reinterpret_cast<__half*>(sw)[n] = __float2half_rn(delta);
    else reinterpret_cast<float*>(sw)[n] = delta;
  }
  int sum = 0;
  const Step fin = make_step(delta);
  const bool fast = no_nan && fin.inv != 0.0f;
  uint32_t* out = reinterpret_cast<uint32_t*>(Wq + (size_t)n * (size_t)(K / 2));
  each_chunk([&](const float (&x)[8], int c) {
    if (c >= chunks) return;
    // one branch for the eight divisions: with one for each value they followed one another, and a row of bf16 values can
    // be full of ties (64 x 4096: 4.1 -> 3.4 us; 14336 x 4096: 58.8 -> 53.3)
    int u[8];
    float close = 0.0f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float far;
      u[j] = biased_mul(x[j], fin.inv, far);
      close = fmaxf(close, far);
    }
    if (!fast || close > kTieClose) {
#pragma unroll
      for (int j = 0; j < 8; ++j) u[j] = biased_div(x[j], fin.d);
    }
    uint32_t word = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      sum += u[j] - 8;
      word |= (uint32_t)((u[j] - 8) & 0xF) << (4 * j);
    }
    out[c] = word;
  });
  if (wsum) {
    sum = block_reduce<NT>(sum, scratch_i, false);
    if (tid == 0) wsum[n] = sum;
  }
}

// Threads by the row's length: sixteen values a thread up to 4096 values, then more passes of the same CTA.  The
// min-max kernel holds up to 8192 values in registers.  The search with a general power: one value a thread;
// sixteen held ones where the rows are too few to fill the chip, so that as many chains of a thread hide the latency
// (p = 2, 64 x 4096: 0.70 -> 0.61 ms, 8 x 131072: 26 -> 19 ms; 4096 x 4096 the other way round: 11.3 -> 10.9 ms).
template <typename T, int kRange>
static void launch_weight_quant(cudaStream_t st, const T* W, int N, int K, float p, int scale_dtype, uint8_t* Wq,
                                void* sw, int32_t* wsum) {
  constexpr int V = kRange == 0 ? 2 : 0;
  auto go = [&](auto kern, int threads) { kern<<<N, threads, 0, st>>>(W, K, p, scale_dtype, Wq, sw, wsum); };
  if constexpr (kRange == 1) {
    if (K >= 16 * kWqThreads && N <= 2 * device_sm_count()) go(weight_quant_kernel<T, kWqThreads, 0, 3>, kWqThreads);
    else if (K > 128) go(weight_quant_kernel<T, kWqThreads, 0, 1>, kWqThreads);
    else if (K > 64) go(weight_quant_kernel<T, 128, 0, 1>, 128);
    else go(weight_quant_kernel<T, 64, 0, 1>, 64);
  } else if (K <= 1024) go(weight_quant_kernel<T, 64, V, kRange>, 64);
  else if (K <= 2048) go(weight_quant_kernel<T, 128, V, kRange>, 128);
  else if (K <= 4096) go(weight_quant_kernel<T, kWqThreads, V, kRange>, kWqThreads);
  else if (K <= 8192) go(weight_quant_kernel<T, kWqThreads, 2 * V, kRange>, kWqThreads);
  else go(weight_quant_kernel<T, kWqThreads, 0, kRange>, kWqThreads);
}
template <typename T>
static void quantize_rows(cudaStream_t st, const void* W, int N, int K, int range_mode, float p, int scale_dtype,
                          uint8_t* Wq, void* sw, int32_t* wsum) {
  const T* w = reinterpret_cast<const T*>(W);
  if (range_mode == FPT_RANGE_MINMAX) launch_weight_quant<T, 0>(st, w, N, K, p, scale_dtype, Wq, sw, wsum);
  else if (p == 3.0f) launch_weight_quant<T, 2>(st, w, N, K, p, scale_dtype, Wq, sw, wsum);
  else launch_weight_quant<T, 1>(st, w, N, K, p, scale_dtype, Wq, sw, wsum);
}

}  // namespace fpt

extern "C" int fpt_quantize_weights(void* stream, const void* W, int w_dtype, int N, int K, const fpt_qparams* qp,
                                    int range_mode, float p, int scale_dtype, uint8_t* Wq, void* sw, int32_t* wsum) {
  if (!W || !qp || !Wq || !sw || N <= 0 || K <= 0) return FPT_ERR_BAD_ARG;
  if (qp->bits != 4 || !qp->symmetric) return FPT_ERR_UNSUPPORTED;
  if (K % 32 != 0) return FPT_ERR_UNSUPPORTED;
  if (w_dtype != FPT_DTYPE_BF16 && w_dtype != FPT_DTYPE_F32) return FPT_ERR_BAD_ARG;
  if (scale_dtype != FPT_DTYPE_F32 && scale_dtype != FPT_DTYPE_F16) return FPT_ERR_BAD_ARG;
  if (range_mode != FPT_RANGE_MINMAX && range_mode != FPT_RANGE_LP) return FPT_ERR_BAD_ARG;
  if (range_mode == FPT_RANGE_LP && !(p > 0.0f)) return FPT_ERR_BAD_ARG;
  if (((uintptr_t)W | (uintptr_t)Wq | (uintptr_t)sw) & 15) return FPT_ERR_ALIGNMENT;
  cudaStream_t st = (cudaStream_t)stream;
  if (w_dtype == FPT_DTYPE_BF16) fpt::quantize_rows<__nv_bfloat16>(st, W, N, K, range_mode, p, scale_dtype, Wq, sw, wsum);
  else fpt::quantize_rows<float>(st, W, N, K, range_mode, p, scale_dtype, Wq, sw, wsum);
  return cudaGetLastError() == cudaSuccess ? FPT_OK : FPT_ERR_CUDA;
}

extern "C" int fpt_interleave_gate_up(void* stream, const uint8_t* Wg_q, const uint8_t* Wu_q, const void* sw_g,
                                      const void* sw_u, int scale_dtype, int d_ff, int K, uint8_t* Wgu_q,
                                      void* sw_gu) {
  if (!Wg_q || !Wu_q || !sw_g || !sw_u || !Wgu_q || !sw_gu || d_ff <= 0 || K <= 0) return FPT_ERR_BAD_ARG;
  if (d_ff % 64 != 0 || K % 32 != 0) return FPT_ERR_UNSUPPORTED;
  if (scale_dtype != FPT_DTYPE_F32 && scale_dtype != FPT_DTYPE_F16) return FPT_ERR_BAD_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t row = (size_t)K / 2, grp = 64 * row;           // bytes of 64 packed rows
  const size_t sgrp = 64 * (scale_dtype == FPT_DTYPE_F16 ? 2 : 4);
  const size_t groups = (size_t)d_ff / 64;
  cudaError_t e;
  e = cudaMemcpy2DAsync(Wgu_q, 2 * grp, Wg_q, grp, grp, groups, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpy2DAsync(Wgu_q + grp, 2 * grp, Wu_q, grp, grp, groups, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpy2DAsync(sw_gu, 2 * sgrp, sw_g, sgrp, sgrp, groups, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess)
    e = cudaMemcpy2DAsync((char*)sw_gu + sgrp, 2 * sgrp, sw_u, sgrp, sgrp, groups, cudaMemcpyDeviceToDevice, st);
  return e == cudaSuccess ? FPT_OK : FPT_ERR_CUDA;
}
