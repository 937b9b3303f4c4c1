// Round-to-nearest baseline (Section 5, "Baselines"): every weight rounded to the nearest value of
// exactly the grid the solver would use for untouched weights -- per-row or per-group min-max,
// asymmetric with an integer zero-point (or symmetric / ternary) -- with no error feedback.
// Output layout is that of gptq_quantize_layer.  One pass over W for groups that are multiples of 32 columns and per-row
// grids (rtn_span_kernel, rtn_held_kernel, rtn_fused_kernel), two plain passes for the small groups (4, 8, 16).
#include "common.cuh"

namespace gptq {
namespace {

struct RtnGrid { int maxq; int symmetric; int f16scale; };

__device__ __forceinline__ float storage_rounded(float scale, int f16scale) {
  if (!f16scale) return scale;
  const float s16 = __half2float(__float2half_rn(scale));
  return (s16 > 0.f && isfinite(s16)) ? s16 : scale;
}

// One warp per (row, group): min / max of the group -> scale (rounded to fp32), integer zero-point.
__global__ void rtn_params_kernel(const __half* __restrict__ W, int R, int C, int g, int G, RtnGrid grid,
                                  float* __restrict__ scales, float* __restrict__ zeros) {
  const int64_t wid = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (wid >= (int64_t)R * G) return;
  const int row = (int)(wid / G), gi = (int)(wid % G);
  const __half* p = W + (int64_t)row * C + (int64_t)gi * g;
  float mn = INFINITY, mx = -INFINITY;
  for (int i = lane; i < g; i += 32) { const float v = __half2float(p[i]); mn = fminf(mn, v); mx = fmaxf(mx, v); }
  for (int o = 16; o > 0; o >>= 1) {
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if (lane == 0) {
    double xmin = fmin((double)mn, 0.0), xmax = fmax((double)mx, 0.0);
    if (xmin == 0.0 && xmax == 0.0) { xmin = -1.0; xmax = 1.0; }
    float scale, zero;
    if (grid.symmetric) {
      scale = storage_rounded((float)(2.0 * fmax(fabs(xmin), xmax) / (double)grid.maxq), grid.f16scale);
      zero = (float)((grid.maxq + 1) / 2);
    } else {
      scale = storage_rounded((float)((xmax - xmin) / (double)grid.maxq), grid.f16scale);
      zero = (float)rint(-xmin / (double)scale);
    }
    scales[wid] = scale; zeros[wid] = zero;
  }
}

// One thread per packed word: quantizes the codes that overlap the word and assembles it.
__global__ void rtn_pack_kernel(const __half* __restrict__ W, int R, int C, int g, int G, int f, int maxq,
                                const float* __restrict__ scales, const float* __restrict__ zeros,
                                uint32_t* __restrict__ qweight) {
  const int nwords = C * f / 32;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)R * nwords) return;
  const int r = (int)(idx / nwords), k = (int)(idx % nwords);
  const __half* w = W + (int64_t)r * C;
  const int lo = 32 * k / f, hi = (32 * k + 31) / f;
  uint32_t word = 0;
  for (int col = lo; col <= hi; ++col) {
    const int gi = col / g;
    const double scale = (double)scales[(int64_t)r * G + gi], zero = (double)zeros[(int64_t)r * G + gi];
    double q = rint((double)__half2float(w[col]) / scale) + zero;
    q = fmin(fmax(q, 0.0), (double)maxq);
    const uint32_t v = (uint32_t)q;
    const int sh = col * f - 32 * k;
    word |= sh >= 0 ? (v << sh) : (v >> (-sh));
  }
  qweight[idx] = word;
}

// ---- one pass for groups that are multiples of 32 columns (and per-row grids) -----------------------------------
// Groups are bound by issue slots (78 % of them filled, 20 instructions a weight with what carries minima and grids between
// lanes); wider ones by the latency of their loads and what each row waits for between them (rtn_held_kernel).  So: one instruction
// a weight for the minimum and maximum (half2), few for the code, several loads in flight.  (12288 x 12288, 4-bit per row: 178 us
// with single-precision minima, a branch per code and one load in flight in the second pass, where the bytes alone take 57.)
__device__ __forceinline__ void rtn_grid_of(float mn, float mx, RtnGrid grid, float& scale, float& zero) {
  double xmin = fmin((double)mn, 0.0), xmax = fmax((double)mx, 0.0);
  if (xmin == 0.0 && xmax == 0.0) { xmin = -1.0; xmax = 1.0; }
  if (grid.symmetric) {
    scale = storage_rounded((float)(2.0 * fmax(fabs(xmin), xmax) / (double)grid.maxq), grid.f16scale);
    zero = (float)((grid.maxq + 1) / 2);
  } else {
    scale = storage_rounded((float)((xmax - xmin) / (double)grid.maxq), grid.f16scale);
    zero = (float)rint(-xmin / (double)scale);
  }
}
// Running minima and maxima of two interleaved halves of the weights.  The minimum passes NaNs over, as fminf does; the
// maximum keeps them, so that a group with one is known (rtn_finite) at no instruction per weight.
__device__ __forceinline__ void rtn_minmax8(const uint4& v, __half2& mn, __half2& mx) {
  const __half2* h = reinterpret_cast<const __half2*>(&v);
#pragma unroll
  for (int k = 0; k < 4; ++k) { mn = __hmin2(mn, h[k]); mx = __hmax2_nan(mx, h[k]); }
}
__device__ __forceinline__ __half2 rtn_half2_const(unsigned short bits) { return __halves2half2(__ushort_as_half(bits), __ushort_as_half(bits)); }
__device__ __forceinline__ float rtn_low(__half2 m) { return fminf(__low2float(m), __high2float(m)); }
__device__ __forceinline__ float rtn_high(__half2 m) {      // NaN if either half is
  const float a = __low2float(m), b = __high2float(m);
  return isnan(a) ? a : isnan(b) ? b : fmaxf(a, b);
}
// True if every weight of a group with these (kept) minimum and maximum is finite.
__device__ __forceinline__ bool rtn_finite(float mn, float mx) { return isfinite(mx) && isfinite(mn); }
// The maximum of pieces first, first + step, ... with NaNs passed over: for a group whose kept maximum is one.
__device__ __noinline__ float rtn_high_of_numbers(const uint4* p, int first, int pieces, int step) {
  float mx = -INFINITY;
#pragma unroll 1
  for (int i = first; i < pieces; i += step) {
    const uint4 v = __ldg(p + i);
    const __half2* h = reinterpret_cast<const __half2*>(&v);
    for (int k = 0; k < 4; ++k) mx = fmaxf(mx, fmaxf(__low2float(h[k]), __high2float(h[k])));
  }
  return mx;
}
template <bool kMin>
__device__ __forceinline__ __half2 rtn_reduce_step(__half2 m, int o) {
  const uint32_t u = __shfl_xor_sync(0xffffffffu, *reinterpret_cast<const uint32_t*>(&m), o);
  const __half2 x = *reinterpret_cast<const __half2*>(&u);
  return kMin ? __hmin2(m, x) : __hmax2_nan(m, x);
}
// The operation the oracle performs, for the eight weights of a piece.
template <int F>
__device__ __noinline__ uint64_t rtn_codes8_by_division(uint4 v, float scale, float zero, int maxq) {
  const __half2* h = reinterpret_cast<const __half2*>(&v);
  uint64_t bits = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float2 w2 = __half22float2(h[k >> 1]);
    const double q = fmin(fmax(rint((double)((k & 1) ? w2.y : w2.x) / (double)scale) + (double)zero, 0.0), (double)maxq);
    bits |= (uint64_t)(uint32_t)q << (k * F);
  }
  return bits;
}
// Eight codes of one 16-byte piece as 8 F bits.  A code is rne(w / scale) + zero, clamped.  w * (1 / scale) + zero + 1/2 is
// added to 1.5 * 2^I: the float then holds it in fixed point, S = 23 - I fraction bits below the integer, which a shift and
// one add-clamp turn into the code.  I leaves room for the code's range (a weight lies inside its own group's minimum and
// maximum).  The reciprocal's and the sum's rounding are below one unit 2^-S; wherever the fraction bits are within that of
// a tie (the constant is one unit high, so bits 0 .. 2) the eight weights go through the division.  So do all weights of a
// group with a NaN or an infinity in it, whose fixed-point values mean nothing (a NaN is 0x7FFFFFFF, which looks like a
// fraction far from a tie): the caller passes rs = 0 for such a group.
template <int F> constexpr int kRtnInt = F == 2 ? 4 : F == 3 ? 5 : F == 4 ? 6 : 10;
template <int F>
__device__ __forceinline__ uint64_t rtn_codes8(const uint4& v, float scale, float rs, float zero, int maxq) {
  constexpr int S = 23 - kRtnInt<F>;
  constexpr float kBig = 1.5f * (float)(1 << kRtnInt<F>);
  constexpr int kBias = (0x3F800000 + (kRtnInt<F> << 23) + 0x400000) >> S;     // upper bits of kBig
  const __half2* h = reinterpret_cast<const __half2*>(&v);
  const float base = zero + (kBig + 0.5f + 1.f / (float)(1 << S));
  uint32_t word[2] = {0u, 0u}, frac = rs > 0.f ? 0xFFFFFFFFu : 0u;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float2 w2 = __half22float2(h[k >> 1]);
    const int b = __float_as_int(fmaf((k & 1) ? w2.y : w2.x, rs, base));
    const uint32_t code = (uint32_t)__viaddmin_s32_relu(b >> S, -kBias, maxq);
    word[F == 8 ? k >> 2 : 0] += code << ((F == 8 ? k & 3 : k) * F);
    frac = min(frac, (uint32_t)b & ((1u << S) - 1u));
  }
  if (frac <= 2u) return rtn_codes8_by_division<F>(v, scale, zero, maxq);
  return F == 8 ? ((uint64_t)word[1] << 32) | word[0] : (uint64_t)word[0];
}
// The lanes of a warp hold consecutive pieces (piece index i, `on` = the piece exists); their 8 F bits become whole words
// of the row with at most one shuffle.  Every lane of the warp must call this.
template <int F>
__device__ __forceinline__ void rtn_store_words(uint32_t* qrow, int i, bool on, uint64_t bits, int lane) {
  if constexpr (F == 4) {
    if (on) qrow[i] = (uint32_t)bits;
  } else if constexpr (F == 8) {
    if (on) reinterpret_cast<uint2*>(qrow)[i] = make_uint2((uint32_t)bits, (uint32_t)(bits >> 32));
  } else if constexpr (F == 2) {
    const uint32_t mine = (uint32_t)bits, next = __shfl_down_sync(0xffffffffu, mine, 1);
    if ((lane & 1) == 0 && on) qrow[i >> 1] = mine | (next << 16);
  } else {                                                  // F == 3: four lanes' 24-bit runs make three words
    const uint32_t mine = (uint32_t)bits, next = __shfl_down_sync(0xffffffffu, mine, 1);
    const int k = lane & 3;
    const uint32_t word = k == 0 ? (mine | (next << 24)) : k == 1 ? ((mine >> 8) | (next << 16)) : ((mine >> 16) | (next << 8));
    if (k != 3 && on) qrow[3 * (i >> 2) + k] = word;
  }
}

// kThreads threads per (row, group) with at most kHeld pieces of 8 columns each: a thread loads its pieces (t, t + kThreads, ...) all at
// once and keeps them in registers, the group's minimum and maximum go through the warps and, if there are several, through shared
// memory, one thread derives the grid, and the codes are made from the registers.  W is read once.  One warp per group, eight of them to
// a CTA, or a CTA per group.  A group's load, minimum, grid and codes follow one another, so what counts is how many bytes of W an SM has
// on their way: the pieces fill the threads (kHeld and kThreads follow the group's width, see rtn_launch) and the minimum of CTAs per SM keeps a
// thread at 64 registers, 80 where a warp holds 6 or 8 (512 threads, 32768 columns: 2 CTAs an SM instead of 1, 107 instead of 154 us for 1.5e8 weights).
// (Spilled: 16 bytes in the 2- and 3-bit instances of 1024 threads, 8 in those of 768; nothing elsewhere.)
// 12288 x 12288, 4-bit: 90 us, where the bytes alone take 57 (192 threads; with 256 of them a quarter idle 103; rtn_fused_kernel, which reads W
// twice, half of it from DRAM: 112; a ring in shared memory that asynchronous copies fill one row ahead: 121).
template <int F, int kThreads, int kHeld>
__global__ void __launch_bounds__(kThreads == 32 ? 256 : kThreads, kThreads == 32 ? (kHeld <= 4 ? 4 : 3) : 1024 / kThreads)
rtn_held_kernel(const __half* __restrict__ W, int R, int C, int g, int G, RtnGrid grid,
                float* __restrict__ scales, float* __restrict__ zeros, uint32_t* __restrict__ qweight) {
  __shared__ float red[kThreads / 32][2], made[2];
  const int lane = threadIdx.x & 31, t = kThreads == 32 ? lane : threadIdx.x, warp = threadIdx.x >> 5;
  const int64_t wid = kThreads == 32 ? (int64_t)blockIdx.x * (blockDim.x >> 5) + warp : (int64_t)blockIdx.x;
  if (wid >= (int64_t)R * G) return;                        // (a whole warp; with more threads per group there is none)
  const int row = (int)(wid / G), gi = (int)(wid % G);
  const uint4* p = reinterpret_cast<const uint4*>(W + (int64_t)row * C + (int64_t)gi * g);
  const int pieces = g / 8;
  uint4 v[kHeld];
#pragma unroll
  for (int u = 0; u < kHeld; ++u)
    if (t + kThreads * u < pieces) v[u] = __ldcs(p + t + kThreads * u);
  __half2 mn = rtn_half2_const(0x7C00), mx = rtn_half2_const(0xFC00);        // +inf, -inf
#pragma unroll
  for (int u = 0; u < kHeld; ++u)
    if (t + kThreads * u < pieces) rtn_minmax8(v[u], mn, mx);
  for (int o = 16; o > 0; o >>= 1) { mn = rtn_reduce_step<true>(mn, o); mx = rtn_reduce_step<false>(mx, o); }
  float lo = rtn_low(mn), hi = rtn_high(mx);                // (the same in every lane)
  if constexpr (kThreads > 32) {
    if (lane == 0) { red[warp][0] = lo; red[warp][1] = hi; }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {               // (a NaN is kept)
      const float h = red[w][1];
      lo = fminf(lo, red[w][0]);
      hi = isnan(hi) ? hi : isnan(h) ? h : fmaxf(hi, h);
    }
  }
  const bool finite = rtn_finite(lo, hi);
  if (isnan(hi)) {                                          // (the same in every thread)
    hi = rtn_high_of_numbers(p, lane, pieces, 32);
    for (int o = 16; o > 0; o >>= 1) hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  float scale = 0.f, zero = 0.f;
  if (t == 0) {
    rtn_grid_of(lo, hi, grid, scale, zero);
    scales[wid] = scale; zeros[wid] = zero;
    if (kThreads > 32) { made[0] = scale; made[1] = zero; }
  }
  if constexpr (kThreads > 32) {
    __syncthreads();
    scale = made[0]; zero = made[1];
  } else {
    scale = __shfl_sync(0xffffffffu, scale, 0);
    zero = __shfl_sync(0xffffffffu, zero, 0);
  }
  const float rs = finite ? 1.0f / scale : 0.f;
  // words of this group inside the row: the group starts at bit gi * g * F, a multiple of 32 F bits
  uint32_t* qrow = qweight + (int64_t)row * (C / 32 * F) + (int64_t)gi * (g / 32 * F);
#pragma unroll
  for (int u = 0; u < kHeld; ++u) {
    if (kThreads * u >= pieces) break;                      // (uniform: every lane of a warp joins the shuffles)
    const int i = t + kThreads * u;
    const bool on = i < pieces;
    uint64_t bits = 0;
    if (on) bits = rtn_codes8<F>(v[u], scale, rs, zero, grid.maxq);
    rtn_store_words<F>(qrow, i, on, bits, lane);
  }
}

// One warp per (row, group), any group that is a multiple of 32 columns.  Phase A: the group's minimum and maximum from 16-byte loads (a
// lane takes the 8-column pieces lane, lane + 32, ...).  Phase B: the same pieces again, eight codes per lane, stored as whole words.
// Nothing waits for another warp, and 32 rows an SM are in flight: the faster form where there are many groups of a width that fills the
// threads of the form above badly, and the only one beyond 65536 columns.
template <int F>
__global__ void __launch_bounds__(256)
rtn_fused_kernel(const __half* __restrict__ W, int R, int C, int g, int G, RtnGrid grid,
                 float* __restrict__ scales, float* __restrict__ zeros, uint32_t* __restrict__ qweight) {
  const int64_t wid = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (wid >= (int64_t)R * G) return;
  const int row = (int)(wid / G), gi = (int)(wid % G);
  const uint4* p = reinterpret_cast<const uint4*>(W + (int64_t)row * C + (int64_t)gi * g);
  const int pieces = g / 8;
  __half2 mn = rtn_half2_const(0x7C00), mx = rtn_half2_const(0xFC00);        // +inf, -inf
  int i0 = lane;
  for (; i0 + 96 < pieces; i0 += 128) {                     // four loads in flight per lane
    const uint4 a = __ldg(p + i0), b = __ldg(p + i0 + 32), c = __ldg(p + i0 + 64), d = __ldg(p + i0 + 96);
    rtn_minmax8(a, mn, mx); rtn_minmax8(b, mn, mx); rtn_minmax8(c, mn, mx); rtn_minmax8(d, mn, mx);
  }
  for (; i0 < pieces; i0 += 32) { const uint4 a = __ldg(p + i0); rtn_minmax8(a, mn, mx); }
  for (int o = 16; o > 0; o >>= 1) { mn = rtn_reduce_step<true>(mn, o); mx = rtn_reduce_step<false>(mx, o); }
  float lo = rtn_low(mn), hi = rtn_high(mx);                // (the same in every lane)
  const bool finite = rtn_finite(lo, hi);
  if (isnan(hi)) {
    hi = rtn_high_of_numbers(p, lane, pieces, 32);
    for (int o = 16; o > 0; o >>= 1) hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  float scale = 0.f, zero = 0.f;
  if (lane == 0) {
    rtn_grid_of(lo, hi, grid, scale, zero);
    scales[wid] = scale; zeros[wid] = zero;
  }
  scale = __shfl_sync(0xffffffffu, scale, 0);
  zero = __shfl_sync(0xffffffffu, zero, 0);
  const float rs = finite ? 1.0f / scale : 0.f;
  // words of this group inside the row: the group starts at bit gi * g * F, a multiple of 32 F bits
  uint32_t* qrow = qweight + (int64_t)row * (C / 32 * F) + (int64_t)gi * (g / 32 * F);
  int base = 0;
#pragma unroll 1
  for (; base + 128 <= pieces; base += 128) {               // four loads in flight per lane
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = __ldg(p + base + 32 * u + lane);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      rtn_store_words<F>(qrow, base + 32 * u + lane, true, rtn_codes8<F>(v[u], scale, rs, zero, grid.maxq), lane);
  }
  for (; base < pieces; base += 32) {                       // uniform trip count: every lane joins the shuffles
    const int i = base + lane;
    const bool on = i < pieces;
    uint64_t bits = 0;
    if (on) { const uint4 v = __ldg(p + i); bits = rtn_codes8<F>(v, scale, rs, zero, grid.maxq); }
    rtn_store_words<F>(qrow, i, on, bits, lane);
  }
}

// Groups of 32, 64, 128 or 256 columns: one warp per run of 32 groups of a row (32 g columns), a group on g / 8
// neighbouring lanes of one 256-column span.  First pass over the run's spans: the group's lanes reduce minimum and
// maximum among themselves and hand them to the lane that owns the group (group t of the run belongs to lane t), so that
// the 32 grids of the run are derived in one go, one per lane.  Second pass: the spans again (from L1 / L2: at most 8 KB
// per warp, just read), quantized with their groups' grids fetched by shuffles.  Both loops stay rolled: the code is
// small enough for the instruction cache.
template <int F, int kLanes>                                // kLanes = g / 8 = lanes per group = spans of one run
__global__ void __launch_bounds__(256)
rtn_span_kernel(const __half* __restrict__ W, int R, int C, int G, RtnGrid grid,
                float* __restrict__ scales, float* __restrict__ zeros, uint32_t* __restrict__ qweight) {
  constexpr int kGroupsPerSpan = 32 / kLanes;
  const int runs = (G + 31) / 32;
  const int64_t wid = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (wid >= (int64_t)R * runs) return;
  const int row = (int)(wid / runs), run = (int)(wid % runs);
  const int piece0 = run * 32 * kLanes;                     // first piece of the run inside the row
  const int row_pieces = C / 8;
  const uint4* p = reinterpret_cast<const uint4*>(W + (int64_t)row * C);
  float my_mn = INFINITY, my_mx = -INFINITY;                // of the group this lane owns (group `lane` of the run)
#pragma unroll 4
  for (int sp = 0; sp < kLanes; ++sp) {
    const int i = piece0 + sp * 32 + lane;
    __half2 mn2 = rtn_half2_const(0x7C00), mx2 = rtn_half2_const(0xFC00);    // +inf, -inf
    if (i < row_pieces) { const uint4 v = __ldg(p + i); rtn_minmax8(v, mn2, mx2); }
#pragma unroll
    for (int o = 1; o < kLanes; o <<= 1) { mn2 = rtn_reduce_step<true>(mn2, o); mx2 = rtn_reduce_step<false>(mx2, o); }
    const float mn = rtn_low(mn2), mx = rtn_high(mx2);
    // group t = sp * kGroupsPerSpan + j of the run sits on lanes j * kLanes ..; its owner is lane t
    const int j = lane - sp * kGroupsPerSpan;               // which group of this span this lane owns, if any
    const float gmn = __shfl_sync(0xffffffffu, mn, (j & (kGroupsPerSpan - 1)) * kLanes);
    const float gmx = __shfl_sync(0xffffffffu, mx, (j & (kGroupsPerSpan - 1)) * kLanes);
    if (j >= 0 && j < kGroupsPerSpan) { my_mn = gmn; my_mx = gmx; }
  }
  float my_scale = 1.f, my_zero = 0.f;
  const int my_group = run * 32 + lane;
  const bool finite = rtn_finite(my_mn, my_mx);
  if (my_group < G) {
    if (isnan(my_mx)) my_mx = rtn_high_of_numbers(p, my_group * kLanes, (my_group + 1) * kLanes, 1);
    rtn_grid_of(my_mn, my_mx, grid, my_scale, my_zero);
    scales[(int64_t)row * G + my_group] = my_scale;
    zeros[(int64_t)row * G + my_group] = my_zero;
  }
  const float my_rs = finite ? 1.0f / my_scale : 0.f;
  uint32_t* qrow = qweight + (int64_t)row * (C / 32 * F);
#pragma unroll 1
  for (int sp = 0; sp < kLanes; ++sp) {
    const int i = piece0 + sp * 32 + lane;
    const int owner = sp * kGroupsPerSpan + lane / kLanes;  // lane that owns this lane's group in span sp
    const float scale = __shfl_sync(0xffffffffu, my_scale, owner), rs = __shfl_sync(0xffffffffu, my_rs, owner);
    const float zero = __shfl_sync(0xffffffffu, my_zero, owner);
    const bool on = i < row_pieces;
    uint64_t bits = 0;
    if (on) { const uint4 v = __ldg(p + i); bits = rtn_codes8<F>(v, scale, rs, zero, grid.maxq); }
    rtn_store_words<F>(qrow, i, on, bits, lane);
  }
}

// Which form a group of g columns gets.  A warp's 32 lanes hold 4, 6 or 8 pieces each, a CTA's threads 8.  Where W is large and the group
// has fewer columns than its form's `least`, rtn_fused_kernel: it needs a few waves of rows to get going (below 1e8 weights the forms that
// hold a group win or tie at every width: 8000 rows of 4096 columns 24 against 26 us, of 10240 57 against 69), and from there on its time per weight
// hardly depends on the width; beyond 2.5e8 weights it is the faster one up to 8192 columns.  Few groups leave SMs idle, so a group gets the
// next wider CTA there (300 rows: 3072 columns on 64 / 128 threads 7.8 / 6.2 us, 12288 on 192 / 256 10.3 / 8.3).  Both sides, 4-bit, held / fused, 1.5e8 weights:
// 288 columns 281 / 330 us, 1024 113 / 117, 1536 99 / 125, 1920 102 / 130, 2048 101 / 97, 2560 101 / 108, 3072 94 / 93, 4096 86 / 85, 5120 92 / 87, 6144 88 / 92,
// 8192 89 / 94, 9216 102 / 98, 10240 97 / 101, 11264 95 / 109, 12288 90 / 112, 16384 92 / 124, 18432 125 / 130, 24576 111 / 141, 32768 107 / 146,
// 36864 160 / 151, 40960 152 / 145 (8-bit 183 / 223: the 768 threads are kept), 49152 140 / 159, 65536 135 / 170;
// 3e8 weights: 4096 163 / 156, 8192 166 / 159, 10240 185 / 170, 12288 172 / 187, 20480 232 / 230, 24576 214 / 236, 40960 296 / 261, 65536 259 / 279.
template <int F>
void rtn_launch(const __half* W, int R, int C, int g, int G, RtnGrid grid, float* scales, float* zeros, uint32_t* qweight, cudaStream_t s) {
  const int64_t groups = (int64_t)R * G, runs = (int64_t)R * ((G + 31) / 32);
  const auto warps = [](int64_t n) { return (unsigned)((n + 7) / 8); };
  if (g == 32) { rtn_span_kernel<F, 4><<<warps(runs), 256, 0, s>>>(W, R, C, G, grid, scales, zeros, qweight); return; }
  if (g == 64) { rtn_span_kernel<F, 8><<<warps(runs), 256, 0, s>>>(W, R, C, G, grid, scales, zeros, qweight); return; }
  if (g == 128) { rtn_span_kernel<F, 16><<<warps(runs), 256, 0, s>>>(W, R, C, G, grid, scales, zeros, qweight); return; }
  if (g == 256) { rtn_span_kernel<F, 32><<<warps(runs), 256, 0, s>>>(W, R, C, G, grid, scales, zeros, qweight); return; }
  using Kernel = void (*)(const __half*, int, int, int, int, RtnGrid, float*, float*, uint32_t*);
  struct Form { int widest, least, threads; Kernel kernel; };    // (least 2049: no group of 2048 columns where W is large)
  static const Form forms[] = {
      {1024, 0, 32, rtn_held_kernel<F, 32, 4>},      {1536, 0, 32, rtn_held_kernel<F, 32, 6>},      {2016, 0, 32, rtn_held_kernel<F, 32, 8>},
      {2048, 2049, 32, rtn_held_kernel<F, 32, 8>},   {4096, 3328, 64, rtn_held_kernel<F, 64, 8>},   {6144, 5632, 96, rtn_held_kernel<F, 96, 8>},
      {8192, 6656, 128, rtn_held_kernel<F, 128, 8>}, {12288, 11264, 192, rtn_held_kernel<F, 192, 8>}, {16384, 0, 256, rtn_held_kernel<F, 256, 8>},
      {24576, 22528, 384, rtn_held_kernel<F, 384, 8>}, {32768, 0, 512, rtn_held_kernel<F, 512, 8>}, {49152, F == 8 ? 0 : 45056, 768, rtn_held_kernel<F, 768, 8>},
      {65536, 0, 1024, rtn_held_kernel<F, 1024, 8>}};
  const int64_t weights = groups * g;
  for (const Form& form : forms) {
    if (g > form.widest || (groups <= 1024 && (form.threads == 64 || form.threads == 96 || form.threads == 192))) continue;
    if ((g < form.least && weights > 100000000) || (g >= 2048 && g <= 8192 && weights > 250000000)) break;
    if (form.threads == 32) form.kernel<<<warps(groups), 256, 0, s>>>(W, R, C, g, G, grid, scales, zeros, qweight);
    else form.kernel<<<(unsigned)groups, form.threads, 0, s>>>(W, R, C, g, G, grid, scales, zeros, qweight);
    return;
  }
  rtn_fused_kernel<F><<<warps(groups), 256, 0, s>>>(W, R, C, g, G, grid, scales, zeros, qweight);
}

}  // namespace
}  // namespace gptq

extern "C" gptq_status_t gptq_rtn_layer(const void* W_fp16, int R, int C, int bits, int group_size, int sym,
                                        uint32_t* qweight, float* scales, float* zeros, void* stream) {
  using namespace gptq;
  if (!W_fp16 || !qweight || !scales || !zeros || R <= 0 || C <= 0 || C % 32 != 0) return GPTQ_ERR_INVALID_ARG;
  if (!(bits == 2 || bits == 3 || bits == 4 || bits == 8 || bits == GPTQ_BITS_TERNARY)) return GPTQ_ERR_UNSUPPORTED;
  const int g = group_size > 0 ? group_size : C;
  if (C % g != 0) return GPTQ_ERR_INVALID_ARG;
  const int G = C / g, f = bits == GPTQ_BITS_TERNARY ? 2 : bits;
  if (sym & ~(GPTQ_GRID_SYMMETRIC | GPTQ_GRID_FP16_SCALES)) return GPTQ_ERR_INVALID_ARG;
  RtnGrid grid{bits == GPTQ_BITS_TERNARY ? 2 : (1 << bits) - 1, ((sym & GPTQ_GRID_SYMMETRIC) != 0 || bits == GPTQ_BITS_TERNARY) ? 1 : 0,
               (sym & GPTQ_GRID_FP16_SCALES) ? 1 : 0};
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const __half* W = static_cast<const __half*>(W_fp16);
  if (g % 32 == 0 && aligned_to(W_fp16, 16)) {              // one pass; (row, group) starts are then 16-byte aligned too
    switch (f) {
      case 2: rtn_launch<2>(W, R, C, g, G, grid, scales, zeros, qweight, s); break;
      case 3: rtn_launch<3>(W, R, C, g, G, grid, scales, zeros, qweight, s); break;
      case 4: rtn_launch<4>(W, R, C, g, G, grid, scales, zeros, qweight, s); break;
      default: rtn_launch<8>(W, R, C, g, G, grid, scales, zeros, qweight, s); break;
    }
    GPTQ_LAUNCH_CHECK();
    return GPTQ_OK;
  }
  {
    const int64_t warps = (int64_t)R * G;
    rtn_params_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(W, R, C, g, G, grid, scales, zeros);
    GPTQ_LAUNCH_CHECK();
  }
  {
    const int64_t total = (int64_t)R * (C * f / 32);
    rtn_pack_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(W, R, C, g, G, f, grid.maxq, scales, zeros, qweight);
    GPTQ_LAUNCH_CHECK();
  }
  return GPTQ_OK;
}
