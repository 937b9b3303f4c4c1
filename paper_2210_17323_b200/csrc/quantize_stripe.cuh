// Row-stripe form of Algorithm 1's loops inside one outer block (included by quantize.cu, inside its
// namespace, after GridSpec / find_params).
//
// Rows of W are independent sub-problems (Section 2), so one CTA can own a stripe of 128 rows for a whole
// outer block of columns and run every inner block of it back to back with no other CTA involved:
//   for each inner block of B columns (Section 3, Step 2), for each 16 columns of it: quantize them one after the other
//   with immediate error feedback (Algorithm 1's inner loop) -- ONE THREAD PER ROW, fp64, the 16 columns in registers --
//   then push their 16 errors onto later columns of the outer block (Algorithm 1's lazy update).
// The pushes are products of the stripe's errors with a panel of U and run on the tensor cores: the row threads write
// their scaled errors as an fp16 hi / lo pair into a 128-byte-swizzled K-major tile, which is the M = 128 left operand of
// tcgen05.mma (kind::f16, three products per term as in gemm_umma_f16.cuh); the right operand is the transposed scaled
// fp16 pair of U that quantize.cu prepares.  What bounds the kernel is the chain of one row: 16 columns, push, 16
// columns, push, ...; everything that the next 16 columns do not need is kept off it, by distance of the target columns:
//   this block and the next one   after every 16 columns, K = 16, into TMEM accumulators that stay there (one set for the
//                                 rest of the block, one for the next block: at most 24 MMAs each); a thread subtracts
//                                 the two sums from its next 16 columns when it reaches them.  A block boundary is
//                                 therefore a step like any other.
//   everything further right      once per block, K = B, in 64-column tiles, WHILE the next block runs: own issuing warp,
//                                 own four drain warps, a second error tile.  The sums leave as f64 reductions onto the
//                                 working weights in global memory, 256 consecutive bytes per warp instruction.
// Beside the chain it is the shared-memory pipe that counts (per column of 128 rows: 60 cycles for the doubles of U that every
// row thread reads, and what the MMAs read of their operands): 64-column far tiles read the error tile half as often as
// 32-column ones, and sums on their way through a shared-memory buffer (bulk reductions) cost 42 cycles a column.
// The columns themselves are read straight from the working weights, sixteen ahead of their use.
// Measured (4096 rows, per-row grids, cycles per 128 columns on an SM): the form with the pushes onto later blocks in line
// and the block's columns staged in shared memory took 71,000 (27,000 of them in that drain, 23,000 in the columns).
// The whole outer block is one launch, and nothing in it waits for another CTA.  Left-looking updates ACROSS outer blocks
// stay with the large two-CTA contraction.
//
// Threads: warps 0-3 own the rows (thread t <-> row t <-> TMEM lane t); warp 4 issues the near pushes, warp 5 the far ones,
// warp 6 stages U's diagonal blocks, warp 7 has nothing to do, warps 8-11 drain the far pushes.  A row thread needs 200
// registers and more (32 doubles of weights); at 168 the loads that run ahead are spilled, and so waited for.  So the three
// warpgroups share out the registers anew: 248 + 112 + 136 of the 3 x 168 the kernel is launched with.
// Neither instance spills.
#pragma once

constexpr int kStripeRows = 128;
constexpr int kStripeThreads = 384;
constexpr int kStripeSB = 16;                 // columns held in registers at a time
constexpr int kStripeMaxB = 128;              // widest inner block this form takes
constexpr int kStripeNT = 64;                 // columns of a far push per TMEM accumulator / staged panel tile
constexpr int kStripeMaxNb2 = 2048;           // widest outer block this form takes

struct StripeMaps { CUtensorMap p_hi, p_lo;    // Pt[c - i2][k] of the outer block: boxes of 64 k x 64 columns, 128-byte swizzle
                    CUtensorMap s_hi, s_lo; }; // the same in boxes of 16 k x 32 columns, 32-byte swizzle

// Working weights of the outer block in STRIPE-MAJOR order: element (row, col) at ((row / 128) * ldw + col) * 128 + row % 128,
// so that the 128 row threads of a stripe read one column of it as 1 KB of consecutive doubles.
struct StripeArgs {
  double* Wblk; int64_t ldw; int nb2;         // working weights of the outer block (stripe-major, see above), its width
  const float* U; int C; int i2;              // first global column of the outer block
  int B;                                      // inner block width: multiple of 32, <= kStripeMaxB
  int R; GridSpec grid; int group;
  float* scales; float* zeros; int G;
  __half* Ehi; __half* Elo;                   // scaled errors E' (see quantize.cu), all columns
  const float* sK; const float* sE; const float* sEinv; const float* sCinv;
  uint8_t* codes; double* loss; int* dev_info;
  int keep_errors;                            // 1: the scaled errors also go to Ehi / Elo in global memory (the left operand of
                                              // later outer blocks' contractions); 0: factor form, a separate kernel writes the
                                              // plain residuals there from the codes
};

// What the sixteen columns of a sub-block need of U: its diagonal block with rows divided by U_jj, 1 / U_jj, sK and 1 / sC.
struct StripeCols { double U[kStripeSB][kStripeSB]; double rdiag[kStripeSB]; float sks[kStripeSB]; float sci[kStripeSB]; };

// shared memory (from a 1024-byte aligned base):
//   error tiles   two (one per parity of the block): hi then lo, each two 64-wide K atoms of [128 rows][128 bytes], swizzled
//   far panel     three stages: hi and lo of one K atom, [64 columns][128 bytes]
//   near panel    two slices: hi and lo, each [<= 256 columns][16 k], 32-byte swizzle
//   StripeCols    two; then the barriers and the TMEM slot
constexpr int kStripeETile = 65536, kStripeStage = 16384, kStripeStages = 3, kStripeSlice = 8192;
constexpr int kStripeOffFar = 2 * kStripeETile, kStripeOffSlice = kStripeOffFar + kStripeStages * kStripeStage;
constexpr int kStripeOffCols = kStripeOffSlice + 4 * kStripeSlice;
constexpr int kStripeOffBars = kStripeOffCols + 2 * (int)sizeof(StripeCols);
struct StripeBars {
  uint64_t cols_full[2], cols_empty[2];       // StripeCols: stager -> row warps -> stager
  uint64_t slice_full[2], slice_empty[2];     // near panel: TMA -> MMA -> TMA
  uint64_t errors;                            // a sub-block's errors are in the tile: row warps -> near pushes
  uint64_t near_done, rest_done;              // its pushes: the next 16 columns' / all of them have been added
  uint64_t block_errors[2];                   // a block's errors are complete: row warps -> far pushes
  uint64_t tile_free[2];                      // the far pushes have read the block's error tile
  uint64_t stage_full[kStripeStages], stage_empty[kStripeStages];     // far panel
  uint64_t acc_full[2], acc_empty[2];         // far accumulators
  uint64_t next_ready[2], all_ready[2];       // the far pushes have reached memory: onto the block after next / all
  uint64_t settled[2];                        // everything that the near / the far pushes have issued is over
  uint32_t tmem;
};
constexpr int kStripeSmem = 1024 + kStripeOffBars + (int)sizeof(StripeBars);
// TMEM columns: sums for the rest of the block, for the next block (by parity), two far accumulators
constexpr uint32_t kTmemRest = 0, kTmemNext = 128, kTmemFar = 384;

// 32 lanes x 16 consecutive fp32 columns of TMEM (warp w reads lanes 32 * (w % 4) ..)
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
// Shared-memory matrix descriptor of a K-major operand 16 fp16 (32 bytes) deep, 32-byte swizzle: 8-row groups 256 B apart.
__device__ __forceinline__ uint64_t make_desc_sw32(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)(256 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)6 << 61;
  return d;
}
// Three products of a pair by a pair: small terms first.
__device__ __forceinline__ void mma_pairs(uint32_t d_tmem, uint64_t ah, uint64_t al, uint64_t bh, uint64_t bl, uint32_t idesc, bool fresh) {
  umma::mma_f16(d_tmem, al, bh, idesc, fresh ? 0u : 1u);
  umma::mma_f16(d_tmem, ah, bl, idesc, 1u);
  umma::mma_f16(d_tmem, ah, bh, idesc, 1u);
}

// Out-of-line pieces of the column loop (kept out of the unrolled body so that it stays small).
__device__ __noinline__ float2 find_params_outofline(double mn, double mx, GridSpec g) {
  float2 r;
  find_params(mn, mx, g, r.x, r.y);
  return r;
}

// A row's current grid, with what the column loop derives from it once per grid.
struct RowGrid {
  double scale, rscale, zero;
  double kz;                            // 2^52 + zero-point: what a code's bits with that exponent stand above code - zero-point
  int bias;                             // what turns the column loop's count, 2048 + code - zero-point, into the code
  __device__ __forceinline__ void set(float2 sz) {
    scale = (double)sz.x; zero = (double)sz.y; rscale = 1.0 / scale;
    kz = 4503599627370496.0 + (double)(int)sz.y; bias = (int)sz.y - 2048;
  }
};
// One column with the division itself, fp64 throughout: for weights whose quotient lies next to a tie (where the
// reciprocal's last-bit error could change the rounding), outside the 32-bit range, or is not finite.
__device__ __noinline__ double column_by_division(double w, double scale, double zero, double maxq, uint32_t* code) {
  double q = rint(w / scale) + zero;
  q = fmin(fmax(q, 0.0), maxq);
  *code = (uint32_t)q;
  return w - scale * (q - zero);
}

// ---- pieces of the row threads' loop ------------------------------------------------------------------
// Sixteen columns of the working weights as memory holds them (rows beyond the matrix: zero, so that nothing of them is ever
// pushed).  Reductions of this launch changed them, so L1 is bypassed.
__device__ __forceinline__ void stripe_fetch(const double* wcol, bool live, double (&x)[kStripeSB]) {
#pragma unroll
  for (int m = 0; m < kStripeSB; ++m) x[m] = live ? __ldcg(wcol + (int64_t)m * kStripeRows) : 0.0;
}
// x -= the sums in sixteen TMEM columns: sum / (sE[row] sC[column])
__device__ __forceinline__ void stripe_subtract(uint32_t taddr, const float* sci, double inv_se, double (&x)[kStripeSB]) {
  float v[kStripeSB];
  tmem_ld_32x16(taddr, v);
  umma::tmem_ld_wait();
#pragma unroll
  for (int m = 0; m < kStripeSB; ++m) x[m] -= (double)(v[m] * sci[m]) * inv_se;
}
// Where a row's columns stand: memory minus what has been pushed onto them and not gone there.
struct StripeAt {
  const double* wcol;                   // first of the columns
  const float* sCinv;                   // 1 / sC of the same columns
  uint32_t next, rest;                  // TMEM columns of the two sums
  bool has_next, has_rest, live;
  double inv_se;
};
// Grid from the minimum and maximum of the row's CURRENT weights in `width` columns, of which the first `pending` have sums
// in TMEM (Section 5, grouping).  Out of line, like everything that not every sub-block runs: the loop of the row threads
// is a few thousand instructions long, and cold code between them costs instruction fetch (136 instead of 95 cycles a
// column in a small model of the loop).
// Two forms: stripe_scan starts from memory; stripe_scan_rest goes on behind the first sixteen columns, whose minimum and maximum the caller
// has from its registers, and is a third shorter for groups of 32 (1000 x 2400, 64-column blocks: 858 -> 795 us; groups of 64, 2048 x 2048
// 604 -> 590).  For wider groups it saves less than the weights that the caller then holds across the call cost (groups of 128, 4096 x 1024
// 273.5 -> 276.5 us), so those keep the first, in an instance of the kernel of their own with the per-row grids (224.8 -> 228.1 there).
__device__ __noinline__ float2 stripe_scan(const StripeAt& at, int width, int pending, GridSpec gs) {
  double mn = INFINITY, mx = -INFINITY, x[kStripeSB], y[kStripeSB];
  stripe_fetch(at.wcol, at.live, x);
#pragma unroll 1
  for (int c = 0; c < width; c += kStripeSB) {
    if (c + kStripeSB < width) stripe_fetch(at.wcol + (int64_t)(c + kStripeSB) * kStripeRows, at.live, y);
    if (c < pending) {
      float sc[kStripeSB];
#pragma unroll
      for (int m = 0; m < kStripeSB; ++m) sc[m] = __ldg(at.sCinv + c + m);
      if (at.has_next) stripe_subtract(at.next + c, sc, at.inv_se, x);
      if (at.has_rest) stripe_subtract(at.rest + c, sc, at.inv_se, x);
    }
#pragma unroll
    for (int m = 0; m < kStripeSB; ++m) { mn = x[m] < mn ? x[m] : mn; mx = x[m] > mx ? x[m] : mx; x[m] = y[m]; }
  }
  float2 r;
  find_params(mn, mx, gs, r.x, r.y);
  return r;
}
__device__ __noinline__ float2 stripe_scan_rest(const StripeAt& at, int width, int pending, GridSpec gs, double mn, double mx) {
  double x[kStripeSB], y[kStripeSB];
  stripe_fetch(at.wcol + (int64_t)kStripeSB * kStripeRows, at.live, x);
#pragma unroll 1
  for (int c = kStripeSB; c < width; c += kStripeSB) {
    if (c + kStripeSB < width) stripe_fetch(at.wcol + (int64_t)(c + kStripeSB) * kStripeRows, at.live, y);
    if (c < pending) {
      float sc[kStripeSB];
#pragma unroll
      for (int m = 0; m < kStripeSB; ++m) sc[m] = __ldg(at.sCinv + c + m);
      if (at.has_next) stripe_subtract(at.next + c, sc, at.inv_se, x);
      if (at.has_rest) stripe_subtract(at.rest + c, sc, at.inv_se, x);
    }
#pragma unroll
    for (int m = 0; m < kStripeSB; ++m) { mn = x[m] < mn ? x[m] : mn; mx = x[m] > mx ? x[m] : mx; x[m] = y[m]; }
  }
  float2 r;
  find_params(mn, mx, gs, r.x, r.y);
  return r;
}
// Small groups (4, 8 or 16 columns): their grids are taken from the weights in registers, inside the column loop.
struct StripeGroups { int g; uint32_t starts; GridSpec gs; float* scales; float* zeros; bool live; };
__device__ __forceinline__ void stripe_small_group(const StripeGroups& sg, int jj, const double (&w)[kStripeSB], RowGrid& grid) {
  double mn = INFINITY, mx = -INFINITY;
#pragma unroll
  for (int m = 0; m < kStripeSB; ++m)
    if (m >= jj && m < jj + sg.g) { mn = w[m] < mn ? w[m] : mn; mx = w[m] > mx ? w[m] : mx; }
  const float2 sz = find_params_outofline(mn, mx, sg.gs);
  grid.set(sz);
  if (sg.live) { sg.scales[jj / sg.g] = sz.x; sg.zeros[jj / sg.g] = sz.y; }
}
// The sixteen columns once more, with the division itself in every one of them.
struct StripeRedo { float err[kStripeSB]; uint32_t cw[kStripeSB / 4]; double loss; };
template <bool kSmallGroups>
__device__ __noinline__ void stripe_redo(const StripeAt& at, const StripeCols& cs, RowGrid grid, const StripeGroups& sg, StripeRedo& out) {
  double w[kStripeSB];
  stripe_fetch(at.wcol, at.live, w);
  if (at.has_next) stripe_subtract(at.next, cs.sci, at.inv_se, w);
  if (at.has_rest) stripe_subtract(at.rest, cs.sci, at.inv_se, w);
  out.loss = 0.0;
#pragma unroll
  for (int m = 0; m < kStripeSB / 4; ++m) out.cw[m] = 0;
#pragma unroll
  for (int jj = 0; jj < kStripeSB; ++jj) {
    if (kSmallGroups && (jj & 3) == 0 && ((sg.starts >> jj) & 1u)) stripe_small_group(sg, jj, w, grid);
    uint32_t code;
    const double r = column_by_division(w[jj], grid.scale, grid.zero, (double)sg.gs.maxq, &code), e = r * cs.rdiag[jj];
    out.err[jj] = (float)e;
    out.loss = fma(e, e, out.loss);
    out.cw[jj >> 2] |= code << (8 * (jj & 3));
#pragma unroll
    for (int m = 0; m < kStripeSB; ++m)
      if (m > jj) w[m] = fma(-r, cs.U[jj][m], w[m]);
  }
}
// Two scaled errors as fp16 pairs: the two high parts and the two remainders, saturating.
__device__ __forceinline__ void stripe_split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(x1), "f"(x0));
  const __half2 h = *reinterpret_cast<const __half2*>(&hi);
  const float2 f = __half22float2(h);
  asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(x1 - f.y), "f"(x0 - f.x));
}

// ---- the roles ------------------------------------------------------------------------------------
// Block b covers columns [b B, b B + width) of the outer block; `next` columns follow in block b + 1 and `far` after that.
struct StripeBlock { int ib, width, next, far; };
__device__ __forceinline__ StripeBlock stripe_block(const StripeArgs& a, int b) {
  StripeBlock k;
  k.ib = b * a.B;
  k.width = min(a.B, a.nb2 - k.ib);
  k.next = min(a.B, a.nb2 - k.ib - k.width);
  k.far = a.nb2 - k.ib - k.width - k.next;
  return k;
}
// mbar_wait for warps that wait most of the time beside one that must not be disturbed: the thread is suspended until the
// phase completes or the time given with the instruction has passed, instead of polling at the pace of the default.
__device__ __forceinline__ bool mbar_wait_asleep(uint64_t* bar, uint32_t parity) {
  auto done = [&]() {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r) : "r"(umma::smem_u32(bar)), "r"(parity), "r"(20000u) : "memory");
    return r != 0;
  };
  if (done()) return true;
  const uint64_t t0 = umma::global_timer_ns(), limit = umma::g_wait_limit_ns;
  while (!done())
    if (umma::global_timer_ns() - t0 > limit) return false;
  return true;
}
// A wait of one role; after the first one that runs out the role stops waiting and leaves.
__device__ __forceinline__ bool stripe_wait(uint64_t* bar, int phase, bool& ok, int* dev_info, int code) {
  if (ok && !mbar_wait_asleep(bar, (uint32_t)phase & 1u)) {
    if ((threadIdx.x & 31) == 0) report_error(dev_info, GPTQ_ERR_TIMEOUT, code);
    ok = false;
  }
  return ok;
}

// The last thing an issuing thread does, however it got there: it waits for what it has in flight, so that shared and tensor memory
// are not given up under a load or an instruction that still uses them -- its MMAs and their commits by one more commit, and the
// last loads into its ring.  These end by themselves, so the limit is a fixed one, not the adjustable one of the roles' waits.
__device__ __forceinline__ void stripe_settle(uint64_t* settled, uint64_t* ring_full, int stages, int loaded, int* dev_info, int code) {
  auto wait = [&](uint64_t* b, uint32_t parity) {
    const uint64_t t0 = umma::global_timer_ns();
    while (!umma::mbar_try_wait(b, parity))
      if (umma::global_timer_ns() - t0 > 1000000000ull) { report_error(dev_info, GPTQ_ERR_TIMEOUT, code); return; }
  };
  umma::mma_commit(settled);
  wait(settled, 0u);
  for (int m = loaded > stages ? loaded - stages : 0; m < loaded; ++m) wait(&ring_full[m % stages], (uint32_t)(m / stages) & 1u);
}

// Warp 6: the 16 x 16 diagonal blocks of U as doubles, 1 / U_jj, sK and 1 / sC, one sub-block ahead of the row warps.
__device__ __forceinline__ void stripe_stage_cols(const StripeArgs& a, StripeCols* cols, StripeBars& bar, int lane) {
  const int n_sub = a.nb2 / kStripeSB;
  const int r0 = lane >> 2, q = lane & 3;
  float4 u[2];
  float sk = 0.f, sc = 0.f;
  auto fetch = [&](int n) {
    const int i = a.i2 + n * kStripeSB;
#pragma unroll
    for (int h = 0; h < 2; ++h) u[h] = *reinterpret_cast<const float4*>(a.U + (int64_t)(i + r0 + 8 * h) * a.C + i + 4 * q);
    if (lane < 16) { sk = a.sK[i + lane]; sc = a.sCinv[i + lane]; }
  };
  fetch(0);
  bool ok = true;
  for (int n = 0; n < n_sub; ++n) {
    if (!__all_sync(0xffffffffu, stripe_wait(&bar.cols_empty[n & 1], (n >> 1) ^ 1, ok, a.dev_info, 38))) return;   // (they shuffle below)
    StripeCols& c = cols[n & 1];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = r0 + 8 * h;
      const float uu[4] = {u[h].x, u[h].y, u[h].z, u[h].w};
      // 1 / U_rr, from the lane of the four that share row r and have column r
      const float dd = r % 4 == 0 ? uu[0] : r % 4 == 1 ? uu[1] : r % 4 == 2 ? uu[2] : uu[3];
      const double rd = 1.0 / (double)__shfl_sync(0xffffffffu, dd, (lane & ~3) + (r >> 2));
      if (q == (r >> 2)) c.rdiag[r] = rd;
#pragma unroll
      for (int e = 0; e < 4; ++e) c.U[r][4 * q + e] = (double)uu[e] * rd;
    }
    if (lane < 16) { c.sks[lane] = sk; c.sci[lane] = sc; }
    __syncwarp();
    if (lane == 0) umma::mbar_arrive(&bar.cols_full[n & 1]);
    if (n + 1 < n_sub) fetch(n + 1);
  }
}

// Warp 4, one lane: after every 16 columns, their errors onto the rest of the block and onto the next block.  loaded: slices asked for.
__device__ __forceinline__ void stripe_push_near(const StripeMaps& maps, const StripeArgs& a, uint8_t* etiles, uint8_t* slices,
                                                 StripeBars& bar, uint32_t tmem, int& loaded) {
  using namespace umma;
  bool ok = true;
  auto load = [&](int b, int s, int n) -> bool {
    const StripeBlock k = stripe_block(a, b);
    const int j0 = s * kStripeSB, boxes = (k.width - j0 - kStripeSB + k.next + 31) / 32;
    if (!stripe_wait(&bar.slice_empty[n & 1], (n >> 1) ^ 1, ok, a.dev_info, 31)) return false;
    uint8_t* dst = slices + (n & 1) * 2 * kStripeSlice;
    loaded = n + 1;
    mbar_arrive_expect_tx(&bar.slice_full[n & 1], (uint32_t)boxes * 2048);
    for (int q = 0; q < boxes; ++q) {
      tma_load_2d(dst + 1024 * q, &maps.s_hi, a.i2 + k.ib + j0, k.ib + j0 + kStripeSB + 32 * q, &bar.slice_full[n & 1]);
      tma_load_2d(dst + kStripeSlice + 1024 * q, &maps.s_lo, a.i2 + k.ib + j0, k.ib + j0 + kStripeSB + 32 * q, &bar.slice_full[n & 1]);
    }
    return true;
  };
  int n = 0;
  if (a.nb2 > kStripeSB && !load(0, 0, 0)) return;
  for (int b = 0; b * a.B < a.nb2; ++b) {
    const StripeBlock k = stripe_block(a, b);
    const int subs = k.width / kStripeSB;
    for (int s = 0; s < subs; ++s, ++n) {
      const int rem = k.width - (s + 1) * kStripeSB;
      if (rem + k.next == 0) return;                     // the last sixteen columns of the outer block
      const bool last = s + 1 == subs;
      {                                                    // the next sub-block's slice, if it has anything to push onto
        const StripeBlock kn = last ? stripe_block(a, b + 1) : k;
        const int sn = last ? 0 : s + 1;
        if (kn.width - (sn + 1) * kStripeSB + kn.next > 0 && !load(last ? b + 1 : b, sn, n + 1)) return;
      }
      if (!stripe_wait(&bar.slice_full[n & 1], n >> 1, ok, a.dev_info, 33) || !stripe_wait(&bar.errors, n, ok, a.dev_info, 34)) return;
      fence_after_thread_sync();
      const uint32_t ea = smem_u32(etiles + (b & 1) * kStripeETile) + (uint32_t)(s >> 2) * 16384 + (uint32_t)(s & 3) * 32;
      const uint32_t sl = smem_u32(slices + (n & 1) * 2 * kStripeSlice);
      const uint64_t ah = make_desc_sw128(ea, 0, 1024), al = make_desc_sw128(ea + 32768, 0, 1024);
      auto push = [&](uint32_t col, int first, int width) { // onto `width` columns, `first` of the slice on
        const uint32_t bh = sl + (uint32_t)first * 32;
        mma_pairs(tmem + col, ah, al, make_desc_sw32(bh), make_desc_sw32(bh + kStripeSlice),
                  make_idesc(kFmtF16, false, false, 128, width), s == 0);
      };
      if (rem > 0) {                                       // the next sixteen columns first: the row threads wait for them
        push(kTmemRest + (uint32_t)(s + 1) * kStripeSB, 0, kStripeSB);
        mma_commit(&bar.near_done);
        if (rem > kStripeSB) push(kTmemRest + (uint32_t)(s + 2) * kStripeSB, kStripeSB, rem - kStripeSB);
      }
      if (k.next > 0) push(kTmemNext + (uint32_t)((b + 1) & 1) * 128, rem, k.next);
      if (rem == 0) mma_commit(&bar.near_done);
      mma_commit(&bar.rest_done);
      mma_commit(&bar.slice_empty[n & 1]);
    }
  }
}

// Warp 5, one lane: a block's errors onto the columns after the next block.  loaded: K atoms asked for.
__device__ __forceinline__ void stripe_push_far(const StripeMaps& maps, const StripeArgs& a, uint8_t* etiles, uint8_t* stages,
                                                StripeBars& bar, uint32_t tmem, int& loaded) {
  using namespace umma;
  bool ok = true;
  const int n_atoms = (a.B + 63) >> 6;                    // 64-wide K atoms in a block
  constexpr uint32_t idesc = make_idesc(kFmtF16, false, false, 128, kStripeNT);
  int f = 0, h = 0;                                       // tiles and staged K atoms so far
  for (int b = 0; b * a.B < a.nb2; ++b) {
    const StripeBlock k = stripe_block(a, b);
    const int n_tiles = (k.far + kStripeNT - 1) / kStripeNT, col0 = k.ib + k.width + k.next, total = n_tiles * n_atoms;
    auto load = [&](int u, int hh) -> bool {              // K atom u % n_atoms of tile u / n_atoms (columns beyond the block: zeros)
      const int st = hh % kStripeStages, x = a.i2 + k.ib + 64 * (u % n_atoms), y = col0 + u / n_atoms * kStripeNT;
      if (!stripe_wait(&bar.stage_empty[st], (hh / kStripeStages) ^ 1, ok, a.dev_info, 32)) return false;
      uint8_t* sp = stages + st * kStripeStage;
      loaded = hh + 1;
      mbar_arrive_expect_tx(&bar.stage_full[st], (uint32_t)kStripeStage);
      tma_load_2d(sp, &maps.p_hi, x, y, &bar.stage_full[st]);
      tma_load_2d(sp + 8192, &maps.p_lo, x, y, &bar.stage_full[st]);
      return true;
    };
    int ahead = 0;
    for (; ahead < min(2, total); ++ahead) if (!load(ahead, h + ahead)) return;
    if (!stripe_wait(&bar.block_errors[b & 1], b >> 1, ok, a.dev_info, 35)) return;
    fence_after_thread_sync();
    const uint32_t ea = smem_u32(etiles + (b & 1) * kStripeETile);
    for (int tl = 0; tl < n_tiles; ++tl, ++f) {
      if (!stripe_wait(&bar.acc_empty[f & 1], (f >> 1) ^ 1, ok, a.dev_info, 40)) return;
      for (int at = 0; at < n_atoms; ++at, ++h) {
        if (ahead < total) { if (!load(ahead, h + 2)) return; ++ahead; }
        const int st = h % kStripeStages;
        if (!stripe_wait(&bar.stage_full[st], h / kStripeStages, ok, a.dev_info, 39)) return;
        fence_after_thread_sync();
        const uint32_t sb = smem_u32(stages + st * kStripeStage), ta = ea + (uint32_t)at * 16384;
        for (int ks = 0; ks < min(4, a.B / 16 - 4 * at); ++ks)
          mma_pairs(tmem + kTmemFar + (uint32_t)(f & 1) * kStripeNT, make_desc_sw128(ta + 32 * ks, 0, 1024),
                    make_desc_sw128(ta + 32768 + 32 * ks, 0, 1024), make_desc_sw128(sb + 32 * ks, 0, 1024),
                    make_desc_sw128(sb + 8192 + 32 * ks, 0, 1024), idesc, at == 0 && ks == 0);
        mma_commit(&bar.stage_empty[st]);
      }
      mma_commit(&bar.acc_full[f & 1]);
    }
    mma_commit(&bar.tile_free[b & 1]);
  }
}

// Warps 8-11: the far sums, scaled back, onto the working weights in memory: -sum / (sE[row] sC[column]).  A column of the
// warp's 32 rows is 256 consecutive bytes: one reduction instruction, no value comes back.
__device__ __forceinline__ void stripe_drain_far(const StripeArgs& a, StripeBars& bar, uint32_t tmem, int quarter, int lane) {
  using namespace umma;
  bool ok = true;
  const int row = blockIdx.x * kStripeRows + 32 * quarter + lane;
  const double inv_se = row < a.R ? (double)a.sEinv[row] : 0.0;
  double* out = a.Wblk + (int64_t)blockIdx.x * a.ldw * kStripeRows + 32 * quarter + lane;
  int f = 0;
  auto performed = [&](uint64_t* b) {                     // everything issued so far has been added in memory
    __threadfence();
    __syncwarp();
    if (lane == 0) mbar_arrive(b);
  };
  for (int b = 0; ok; ++b) {
    const StripeBlock k = stripe_block(a, b);
    if (k.far <= 0) break;                                // (the last two blocks push nothing this far, and nobody waits for them)
    const int n_tiles = (k.far + kStripeNT - 1) / kStripeNT, col0 = k.ib + k.width + k.next;
    const int near_tiles = (min(k.far, a.B) + kStripeNT - 1) / kStripeNT;   // onto the block after next, which needs them first
    for (int tl = 0; tl < n_tiles; ++tl, ++f) {
      const int col = col0 + tl * kStripeNT, halves = min(2, (a.nb2 - col) / 32);
      float sc[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) sc[q] = q < halves ? a.sCinv[a.i2 + col + 32 * q + lane] : 0.f;
      if (!stripe_wait(&bar.acc_full[f & 1], f >> 1, ok, a.dev_info, 41)) break;
      fence_after_thread_sync();
      float v[2][32];
#pragma unroll
      for (int q = 0; q < 2; ++q)
        tmem_ld_32x32(tmem + ((uint32_t)(32 * quarter) << 16) + kTmemFar + (uint32_t)(f & 1) * kStripeNT + 32 * q, v[q]);
      tmem_ld_wait();
      fence_before_thread_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar.acc_empty[f & 1]);
      double* d = out + (int64_t)col * kStripeRows;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (q < halves) {
#pragma unroll
          for (int u = 0; u < 32; ++u)
            asm volatile("red.relaxed.gpu.global.add.f64 [%0], %1;" ::"l"(d + (int64_t)(32 * q + u) * kStripeRows),
                         "d"(-(double)(v[q][u] * __shfl_sync(0xffffffffu, sc[q], u)) * inv_se) : "memory");
        }
      }
      if (tl + 1 == near_tiles) performed(&bar.next_ready[b & 1]);
    }
    if (!ok) break;
    performed(&bar.all_ready[b & 1]);
  }
}

// kGroups: kSmall groups of 4, 8 or 16 columns (their grids are taken inside the column loop; the tests for that cost every
// other grid 14 cycles a column), kNarrow groups of 32 to 127 (see stripe_scan_rest), kWide the rest and per-row grids.
enum StripeGroupWidth { kWide, kSmall, kNarrow };
template <int kGroups>
__global__ void __launch_bounds__(kStripeThreads, 1)
stripe_kernel(const __grid_constant__ StripeMaps maps, const StripeArgs a) {
  using namespace umma;
  constexpr bool kSmallGroups = kGroups == kSmall;
  extern __shared__ uint8_t smem_raw[];
  // An offset onto the array, not a rounded address: that would lose the address space, and every read of U in the column loop would
  // be a generic load (4096 rows x 1024 columns, 4-bit: 226 us with those, 198 with shared loads; groups of 128: 287, 249).
  uint8_t* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  StripeCols* cols = reinterpret_cast<StripeCols*>(base + kStripeOffCols);
  StripeBars& bar = *reinterpret_cast<StripeBars*>(base + kStripeOffBars);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;

  if (t == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bar.cols_full[s], 1); mbar_init(&bar.cols_empty[s], 4);
      mbar_init(&bar.slice_full[s], 1); mbar_init(&bar.slice_empty[s], 1);
      mbar_init(&bar.block_errors[s], 4); mbar_init(&bar.tile_free[s], 1);
      mbar_init(&bar.acc_full[s], 1); mbar_init(&bar.acc_empty[s], 4);
      mbar_init(&bar.next_ready[s], 4); mbar_init(&bar.all_ready[s], 4);
    }
    for (int s = 0; s < kStripeStages; ++s) { mbar_init(&bar.stage_full[s], 1); mbar_init(&bar.stage_empty[s], 1); }
    mbar_init(&bar.errors, 4); mbar_init(&bar.near_done, 1); mbar_init(&bar.rest_done, 1);
    mbar_init(&bar.settled[0], 1); mbar_init(&bar.settled[1], 1);
    fence_barrier_init();
    fence_proxy_async();
    prefetch_tmap(&maps.p_hi); prefetch_tmap(&maps.p_lo); prefetch_tmap(&maps.s_hi); prefetch_tmap(&maps.s_lo);
  }
  if (warp == 4) { tmem_alloc(&bar.tmem, 512); tmem_relinquish(); }
  fence_before_thread_sync();
  pdl_wait();                                             // (nothing above reads or writes what another kernel does)
  __syncthreads();
  fence_after_thread_sync();
  const uint32_t tmem = bar.tmem;

  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 136;");
    stripe_drain_far(a, bar, tmem, warp & 3, lane);
  } else if (warp >= 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 112;");
    int loaded = 0;
    if (warp == 4 && lane == 0) {
      stripe_push_near(maps, a, base, base + kStripeOffSlice, bar, tmem, loaded);
      stripe_settle(&bar.settled[0], bar.slice_full, 2, loaded, a.dev_info, 46);
    } else if (warp == 5 && lane == 0) {
      stripe_push_far(maps, a, base, base + kStripeOffFar, bar, tmem, loaded);
      stripe_settle(&bar.settled[1], bar.stage_full, kStripeStages, loaded, a.dev_info, 47);
    } else if (warp == 6) {
      stripe_stage_cols(a, cols, bar, lane);
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 248;");
    // ---------------------------------------------------------------- the rows, one thread each
    const int row = blockIdx.x * kStripeRows + t;
    const bool live = row < a.R;
    const int G = a.G, g = a.group;
    const uint32_t tmem_lane = tmem + ((uint32_t)(warp * 32) << 16);
    const double* wg = a.Wblk + (int64_t)blockIdx.x * a.ldw * kStripeRows + t;
    const float se_row = live ? a.sE[row] : 1.f;
    const double inv_se = live ? (double)a.sEinv[row] : 0.0;
    RowGrid grid;
    grid.set(live && g <= 0 ? make_float2(a.scales[row], a.zeros[row]) : make_float2(1.f, 0.f));
    double loss = 0.0;
    bool bad = false, ok = true;
    // columns of a 16-column sub-block at which a small group (4, 8 or 16 columns) starts
    const uint32_t small_group_starts = g == 4 ? 0x1111u : (g == 8 ? 0x0101u : (g == 16 ? 0x0001u : 0u));
    double ahead[kStripeSB];                              // the next sixteen columns, on their way
    stripe_fetch(wg, live, ahead);
    int n = 0;                                            // sub-blocks so far
#pragma unroll 1
    for (int b = 0; b * a.B < a.nb2; ++b) {
      const StripeBlock k = stripe_block(a, b);
      const int i = a.i2 + k.ib;                          // first global column of the block
      uint8_t* etile = base + (b & 1) * kStripeETile;
      const uint32_t tm_next = tmem_lane + kTmemNext + (uint32_t)(b & 1) * 128, tm_rest = tmem_lane + kTmemRest;
#pragma unroll 1
      for (int j0 = 0; j0 < k.width; j0 += kStripeSB, ++n) {
        const StripeCols& cs = cols[n & 1];
        if (t == 0 && k.ib + j0 + kStripeSB >= a.nb2) pdl_next();                 // the last sixteen columns
        auto at = [&]() {
          return StripeAt{wg + (int64_t)(k.ib + j0) * kStripeRows, a.sCinv + i + j0, tm_next + j0, tm_rest + j0, b > 0, j0 > 0, live, inv_se};
        };
        stripe_wait(&bar.cols_full[n & 1], n >> 1, ok, a.dev_info, 36);
        if (n > 0) stripe_wait(&bar.near_done, n - 1, ok, a.dev_info, 37);
        fence_after_thread_sync();
        const bool starts = !kSmallGroups && g >= 32 && ((i + j0) % g) == 0;     // a group starts (wider than the block: only at j0 = 0)
        auto set_grid = [&](float2 sz) {
          grid.set(sz);
          if (live) { a.scales[(int64_t)row * G + (i + j0) / g] = sz.x; a.zeros[(int64_t)row * G + (i + j0) / g] = sz.y; }
        };
        if (starts) {
          if (g > a.B) {
            const int q = min(b - 1, (a.nb2 + a.B - 1) / a.B - 3);        // the last block before this one with far pushes
            if (q >= 0) stripe_wait(&bar.all_ready[q & 1], q >> 1, ok, a.dev_info, 42);
          } else if (j0 > 0) {
            stripe_wait(&bar.rest_done, n - 1, ok, a.dev_info, 43);
            fence_after_thread_sync();
          }
          if (kGroups != kNarrow) set_grid(stripe_scan(at(), g, k.width - j0, a.grid));
        }
        double w[kStripeSB];
#pragma unroll
        for (int m = 0; m < kStripeSB; ++m) w[m] = ahead[m];
        if (b > 0 && j0 > 0) {                             // (both on their way before the wait)
          float v[kStripeSB], u[kStripeSB];
          tmem_ld_32x16(tm_next + j0, v); tmem_ld_32x16(tm_rest + j0, u);
          umma::tmem_ld_wait();
#pragma unroll
          for (int m = 0; m < kStripeSB; ++m) w[m] = (w[m] - (double)(v[m] * cs.sci[m]) * inv_se) - (double)(u[m] * cs.sci[m]) * inv_se;
        } else if (b > 0 || j0 > 0) {
          stripe_subtract(b > 0 ? tm_next + j0 : tm_rest + j0, cs.sci, inv_se, w);
        }
        // the next sixteen columns' loads go out now
        {
          const int col = k.ib + j0 + kStripeSB;
          if (j0 + kStripeSB == k.width && b >= 1 && col < a.nb2) stripe_wait(&bar.next_ready[(b - 1) & 1], (b - 1) >> 1, ok, a.dev_info, 44);
          if (col < a.nb2) stripe_fetch(wg + (int64_t)col * kStripeRows, live, ahead);
        }
        if (kGroups == kNarrow && starts) {
          double mn = w[0], mx = w[0];
#pragma unroll
          for (int m = 1; m < kStripeSB; ++m) { mn = w[m] < mn ? w[m] : mn; mx = w[m] > mx ? w[m] : mx; }
          set_grid(stripe_scan_rest(at(), g, k.width - j0, a.grid, mn, mx));
        }
        StripeGroups sg{g, small_group_starts, a.grid, a.scales + (int64_t)row * G + (i + j0) / (g > 0 ? g : 1),
                        a.zeros + (int64_t)row * G + (i + j0) / (g > 0 ? g : 1), live};
        // The sixteen columns.  What bounds them is the chain from one column's weight to the next column's, so it is kept to
        // three fp64 operations and two integer ones, and the instructions beside it are counted too.  The quotient
        // w / scale + 1/2 is formed with the reciprocal, added to 2^32 + 2048: the low word then holds it in units of 2^-20,
        // its upper twelve bits the code (rounded, counted from zero-point - 2048), to be clamped as an integer.  With U's row
        // divided by U_jj (n) the next column's weight is (w' - w n) + (scale n) (code - zero-point): everything but the last
        // multiply-add is ready when the code is.  (w n is formed before it cancels: the next weight's rounding error is 2^-53 of |w n|, not of
        // |w - q| n: 2^-29 of the fp32-level sums that weight has met.)  The other columns take (w - scale (code - zero-point)) n, exact in its one
        // multiply-add (24-bit scale).  Where the quotient lies within 2^-20 of a tie (the fraction bits are next to zero) or
        // outside twelve bits (the upper word is another one), the sixteen columns are done again with the division itself.
        // (rint, fmin and fmax take 20 to 25 cycles each in fp64.)  The errors' way into the tile fills the chain's gaps, pair by
        // pair.  4096 rows x 1024 columns, 4-bit: 195 us with the error's five operations on the chain; 189 with it; 190 with the
        // tile written here instead of after the loop, 189 with both sums of the sub-block asked for at once; 184 with all three.
        constexpr double kQuot = 4294967296.0 + 2048.5;
        float err[kStripeSB];
        uint32_t cw[kStripeSB / 4];
        uint32_t frac = 0xFFFFFu;                          // smallest distance of the fraction bits above -1 seen
        int range = 0;
        double l0 = 0.0;
        uint32_t hw[kStripeSB / 2], lw[kStripeSB / 2];
        float big = 0.f;
        uint8_t* rowp = etile + (j0 >> 6) * 16384 + t * 128;
        // the tile was last read by the pushes of the block before the previous one
        if (j0 == 0 && b >= 2) stripe_wait(&bar.tile_free[b & 1], (b >> 1) - 1, ok, a.dev_info, 45);
        // scaled errors u and u + 1 as fp16 hi / lo pairs, and with the eighth and the sixteenth column eight of them into the swizzled
        // K-major tile (row t, 16-byte chunk (k / 8) ^ (t & 7) of the 128-byte row of K atom k / 64)
        auto put = [&](int u) {
          const float x0 = err[u] * cs.sks[u] * se_row, x1 = err[u + 1] * cs.sks[u + 1] * se_row;
          big = fmaxf(big, fmaxf(fabsf(x0), fabsf(x1)));
          stripe_split2(x0, x1, hw[u >> 1], lw[u >> 1]);
          if ((u & 7) != 6) return;
          uint8_t* d = rowp + (((((j0 & 63) + u) >> 3) ^ (t & 7)) << 4);
          *reinterpret_cast<uint4*>(d) = make_uint4(hw[u / 2 - 3], hw[u / 2 - 2], hw[u / 2 - 1], hw[u / 2]);
          *reinterpret_cast<uint4*>(d + 32768) = make_uint4(lw[u / 2 - 3], lw[u / 2 - 2], lw[u / 2 - 1], lw[u / 2]);
        };
#pragma unroll
        for (int jj = 0; jj < kStripeSB; ++jj) {
          if (kSmallGroups && (jj & 3) == 0 && ((small_group_starts >> jj) & 1u)) stripe_small_group(sg, jj, w, grid);
          const double t0 = fma(w[jj], grid.rscale, kQuot);
          const uint32_t q = (uint32_t)__double2loint(t0);
          const uint32_t c = (uint32_t)__viaddmin_s32_relu((int)(q >> 20), grid.bias, a.grid.maxq);
          const double cd = __hiloint2double(0x43300000, (int)c) - grid.kz;         // code - zero-point
          if (jj + 1 < kStripeSB) {
            const double nx = cs.U[jj][jj + 1];
            w[jj + 1] = fma(cd, grid.scale * nx, fma(-w[jj], nx, w[jj + 1]));
          }
          const double r = fma(-grid.scale, cd, w[jj]), e = r * cs.rdiag[jj];
#pragma unroll
          for (int m = 0; m < kStripeSB; ++m)             // immediate feedback onto the later columns in registers
            if (m > jj + 1) w[m] = fma(-r, cs.U[jj][m], w[m]);
          cw[jj >> 2] = (jj & 3) == 0 ? c : cw[jj >> 2] + (c << (8 * (jj & 3)));
          err[jj] = (float)e;
          l0 = fma(e, e, l0);
          if (jj & 1) put(jj - 1);
          frac = min(frac, (q + 1u) & 0xFFFFFu);
          range |= __double2hiint(t0) ^ 0x41F00000;
        }
        if (__any_sync(0xffffffffu, frac <= 2u || range != 0)) {
          StripeRedo r;
          stripe_redo<kSmallGroups>(at(), cs, grid, sg, r);
#pragma unroll
          for (int m = 0; m < kStripeSB; ++m) err[m] = r.err[m];
#pragma unroll
          for (int m = 0; m < kStripeSB / 4; ++m) cw[m] = r.cw[m];
          l0 = r.loss;
          big = 0.f;
#pragma unroll
          for (int m = 0; m < kStripeSB; m += 2) put(m);
        }
        if (live) { bad |= big > 65504.f || !isfinite(l0); loss += l0; }
        fence_proxy_async();                              // the tile was written through the generic proxy
        fence_before_thread_sync();                       // this sub-block's tcgen05.ld are done
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&bar.errors);
          mbar_arrive(&bar.cols_empty[n & 1]);
          if (j0 + kStripeSB == k.width) mbar_arrive(&bar.block_errors[b & 1]);
        }
        if (live) {
          const int64_t o = (int64_t)row * a.C + i + j0;
          if (a.keep_errors) {
            uint4* gh = reinterpret_cast<uint4*>(a.Ehi + o);
            uint4* gl = reinterpret_cast<uint4*>(a.Elo + o);
            gh[0] = make_uint4(hw[0], hw[1], hw[2], hw[3]); gh[1] = make_uint4(hw[4], hw[5], hw[6], hw[7]);
            gl[0] = make_uint4(lw[0], lw[1], lw[2], lw[3]); gl[1] = make_uint4(lw[4], lw[5], lw[6], lw[7]);
          }
          *reinterpret_cast<uint4*>(a.codes + o) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
        }
      }
    }
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_down_sync(0xffffffffu, loss, o);
    if (lane == 0 && loss != 0.0) atomicAdd(a.loss, loss);
    if (bad) report_error(a.dev_info, GPTQ_ERR_NONFINITE, row);
  }
  fence_before_thread_sync();
  __syncthreads();
  if (warp == 4) { fence_after_thread_sync(); tmem_dealloc(tmem, 512); }
}
