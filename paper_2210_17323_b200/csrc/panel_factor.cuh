// Factor and invert one outer panel's diagonal block in ONE launch: A = T T^T with T upper triangular (a Cholesky
// factorisation run from the last row backwards) and V = T^-1, for a w x w block, w <= 1024 (included by hinv.cu).
//
// The block is cut into 64 x 64 tiles M[i][c].  Upper tiles (i <= c) start as A and end as T, strictly lower tiles start
// as zero and end as the TRANSPOSED inverse (tile (i, c), i > c, holds V[c][i]^T): with that convention both the trailing
// update of the factorisation and the forward substitution T V = I are the same statement.  Step k (last tile column
// first):
//   factor   M[k][k] = T_kk T_kk^T, V_kk = T_kk^-1                                (fp64, one CTA)
//   solve    M[i][k] <- M[i][k] V_kk^T                          for every i != k   (T_ik above, V_ki^T below the diagonal)
//   update   M[i][c] -= M[i][k] T_ck^T                          for c < k and (i <= c or i >= k)     (M[k][k] := V_kk^T)
// Two neighbouring tile columns (2 m, 2 m + 1) are factored and inverted in fp64 as one 128 x 128 block: what they exchange
// (V of column 2 m + 1, the tile between them, V of column 2 m) is kept in fp64 beside the matrix, and only finished entries of
// T and V are rounded to fp32.  (With fp32 products between them U was 2 to 6 times as far from 64 bits for 96 .. 128 columns.)
//
// What bounds it: the chain factor -> solve of the tile above -> update of the next diagonal tile -> factor.  Everything
// else (about 1600 tile products for w = 1024) has one step's time to finish.  So the first CTA to arrive runs that chain
// and nothing else, and the others take the remaining tile products from a list in step order.  Nothing here needs the
// CTAs to be resident together: a product waits only for products EARLIER in the list and for chain steps, and the
// chain, if what it waits for has not been taken by anybody, takes it itself (chain_wait).  Every wait is bounded.
// As separate launches (one 128-wide diagonal kernel of 97 us, two small GEMMs, two more on a side stream for the
// inverse, per 128 columns) a 1024-wide call took 1.29 ms; this form 0.254 ms (768 columns: 0.94 -> 0.195 ms), of which the
// fp64 products of the pairs are 0.006 ms and rsqrt() 0.009.  A chain step is about 15 us; on the chain's SM no pipe is more than
// half busy (shared memory 46 %, DMMA 16 %).
#pragma once

namespace gptq {
namespace {
namespace panel {

constexpr int TB = 64;               // tile edge
constexpr int kMaxTiles = 16;        // w <= 1024
constexpr int kThreads = 256;
constexpr int LDF = 68;              // fp32 tile pitch (floats): 16-byte rows, eight rows on distinct bank groups
constexpr int LDD = 68;              // fp64 tile pitch (doubles): four rows 32 bytes apart modulo 128, conflict-free fragments
// fp64 tiles of a pair of tile columns (k, k + 1), k even: the inverse of column k + 1's diagonal tile, the tile between them, the
// inverse of column k's.  An inverse is kept transposed, as the factorisation leaves it: entry (m, c) is V[c][m], c <= m.
constexpr int kPairV1 = 0, kPairT = 1, kPairV0 = 2, kPairTiles = 3;

// Progress of one launch, in the caller's workspace; all zero when the kernel starts.
struct Flags {
  int role;                          // order of arrival: 0 runs the chain
  int ticket;                        // next entry of the list of products
  int factored;                      // tile columns factored so far (from the last one)
  int abort;                         // a wait ran out: everybody leaves
  int solved[kMaxTiles * kMaxTiles]; // tile (i, k) has been through step k's solve
  int updated[kMaxTiles * kMaxTiles];// updates applied to tile (i, c)
  int paired[kMaxTiles / 2];         // the fp64 tiles of pair (2 m, 2 m + 1) are complete
};
// doubles of the pairs of a block of w columns
constexpr size_t pair_doubles(int w) { return (size_t)((w + TB - 1) / TB / 2) * kPairTiles * TB * TB; }

struct Args {
  float* A;                          // first element of the block inside the C x C matrix
  int64_t ld;
  int w, nt, k_global;               // width, tiles, global index of the block's first row (for reports)
  Flags* fl;
  double* pairs;                     // pair_doubles(w)
  int* dev_info;
};

struct Smem {
  union {
    struct { float As[TB][LDF]; float Bs[TB][LDF]; };
    double E[TB][LDD];
  };
  double D[TB][LDD];
  int msg[4];
};

// ---- waiting -------------------------------------------------------------------------------------
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// One thread: waits until *p >= v; false if the launch is being abandoned.
__device__ __forceinline__ bool wait_ge(const int* p, int v, const Args& a) {
  if (ld_acquire(p) >= v) return true;
  const uint64_t t0 = umma::global_timer_ns(), limit = umma::g_wait_limit_ns;
  for (uint32_t spins = 1;; ++spins) {
    if (ld_acquire(p) >= v) return true;
    if ((spins & 0x3F) == 0) {
      if (ld_acquire(&a.fl->abort)) return false;
      if (umma::global_timer_ns() - t0 > limit) {
        report_error(a.dev_info, GPTQ_ERR_TIMEOUT, 61);
        st_release(&a.fl->abort, 1);
        return false;
      }
    }
  }
}

// ---- the list of products ---------------------------------------------------------------------------
// Step k: the solves (rows k - 2 .. 0, then k + 1 .. nt - 1; row k - 1 belongs to the chain), then the updates column by
// column, c = k - 1 .. 0, rows c .. 0 and then k .. nt - 1 (tile (k - 1, k - 1) belongs to the chain): what the chain needs
// next comes first.
__host__ __device__ __forceinline__ int step_solves(int nt, int k) { return nt - 1 - (k > 0 ? 1 : 0); }
__host__ __device__ __forceinline__ int step_updates(int nt, int k) { return k * (k + 1) / 2 + k * (nt - k) - (k > 0 ? 1 : 0); }
struct Task { int kind, i, c, k; };  // kind 0: solve tile (i, k); 1: update tile (i, c) with step k; -1: nothing left
__host__ __device__ inline Task task_of(int nt, int t) {
  for (int k = nt - 1; k >= 0; --k) {
    const int ns = step_solves(nt, k), nu = step_updates(nt, k);
    if (t < ns) {
      const int above = k > 1 ? k - 1 : 0;
      return Task{0, t < above ? k - 2 - t : k + 1 + (t - above), k, k};
    }
    t -= ns;
    if (t < nu) {
      for (int c = k - 1; c >= 0; --c) {
        const int skip = c == k - 1 ? 1 : 0, above = c + 1 - skip, n = above + nt - k;
        if (t < n) return Task{1, t < above ? c - skip - t : k + (t - above), c, k};
        t -= n;
      }
    }
    t -= nu;
  }
  return Task{-1, 0, 0, 0};
}
// entries of the list that belong to steps > k: all of them can run once the chain has passed step k + 1
__host__ __device__ inline int tasks_before_step(int nt, int k) {
  int n = 0;
  for (int q = nt - 1; q > k; --q) n += step_solves(nt, q) + step_updates(nt, q);
  return n;
}
// updates that tile (i, c) has seen before step k
__host__ __device__ __forceinline__ int updates_before(int nt, int i, int c, int k) { return i <= c ? nt - 1 - k : i - k; }

// ---- tile products (fp32) ------------------------------------------------------------------------------
// acc[p][q] = sum_m As[ty + 16 p][m] * Bs[tx + 16 q][m]; kUpper: only the 16 x 16 pieces on or above the diagonal (p <= q)
template <bool kUpper = false>
__device__ __forceinline__ void product(const float (*As)[LDF], const float (*Bs)[LDF], float (&acc)[4][4], int tx, int ty) {
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[p][q] = 0.f;
#pragma unroll 4
  for (int m = 0; m < TB; m += 4) {
    float4 x[4], y[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) x[p] = *reinterpret_cast<const float4*>(&As[ty + 16 * p][m]);
#pragma unroll
    for (int q = 0; q < 4; ++q) y[q] = *reinterpret_cast<const float4*>(&Bs[tx + 16 * q][m]);
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = kUpper ? p : 0; q < 4; ++q) {
        acc[p][q] = fmaf(x[p].x, y[q].x, acc[p][q]); acc[p][q] = fmaf(x[p].y, y[q].y, acc[p][q]);
        acc[p][q] = fmaf(x[p].z, y[q].z, acc[p][q]); acc[p][q] = fmaf(x[p].w, y[q].w, acc[p][q]);
      }
  }
}
// Tile (i, c) of the block into shared memory, zeros beyond the block.  The tiles were written by other CTAs of this
// launch: loads bypass L1.
__device__ __forceinline__ void load_tile(const Args& a, int i, int c, float (*S)[LDF], int t) {
  const int q = t & 15, r0 = t >> 4;
  float4 v[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int r = TB * i + r0 + 16 * p, col = TB * c + 4 * q;
    v[p] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < a.w && col < a.w) v[p] = __ldcg(reinterpret_cast<const float4*>(a.A + (int64_t)r * a.ld + col));
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) *reinterpret_cast<float4*>(&S[r0 + 16 * p][4 * q]) = v[p];
}
__device__ __forceinline__ void load_tile_t(const Args& a, int i, int c, float (*S)[LDF], int t) {   // S = tile^T
  const int q = t & 15, r0 = t >> 4;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int r = TB * i + r0 + 16 * p, col = TB * c + 4 * q;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < a.w && col < a.w) v = __ldcg(reinterpret_cast<const float4*>(a.A + (int64_t)r * a.ld + col));
    S[4 * q][r0 + 16 * p] = v.x; S[4 * q + 1][r0 + 16 * p] = v.y; S[4 * q + 2][r0 + 16 * p] = v.z; S[4 * q + 3][r0 + 16 * p] = v.w;
  }
}

// ---- fp64 tiles of a pair -------------------------------------------------------------------------------
// c += a (8 x 4, row) * b (4 x 8, col): lane holds a[lane / 4][lane % 4], b[lane % 4][lane / 4], c[lane / 4][2 (lane % 4) + {0, 1}]
__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
               : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}
__device__ __forceinline__ double* pair_tile(const Args& a, int k, int which) { return a.pairs + ((size_t)(k >> 1) * kPairTiles + which) * (TB * TB); }
__device__ __forceinline__ void load_pair_tile(const double* src, double (*S)[LDD], int t) {
  double2 v[8];
#pragma unroll
  for (int p = 0; p < 8; ++p) v[p] = __ldcg(reinterpret_cast<const double2*>(src) + t + kThreads * p);
#pragma unroll
  for (int p = 0; p < 8; ++p) { const int e = t + kThreads * p; *reinterpret_cast<double2*>(&S[e >> 5][2 * (e & 31)]) = v[p]; }
}
__device__ __forceinline__ void store_pair_tile(double* dst, const double (*S)[LDD], int t) {
#pragma unroll
  for (int p = 0; p < 8; ++p) { const int e = t + kThreads * p; reinterpret_cast<double2*>(dst)[e] = *reinterpret_cast<const double2*>(&S[e >> 5][2 * (e & 31)]); }
}
// A pair's tile of the inverse, all threads: V[k][k + 1] = -V_kk T[k][k + 1] V_{k+1,k+1}, transposed into tile (k + 1, k).  Warp
// `rt` makes the eight rows 8 rt .. of each product; entries on the wrong side of a triangle are skipped or read as zero.
__device__ __forceinline__ bool pair_inverse(const Args& a, Smem& s, int k, int t) {
  const int rt = t >> 5, r = (t & 31) >> 2, q = t & 3;
  if (t == 0) s.msg[3] = wait_ge(&a.fl->paired[k >> 1], 1, a) ? 1 : 0;
  __syncthreads();                                      // (also: the previous product is done with the tiles)
  if (!s.msg[3]) return false;
  load_pair_tile(pair_tile(a, k, kPairT), s.E, t);
  load_pair_tile(pair_tile(a, k, kPairV1), s.D, t);
  __syncthreads();
  double y[8][2];
#pragma unroll
  for (int ct = 0; ct < 8; ++ct) y[ct][0] = y[ct][1] = 0.0;
#pragma unroll
  for (int kc = 0; kc < 16; ++kc) {
    const double x = s.E[8 * rt + r][4 * kc + q];
#pragma unroll
    for (int ct = kc / 2; ct < 8; ++ct) {
      const double v = s.D[8 * ct + r][4 * kc + q];
      dmma(y[ct], x, 4 * kc + q <= 8 * ct + r ? v : 0.0);
    }
  }
  __syncthreads();
#pragma unroll
  for (int ct = 0; ct < 8; ++ct) *reinterpret_cast<double2*>(&s.E[8 * rt + r][8 * ct + 2 * q]) = make_double2(y[ct][0], y[ct][1]);
  load_pair_tile(pair_tile(a, k, kPairV0), s.D, t);
  __syncthreads();
#pragma unroll
  for (int ct = 0; ct < 8; ++ct) y[ct][0] = y[ct][1] = 0.0;
#pragma unroll 2
  for (int kc = 2 * rt; kc < 16; ++kc) {
    const double v = s.D[4 * kc + q][8 * rt + r], x = 4 * kc + q >= 8 * rt + r ? v : 0.0;
#pragma unroll
    for (int ct = 0; ct < 8; ++ct) dmma(y[ct], x, s.E[4 * kc + q][8 * ct + r]);
  }
  float* out = a.A + (int64_t)(TB * (k + 1)) * a.ld + TB * k + 8 * rt + r;
#pragma unroll
  for (int ct = 0; ct < 8; ++ct)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int c = 8 * ct + 2 * q + e;
      if (TB * (k + 1) + c < a.w) out[(int64_t)c * a.ld] = (float)-y[ct][e];
    }
  __syncthreads();
  if (t == 0) st_release(&a.fl->solved[(k + 1) * kMaxTiles + k], 1);
  return true;
}

// One product of the list, all threads of the CTA.  False if the launch is being abandoned.
__device__ __forceinline__ bool run_task(const Args& a, Smem& s, const Task& k, int t) {
  const int nt = a.nt, tx = t & 15, ty = t >> 4;
  Flags* fl = a.fl;
  if (k.c + 1 == k.k && (k.k & 1) && k.i == k.k) return true;                     // part of pair_inverse
  if (k.kind == 0 && k.i == k.k + 1 && !(k.k & 1)) return pair_inverse(a, s, k.k, t);
  if (t == 0) {
    bool ok;
    if (k.kind == 0) {
      ok = wait_ge(&fl->updated[k.i * kMaxTiles + k.k], updates_before(nt, k.i, k.k, k.k), a) && wait_ge(&fl->factored, nt - k.k, a);
    } else {
      ok = wait_ge(&fl->updated[k.i * kMaxTiles + k.c], updates_before(nt, k.i, k.c, k.k), a) &&
           (k.i == k.k ? wait_ge(&fl->factored, nt - k.k, a) : wait_ge(&fl->solved[k.i * kMaxTiles + k.k], 1, a)) &&
           wait_ge(&fl->solved[k.c * kMaxTiles + k.k], 1, a);
    }
    s.msg[3] = ok ? 1 : 0;
  }
  __syncthreads();                                      // (also: the previous product is done with As and Bs)
  if (!s.msg[3]) return false;
  float* out = a.A + (int64_t)(TB * k.i + ty) * a.ld + TB * k.c + tx;
  float old[4][4];
  const bool first = k.kind == 1 && k.i == k.k;         // a lower tile's first update: it starts as zero
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      old[p][q] = 0.f;
      if (k.kind == 1 && !first && TB * k.i + ty + 16 * p < a.w && TB * k.c + tx + 16 * q < a.w)
        old[p][q] = __ldcg(out + (int64_t)(16 * p) * a.ld + 16 * q);
    }
  if (k.kind == 0) {
    load_tile(a, k.i, k.k, s.As, t);
    load_tile(a, k.k, k.k, s.Bs, t);
  } else {
    if (k.i == k.k) load_tile_t(a, k.k, k.k, s.As, t); else load_tile(a, k.i, k.k, s.As, t);
    load_tile(a, k.c, k.k, s.Bs, t);
  }
  __syncthreads();
  float acc[4][4];
  product(s.As, s.Bs, acc, tx, ty);
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (TB * k.i + ty + 16 * p < a.w && TB * k.c + tx + 16 * q < a.w)
        out[(int64_t)(16 * p) * a.ld + 16 * q] = k.kind == 0 ? acc[p][q] : old[p][q] - acc[p][q];
  __syncthreads();
  if (t == 0) {                                         // (the release covers what the barrier has collected from all threads)
    if (k.kind == 0) st_release(&fl->solved[k.i * kMaxTiles + k.k], 1);
    else st_release(&fl->updated[k.i * kMaxTiles + k.c], updates_before(nt, k.i, k.c, k.k) + 1);
  }
  return true;
}

// ---- factor + inverse of one 64 x 64 tile (fp64) ----------------------------------------------------------
// Columns 8 jb .. 8 jb + 7 of the sweep over the 64 rows of D, by two warps: lane l of warp h holds row 32 h + l.  Column j,
// last to first: x[i] = D[i][j] / sqrt(pivot) is T[i][j] for i < j and, because a row restarts from zero when its own column
// comes, V[j][i] for i >= j; then D[i][c] -= x[i] x[c] for the earlier columns c of the eight.
// Every lane carries the 8 x 8 diagonal block beside its own row and factors it redundantly: pivots and multipliers are in
// registers everywhere, and the chain per column is a reciprocal root, a multiplication and a multiply-add (85 cycles).
// (With the block's rows in eight lanes and two shuffles per multiplier and pivot a column took 240 cycles, half of the whole
// kernel's chain.  A real loop over eight columns at a time: one warp running 32 columns unrolled, 32 KB of straight code,
// was bound by instruction fetch and took twice as long again.)
__device__ __forceinline__ void sweep8(double (*D)[LDD], int jb, int row, int k_global, int* dev_info) {
  double g[8][8], a[8];                                  // g[i][c], i <= c: the diagonal block
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int u = i & ~1; u < 8; u += 2) {
      const double2 v = *reinterpret_cast<const double2*>(&D[8 * jb + i][8 * jb + u]);
      g[i][u] = v.x; g[i][u + 1] = v.y;
    }
#pragma unroll
  for (int u = 0; u < 8; u += 2) {
    const double2 v = *reinterpret_cast<const double2*>(&D[row][8 * jb + u]);
    a[u] = v.x; a[u + 1] = v.y;
  }
  asm volatile("bar.sync 2, 64;" ::: "memory");          // both warps have read the diagonal rows, which one of them overwrites
#pragma unroll
  for (int j = 7; j >= 0; --j) {
    double d = g[j][j];
    if (!(d > 0.0)) {
      if (row == 0) report_error(dev_info, GPTQ_ERR_NOT_PD, k_global + 8 * jb + j);
      d = 1.0;
    }
    const double rp = rsqrt(d);
    const bool own = row == 8 * jb + j;
    double xc[8];
#pragma unroll
    for (int c = 0; c < j; ++c) xc[c] = g[c][j] * rp;
    const double x = own ? rp : a[j] * rp;
#pragma unroll
    for (int c = j - 1; c >= 0; --c) {
#pragma unroll
      for (int i = c; i >= 0; --i) g[i][c] = fma(-xc[i], xc[c], g[i][c]);
      a[c] = fma(-x, xc[c], own ? 0.0 : a[c]);
    }
    a[j] = x;
  }
#pragma unroll
  for (int u = 0; u < 8; u += 2) *reinterpret_cast<double2*>(&D[row][8 * jb + u]) = make_double2(a[u], a[u + 1]);
}
// One warp: the eight columns' update of the 8 x 8 piece (rt, ct), ct < jb.  The rows of piece row jb restart: they take
// only the contributions from their own column on, from zero.
__device__ __forceinline__ void update8(double (*D)[LDD], int rt, int ct, int jb, int lane) {
  const int r = lane >> 2, q = lane & 3;
  double c[2] = {0.0, 0.0};
#pragma unroll
  for (int k = 0; k < 8; k += 4) {
    double x = D[8 * rt + r][8 * jb + k + q];
    if (rt == jb && r < k + q) x = 0.0;
    dmma(c, x, D[8 * ct + r][8 * jb + k + q]);
  }
  double2* out = reinterpret_cast<double2*>(&D[8 * rt + r][8 * ct + 2 * q]);
  double2 v = make_double2(0.0, 0.0);
  if (rt != jb) v = *out;
  *out = make_double2(v.x - c[0], v.y - c[1]);
}
// All threads: D (upper triangle valid) -> D[i][j] = V[j][i] for i >= j, V = T^-1.  The same fused sweep as over the tiles,
// eight columns at a time: warps 0 and 1 run the columns, then every warp updates one 8 x 8 piece of the next eight columns,
// and while warps 0 and 1 go on with those the other warps update the rest.
__device__ __forceinline__ void factor64(Smem& s, int t, int k_global, int* dev_info) {
  const int warp = t >> 5, lane = t & 31;
#pragma unroll 1
  for (int jb = 7; jb >= 0; --jb) {
    if (warp < 2) {
      sweep8(s.D, jb, t, k_global, dev_info);
    } else {                                            // panel jb + 1's update of the columns before panel jb
      for (int e = warp - 2; e < 8 * jb && jb < 7; e += 6) {
        const int rt = e & 7, ct = e >> 3;
        if (rt <= ct || rt > jb) update8(s.D, rt, ct, jb + 1, lane);
      }
    }
    __syncthreads();
    if (jb > 0) update8(s.D, warp, jb - 1, jb, lane);
    __syncthreads();
  }
}

// ---- the chain ----------------------------------------------------------------------------------------------
// All threads: waits until tiles (k, k) and (k, k + 1) have seen n updates.  If nobody has taken the entries of the list that
// lead there (no other CTA of this launch is resident), this CTA runs them itself: entries below `limit` depend only on
// steps that the chain has already passed.  helped: it ran some, and the tiles in shared memory are not what they were.
__device__ __forceinline__ bool chain_wait(const Args& a, Smem& s, int k, int n, int limit, int t, bool& helped) {
  const int* p = &a.fl->updated[k * kMaxTiles + k];
  uint64_t t0 = 0;
  helped = false;
  for (;;) {
    // two threads look at one tile each
    bool ready = true;
    if (t == 0) ready = ld_acquire(p) >= n;
    if (t == 32) ready = ld_acquire(p + 1) >= n;
    if (__syncthreads_and(ready)) return true;
    if (t == 0) {
      int m = 0;
      const uint64_t now = umma::global_timer_ns();
      if (t0 == 0) t0 = now;
      if (ld_acquire(&a.fl->abort)) m = 3;
      else if (now - t0 > umma::g_wait_limit_ns) {
        report_error(a.dev_info, GPTQ_ERR_TIMEOUT, 62);
        st_release(&a.fl->abort, 1);
        m = 3;
      } else if (now - t0 > 20000) {
        int cur = ld_acquire(&a.fl->ticket);
        while (cur < limit) {
          const int seen = atomicCAS(&a.fl->ticket, cur, cur + 1);
          if (seen == cur) { m = 2; s.msg[1] = cur; break; }
          cur = seen;
        }
      }
      s.msg[0] = m;
    }
    __syncthreads();
    const int m = s.msg[0], ticket = s.msg[1];
    __syncthreads();
    if (m == 3) return false;
    if (m == 2) {
      helped = true;
      if (!run_task(a, s, task_of(a.nt, ticket), t)) return false;
    }
  }
}

// Step k of an even column with a right neighbour, fp64: T[k][k + 1] = M[k][k + 1] V^T, and D = M[k][k] - T T^T.  D holds the
// neighbour's inverse (transposed) on entry.
__device__ __forceinline__ void pair_step(const Args& a, Smem& s, int k, int t) {
  const int warp = t >> 5, r = (t & 31) >> 2, q = t & 3;
  load_tile(a, k, k + 1, s.As, t);
  load_tile(a, k, k, s.Bs, t);
  __syncthreads();
  double y[8][2];
#pragma unroll
  for (int ct = 0; ct < 8; ++ct) y[ct][0] = y[ct][1] = 0.0;
#pragma unroll
  for (int kc = 0; kc < 16; ++kc) {
    const double x = (double)s.As[8 * warp + r][4 * kc + q];
#pragma unroll
    for (int ct = 0; ct < kc / 2 + 1; ++ct) {
      const double v = s.D[4 * kc + q][8 * ct + r];
      dmma(y[ct], x, 4 * kc + q >= 8 * ct + r ? v : 0.0);
    }
  }
  __syncthreads();                                      // everybody has read V
  float* out = a.A + (int64_t)(TB * k + 8 * warp + r) * a.ld + TB * (k + 1) + 2 * q;
#pragma unroll
  for (int ct = 0; ct < 8; ++ct) {
    *reinterpret_cast<double2*>(&s.D[8 * warp + r][8 * ct + 2 * q]) = make_double2(y[ct][0], y[ct][1]);
    if (TB * (k + 1) + 8 * ct + 2 * q < a.w) *reinterpret_cast<float2*>(out + 8 * ct) = make_float2((float)y[ct][0], (float)y[ct][1]);
  }
  __syncthreads();
  if (t == 0) st_release(&a.fl->solved[k * kMaxTiles + k + 1], 1);
  store_pair_tile(pair_tile(a, k, kPairT), s.D, t);
  // The 36 8 x 8 pieces on or above the diagonal, column by column (piece e = rt + ct (ct + 1) / 2), five per warp side by side;
  // the fifth of warps 4 .. 7 is not there (they repeat their first and drop it).
  int ar[5], br[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const int e = warp + 8 * i < 36 ? warp + 8 * i : warp;
    const int ct = e < 1 ? 0 : e < 3 ? 1 : e < 6 ? 2 : e < 10 ? 3 : e < 15 ? 4 : e < 21 ? 5 : e < 28 ? 6 : 7;
    ar[i] = 8 * (e - ct * (ct + 1) / 2); br[i] = 8 * ct;
  }
  double z[5][2];
#pragma unroll
  for (int i = 0; i < 5; ++i) z[i][0] = z[i][1] = 0.0;
#pragma unroll 4
  for (int kc = 0; kc < 16; ++kc)
#pragma unroll
    for (int i = 0; i < 5; ++i) dmma(z[i], s.D[ar[i] + r][4 * kc + q], s.D[br[i] + r][4 * kc + q]);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    if (warp + 8 * i >= 36) continue;
    const float2 m = *reinterpret_cast<const float2*>(&s.Bs[ar[i] + r][br[i] + 2 * q]);
    *reinterpret_cast<double2*>(&s.D[ar[i] + r][br[i] + 2 * q]) = make_double2((double)m.x - z[i][0], (double)m.y - z[i][1]);
  }
  __syncthreads();
}

__device__ __forceinline__ bool run_chain(const Args& a, Smem& s, int t) {
  const int nt = a.nt, tx = t & 15, ty = t >> 4;
  for (int k = nt - 1; k >= 0; --k) {
    const bool paired = !(k & 1) && k + 1 < nt;          // with column k + 1
    bool helped = false;
    const int limit = tasks_before_step(nt, k + 1);
    if (k < nt - 1 && !chain_wait(a, s, k, nt - 2 - k, limit, t, helped)) return false;
    if (paired) {
      if (helped) load_pair_tile(pair_tile(a, k, kPairV1), s.D, t);
      pair_step(a, s, k, t);
    } else {
      float old[4][4], acc[4][4];
      const float* Mkk = a.A + (int64_t)(TB * k + ty) * a.ld + TB * k + tx;
      auto load_diag = [&]() {
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int r = ty + 16 * p, c = tx + 16 * q;
            old[p][q] = r == c ? 1.f : 0.f;                             // rows beyond the block: identity
            if (TB * k + r < a.w && TB * k + c < a.w && r <= c) old[p][q] = __ldcg(Mkk + (int64_t)(16 * p) * a.ld + 16 * q);
            acc[p][q] = 0.f;
          }
      };
      if (k < nt - 1) {
        // T[k][k + 1] = M[k][k + 1] V^T, and its update of tile (k, k).  (Bs holds V_{k+1}, left there by the last step.)
        load_tile(a, k, k + 1, s.As, t);
        if (limit > 0) load_tile(a, k + 1, k + 1, s.Bs, t);             // (helping out may have overwritten Bs)
        load_diag();
        __syncthreads();
        product(s.As, s.Bs, acc, tx, ty);
        __syncthreads();
        float* out = a.A + (int64_t)(TB * k + ty) * a.ld + TB * (k + 1) + tx;
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            s.As[ty + 16 * p][tx + 16 * q] = acc[p][q];
            if (TB * (k + 1) + tx + 16 * q < a.w) out[(int64_t)(16 * p) * a.ld + 16 * q] = acc[p][q];
          }
        __syncthreads();
        if (t == 0) { st_release(&a.fl->solved[k * kMaxTiles + k + 1], 1); }
        product<true>(s.As, s.As, acc, tx, ty);
      } else {
        load_diag();
      }
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) s.D[ty + 16 * p][tx + 16 * q] = (double)old[p][q] - (double)acc[p][q];
      __syncthreads();
    }
    factor64(s, t, a.k_global + TB * k, a.dev_info);
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = ty + 16 * p, c = tx + 16 * q;
        const float v = c >= r ? (float)s.D[c][r] : 0.f;
        s.Bs[r][c] = v;
        if (TB * k + r < a.w && TB * k + c < a.w) a.A[(int64_t)(TB * k + r) * a.ld + TB * k + c] = v;
      }
    __syncthreads();
    if (t == 0) st_release(&a.fl->factored, nt - k);
    // the inverse in fp64, for the pair (off the chain: what waits for it has most of a step's time)
    if (k & 1) {
      store_pair_tile(pair_tile(a, k, kPairV1), s.D, t);
    } else if (paired) {
      store_pair_tile(pair_tile(a, k, kPairV0), s.D, t);
      __syncthreads();
      if (t == 0) st_release(&a.fl->paired[k >> 1], 1);
    }
  }
  return true;
}

__global__ void __launch_bounds__(kThreads, 2) panel_factor_kernel(const Args a) {
  extern __shared__ __align__(16) unsigned char panel_smem[];
  Smem& s = *reinterpret_cast<Smem*>(panel_smem);
  const int t = threadIdx.x;
  if (t == 0) s.msg[0] = atomicAdd(&a.fl->role, 1);
  __syncthreads();
  const bool chain = s.msg[0] == 0;
  __syncthreads();
  if (!chain && umma::g_skip_loads_of_item == umma::kPanelChainAlone) return;       // (test knob)
  if (chain && !run_chain(a, s, t)) return;
  for (;;) {
    if (t == 0) s.msg[0] = atomicAdd(&a.fl->ticket, 1);
    __syncthreads();
    const Task k = task_of(a.nt, s.msg[0]);
    __syncthreads();
    if (k.kind < 0 || !run_task(a, s, k, t)) return;
  }
}

// Second launch: the transposed inverse moves from the lower tiles to its place above the diagonal, zeros below it, and the
// progress words are cleared for the next panel.  32 x 32 pieces, grid (w / 32, w / 32), block (32, 8).
__global__ void __launch_bounds__(256) panel_place_inverse_kernel(float* __restrict__ A, int64_t ld, Flags* fl) {
  __shared__ float tile[32][33];
  const int bi = blockIdx.y, bj = blockIdx.x, tx = threadIdx.x, ty = threadIdx.y;
  if (bi == 0 && bj == 0) {
    int* f = reinterpret_cast<int*>(fl);
    for (int e = ty * 32 + tx; e < (int)(sizeof(Flags) / 4); e += 256) f[e] = 0;
  }
  if ((bi >> 1) <= (bj >> 1)) return;                    // inside a diagonal tile V stands already
  float* src = A + (int64_t)(32 * bi) * ld + 32 * bj;
  float* dst = A + (int64_t)(32 * bj) * ld + 32 * bi;
#pragma unroll
  for (int p = 0; p < 4; ++p) { tile[ty + 8 * p][tx] = src[(int64_t)(ty + 8 * p) * ld + tx]; src[(int64_t)(ty + 8 * p) * ld + tx] = 0.f; }
  __syncthreads();
#pragma unroll
  for (int p = 0; p < 4; ++p) dst[(int64_t)(ty + 8 * p) * ld + tx] = tile[tx][ty + 8 * p];
}

// Factors and inverts the w x w block at A (leading dimension ld) on stream s: its upper triangle holds V = T^-1
// afterwards, zeros below.  `fl` must be all zero and is left so; `pairs`: pair_doubles(w) of scratch.  max_ctas: how many CTAs
// may be spent on it.
inline gptq_status_t launch(float* A, int64_t ld, int w, int k_global, Flags* fl, double* pairs, int* dev_info, int max_ctas, cudaStream_t s) {
  Args a{A, ld, w, ceil_div(w, TB), k_global, fl, pairs, dev_info};
  const int products = tasks_before_step(a.nt, -1);
  // no more CTAs than the widest step has products
  int widest = 1;
  for (int k = 0; k < a.nt; ++k) widest = step_updates(a.nt, k) + 1 > widest ? step_updates(a.nt, k) + 1 : widest;
  int ctas = widest < max_ctas ? widest : max_ctas;
  if (ctas > products + 1) ctas = products + 1;
  GPTQ_CUDA_TRY(cudaFuncSetAttribute(panel_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem)));
  panel_factor_kernel<<<ctas, kThreads, sizeof(Smem), s>>>(a);
  GPTQ_LAUNCH_CHECK();
  dim3 grid(w / 32, w / 32), blk(32, 8);
  panel_place_inverse_kernel<<<grid, blk, 0, s>>>(A, ld, fl);
  GPTQ_LAUNCH_CHECK();
  return GPTQ_OK;
}

}  // namespace panel
}  // namespace
}  // namespace gptq
