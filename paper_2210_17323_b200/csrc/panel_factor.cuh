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
// The chain in turn is that of one warp: eight columns, the next 8 x 8 piece, eight columns (factor_chain).  Its SM does the other fp64
// products of a step (about 1000 DMMAs of 16 cycles on three quarters of the SM) in warps that run beside it, each with a row of pieces
// in registers; T T^T and the inverse, which nothing else waits for, follow at their own pace.
// Measured, columns of one call: as separate launches 768 / 1024 0.94 / 1.29 ms; this list with a chain of eight warps that met at a barrier
// twice every eight columns, roots on it, 0.189 / 0.247 (30,600 cycles a step); this form 0.141 / 0.182 (20,000, of which 17,500 the chain's
// own and the rest waiting for products; 0.135 / 0.176 with the launches around it set up early).
#pragma once

namespace gptq {
namespace {
namespace panel {

constexpr int TB = 64;               // tile edge
constexpr int kMaxTiles = 16;        // w <= 1024
constexpr int kThreads = 512;        // the chain's; products are made by the first kGroup
constexpr int kGroup = 256;
constexpr int LDF = 68;              // fp32 tile pitch (floats): 16-byte rows, eight rows on distinct bank groups
constexpr int LDD = 72;              // fp64 tile pitch (doubles): two rows 64 bytes apart modulo 128, conflict-free 16-byte fragments
// fp64 tiles of a pair of tile columns (k, k + 1), k even: the inverse of column k + 1's diagonal tile, the tile between them, the
// inverse of column k's.
constexpr int kPairV1 = 0, kPairT = 1, kPairV0 = 2, kPairTiles = 3;

// Progress of one launch, in the caller's workspace; all zero when the kernel starts.
struct Flags {
  int factored;                      // tile columns factored so far (from the last one); on a line of its own, which most of the waiting look at
  int unused[31];
  int role;                          // order of arrival: 0 runs the chain
  int ticket;                        // next half of an entry of the list of products
  int abort;                         // a wait ran out: everybody leaves
  int unused2[21];
  int solved[kMaxTiles * kMaxTiles]; // halves of tile (i, k) that have been through step k's solve
  int updated[kMaxTiles * kMaxTiles];// updates applied to halves of tile (i, c)
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

// What 256 threads need for one entry of the list of products.
struct TaskSmem {
  union {
    struct { float As[32][LDF]; float Bs[TB][LDF]; };
    double E[TB][LDD];
  };
  union {
    double P[TB][LDD];
    float sums[2][2][4][128];
  };
  int msg[4];
};
struct ChainSmem {
  double D[TB][LDD];                 // pieces (i, c), c >= i: V_kk, rows times 1 / root; (i, c), c < i: Y of panel i, row c (see factor_chain)
  double T[TB][LDD];                 // T[k][k + 1]
  float Md[TB][LDD], Mx[TB][LDD];    // tiles (k, k) and (k, k + 1) before step k
  double vg[8][64], rcp[8][8], piv[8][8];   // of every panel of a step, see eliminate8
  double next[2][2][64], G[64];
  double root[TB];                   // 1 / sqrt(pivot) of the tile's columns
  uint64_t ttt[8], solved[8], inverse[8];   // column c's T T^T is there; panel jb's V_g and Y; rows 8 jb .. of V (one phase each per step)
  int got, done, go;                 // step whose tiles are in Md and Mx; step whose chain is over; the chain may go on
};
struct Smem {
  TaskSmem task;                     // (task.E: T T^T, beside the chain)
  ChainSmem c;
  int role;
};

__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int threads) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
// Named barriers.  Of a step of the chain: V_g of panel jb is there (1 + jb % 2), its Y is (3), the chain's next two pieces are (4), the
// step's tiles have been read (5), the warps that fetch tiles (6), those that hand the last rows of V out (7), the roots of a panel (9), the
// next step's tiles are there (10).
// Of products: 8.
constexpr int kBarV = 1, kBarY = 3, kBarNext = 4, kBarRead = 5, kBarFetch = 6, kBarOut = 7, kBarGroup = 8, kBarRoot = 9, kBarTiles = 10;
constexpr int kRows = 8 * 32, kFetch = 3 * 32, kOut = 3 * 32;   // threads that own a row of pieces; that fetch; that hand the last rows out

// ---- waiting -------------------------------------------------------------------------------------
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int ld_relaxed(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void add_release(int* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// The first n <= 32 lanes of a warp: each waits until its own *p >= v, looking at the same time (a look takes 700 cycles); false if the
// launch is being abandoned.
__device__ __forceinline__ bool wait_all_ge(const int* p, int v, int n, const Args& a) {
  const int lane = threadIdx.x & 31;
  uint64_t t0 = 0;
  uint32_t looks = 0;
  for (;;) {
    if (__all_sync(0xffffffffu, lane >= n || ld_acquire(p) >= v)) return true;
    const uint64_t now = umma::global_timer_ns();
    bool out = false;
    if (t0 == 0) {
      t0 = now;
    } else if (now - t0 > umma::g_wait_limit_ns) {
      if (lane == 0) {
        report_error(a.dev_info, GPTQ_ERR_TIMEOUT, 61);
        st_release(&a.fl->abort, 1);
      }
      out = true;
    } else if (lane == 0 && (++looks & 15) == 0) {
      out = ld_acquire(&a.fl->abort) != 0;
    }
    if (__any_sync(0xffffffffu, out)) return false;
    __nanosleep(40);                                     // (a hundred warps wait like this one, and a look delays the others')
  }
}

// ---- the list of products ---------------------------------------------------------------------------
// Step k: the solves (rows k - 2 .. 0, then k + 1 .. nt - 1; row k - 1 belongs to the chain), then the updates column by
// column, c = k - 1 .. 0, rows c .. 0 and then k .. nt - 1 (tile (k - 1, k - 1) belongs to the chain): what the chain needs
// next comes first.  An entry is taken in two halves of 32 rows, two tickets.
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
// 32 rows of a tile product by 256 threads, half of the 64 products of an entry by each 128 of them: acc[p][q] = sum_m As[ty + 8 p][m] *
// Bs[tx + 16 q][m] over the half's m.  What bounds it is the shared-memory pipe, four cycles per 16-byte load and warp: 64 loads a thread
// (with 2 x 4 entries a thread and all 64 products 96, 2700 cycles; 768 / 1024 columns 142 / 185 us against 141 / 182).
__device__ __forceinline__ void product(const float (*As)[LDF], const float (*Bs)[LDF], float (&acc)[4][4], int tx, int ty, int m0) {
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[p][q] = 0.f;
#pragma unroll
  for (int m = 0; m < TB / 2; m += 4) {
    float4 x[4], y[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) x[p] = *reinterpret_cast<const float4*>(&As[ty + 8 * p][m0 + m]);
#pragma unroll
    for (int q = 0; q < 4; ++q) y[q] = *reinterpret_cast<const float4*>(&Bs[tx + 16 * q][m0 + m]);
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        acc[p][q] = fmaf(x[p].x, y[q].x, acc[p][q]); acc[p][q] = fmaf(x[p].y, y[q].y, acc[p][q]);
        acc[p][q] = fmaf(x[p].z, y[q].z, acc[p][q]); acc[p][q] = fmaf(x[p].w, y[q].w, acc[p][q]);
      }
  }
}
__device__ __forceinline__ void copy_async_16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(umma::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// kLoad rows of tile (i, c) of the block, from row r0 of it on, into shared memory, zeros beyond the block.  The tiles were written by other
// CTAs of this launch: the copies bypass L1.
template <int kLoad>
__device__ __forceinline__ void load_tile(const Args& a, int i, int c, int r0, float (*S)[LDF], int t) {
  const int q = t & 15, row = t >> 4;
#pragma unroll
  for (int p = 0; p < kLoad / 16; ++p) {
    const int r = TB * i + r0 + row + 16 * p, col = TB * c + 4 * q;
    float* d = &S[row + 16 * p][4 * q];
    if (r < a.w && col < a.w) copy_async_16(d, a.A + (int64_t)r * a.ld + col);
    else *reinterpret_cast<float4*>(d) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}
// S = rows r0 .. r0 + 31 of tile (i, c)^T
__device__ __forceinline__ void load_tile_t(const Args& a, int i, int c, int r0, float (*S)[LDF], int t) {
  const int q = t & 7, row = t >> 3;
  float4 v[2];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const int r = TB * i + row + 32 * p, col = TB * c + r0 + 4 * q;
    v[p] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < a.w && col < a.w) v[p] = __ldcg(reinterpret_cast<const float4*>(a.A + (int64_t)r * a.ld + col));
  }
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    S[4 * q][row + 32 * p] = v[p].x; S[4 * q + 1][row + 32 * p] = v[p].y; S[4 * q + 2][row + 32 * p] = v[p].z; S[4 * q + 3][row + 32 * p] = v[p].w;
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
  for (int p = 0; p < 8; ++p) v[p] = __ldcg(reinterpret_cast<const double2*>(src) + t + kGroup * p);
#pragma unroll
  for (int p = 0; p < 8; ++p) { const int e = t + kGroup * p; *reinterpret_cast<double2*>(&S[e >> 5][2 * (e & 31)]) = v[p]; }
}
// A pair's tile of the inverse, 256 threads: V[k][k + 1] = -V_kk T[k][k + 1] V_{k+1,k+1}, transposed into tile (k + 1, k).  Warp
// `rt` makes the eight rows 8 rt .. of each product; entries on the wrong side of a triangle are skipped or read as zero.
__device__ __forceinline__ bool pair_inverse(const Args& a, TaskSmem& s, int k, int t) {
  const int rt = t >> 5, r = (t & 31) >> 2, q = t & 3;
  if (t < 32) {
    const bool ok = wait_all_ge(&a.fl->paired[k >> 1], 1, 1, a);
    if (t == 0) s.msg[3] = ok ? 1 : 0;
  }
  bar_sync(kBarGroup, kGroup);                                      // (also: the previous product is done with the tiles)
  if (!s.msg[3]) return false;
  load_pair_tile(pair_tile(a, k, kPairT), s.E, t);
  load_pair_tile(pair_tile(a, k, kPairV1), s.P, t);
  bar_sync(kBarGroup, kGroup);
  double y[8][2];
#pragma unroll
  for (int ct = 0; ct < 8; ++ct) y[ct][0] = y[ct][1] = 0.0;
#pragma unroll
  for (int kc = 0; kc < 16; ++kc) {
    const double x = s.E[8 * rt + r][4 * kc + q];
#pragma unroll
    for (int ct = kc / 2; ct < 8; ++ct) {
      const double v = s.P[4 * kc + q][8 * ct + r];
      dmma(y[ct], x, 4 * kc + q <= 8 * ct + r ? v : 0.0);
    }
  }
  bar_sync(kBarGroup, kGroup);
#pragma unroll
  for (int ct = 0; ct < 8; ++ct) *reinterpret_cast<double2*>(&s.E[8 * rt + r][8 * ct + 2 * q]) = make_double2(y[ct][0], y[ct][1]);
  load_pair_tile(pair_tile(a, k, kPairV0), s.P, t);
  bar_sync(kBarGroup, kGroup);
#pragma unroll
  for (int ct = 0; ct < 8; ++ct) y[ct][0] = y[ct][1] = 0.0;
#pragma unroll 2
  for (int kc = 2 * rt; kc < 16; ++kc) {
    const double v = s.P[8 * rt + r][4 * kc + q], x = 4 * kc + q >= 8 * rt + r ? v : 0.0;
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
  bar_sync(kBarGroup, kGroup);
  if (t == 0) st_release(&a.fl->solved[(k + 1) * kMaxTiles + k], 2);
  return true;
}

// One half (rows 32 half .. 32 half + 31) of an entry of the list, 256 threads.  False if the launch is being abandoned.  (A pair's inverse
// is made whole, with the first half.)
__device__ __forceinline__ bool run_task(const Args& a, TaskSmem& s, const Task& k, int half, int t) {
  const int nt = a.nt, tx = t & 15, ty = (t >> 4) & 7, h = t >> 7;
  Flags* fl = a.fl;
  if (k.c + 1 == k.k && (k.k & 1) && k.i == k.k) return true;                     // part of pair_inverse
  if (k.kind == 0 && k.i == k.k + 1 && !(k.k & 1)) return half != 0 || pair_inverse(a, s, k.k, t);
  const bool own = k.i == k.k && k.kind == 1;           // a lower tile's first update: it starts as zero, from the inverse itself
  if (t < 32) {
    const int* p = &fl->updated[k.i * kMaxTiles + k.c];
    int v = 2 * updates_before(nt, k.i, k.c, k.k);
    if (t == 1) { p = k.kind == 0 || own ? &fl->factored : &fl->solved[k.i * kMaxTiles + k.k]; v = k.kind == 0 || own ? nt - k.k : 2; }
    if (t == 2) { p = &fl->solved[k.c * kMaxTiles + k.k]; v = 2; }
    const bool ok = wait_all_ge(p, v, k.kind == 0 ? 2 : 3, a);
    if (t == 0) s.msg[3] = ok ? 1 : 0;
  }
  bar_sync(kBarGroup, kGroup);                          // (also: the previous product is done with As and Bs)
  if (!s.msg[3]) return false;
  const int r0 = 32 * half, row = r0 + ty + 16 * h;      // this thread's results: rows row and row + 8, columns tx + 16 q
  float* out = a.A + (int64_t)(TB * k.i + row) * a.ld + TB * k.c + tx;
  float old[2][4];
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      old[p][q] = 0.f;
      if (k.kind == 1 && !own && TB * k.i + row + 8 * p < a.w && TB * k.c + tx + 16 * q < a.w)
        old[p][q] = __ldcg(out + (int64_t)(8 * p) * a.ld + 16 * q);
    }
  load_tile<TB>(a, k.kind == 0 ? k.k : k.c, k.k, 0, s.Bs, t);
  if (own) load_tile_t(a, k.k, k.k, r0, s.As, t); else load_tile<32>(a, k.i, k.k, r0, s.As, t);
  copy_async_wait();
  bar_sync(kBarGroup, kGroup);
  float acc[4][4];
  product(s.As, s.Bs, acc, tx, ty, TB / 2 * h);
  // the other half's rows (p = 0, 1 belong to h = 0, p = 2, 3 to h = 1) through shared memory
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) s.sums[h][p][q][t & 127] = h ? acc[p][q] : acc[p + 2][q];
  bar_sync(kBarGroup, kGroup);
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float v = (h ? acc[p + 2][q] : acc[p][q]) + s.sums[h ^ 1][p][q][t & 127];
      if (TB * k.i + row + 8 * p < a.w && TB * k.c + tx + 16 * q < a.w)
        out[(int64_t)(8 * p) * a.ld + 16 * q] = k.kind == 0 ? v : old[p][q] - v;
    }
  bar_sync(kBarGroup, kGroup);
  if (t == 0)                                           // (the release covers what the barrier has collected from all threads)
    add_release(k.kind == 0 ? &fl->solved[k.i * kMaxTiles + k.k] : &fl->updated[k.i * kMaxTiles + k.c], 1);
  return true;
}

// ---- factor + inverse of one 64 x 64 tile (fp64) ----------------------------------------------------------
// Everything is made of 8 x 8 pieces, the shape of one DMMA accumulator: lane (r, q) = (lane / 4, lane % 4) holds entries (r, 2 q) and
// (r, 2 q + 1).  A product's index may be taken in any order, so with the even entries as one k step and the odd ones as the other an
// accumulator IS a left operand (x[0], x[1]), and a right operand is the same pair of a row-major piece's row r.
__device__ __forceinline__ void dmma8(double (&c)[2], double a0, double a1, double2 b) { dmma(c, a0, b.x); dmma(c, a1, b.y); }

// One panel of eight columns: G = T_g T_g^T, its diagonal piece (upper triangle, row-major).  What leaves here is not scaled by roots:
// with T_g = Y sqrt(1 / piv), vg[j][i] = entry j of unit row i after the elimination (V_g^T before its columns are scaled; zero for j > i),
// rcp[j] = 1 / piv[j].  So nothing but a reciprocal stands between one column and the next, and whoever needs V scales it himself.
// Every lane carries all of G and eliminates it redundantly; lane i % 8 == lane carries unit row i beside it, which starts at column i.
// The quotient of the next pivot's column is formed by Goldschmidt's method (R. E. Goldschmidt, 1964): with y an approximation of 1 / d to 20
// bits and e = 1 - d y, g / d = (g y)(1 + e)(1 + e^2) up to e^4.  The range of d is checked for all eight columns at the end.  (Cycles for
// eight columns: rsqrt() one after the other 1290, two at a time through determinants 1700 -- each call is a branch --, this 660.)
__device__ __forceinline__ bool eliminate8(const double* G, double* vg, double* rcp, double* piv, int lane) {
  double g[8][8], a[8], rc[8];                           // g[i][c], i <= c
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int u = i & ~1; u < 8; u += 2) {
      const double2 v = *reinterpret_cast<const double2*>(G + 8 * i + u);
      g[i][u] = v.x; g[i][u + 1] = v.y;
    }
#pragma unroll
  for (int u = 0; u < 8; ++u) a[u] = (lane & 7) == u ? 1.0 : 0.0;
  bool in_range = true;
#pragma unroll
  for (int j = 7; j >= 0; --j) {
    const double d = g[j][j];
    in_range &= (uint32_t)__double2hiint(d) - (123u << 20) < (1800u << 20);            // 2^-900 <= d < 2^900
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-d, y, 1.0), e2 = e * e;
    double l[8];
    if (j > 0) {
      const double n = g[j - 1][j] * y, m = fma(n, e, n);
      l[j - 1] = fma(m, e2, m);
      g[j - 1][j - 1] = fma(-l[j - 1], g[j - 1][j], g[j - 1][j - 1]);
    }
    const double y1 = fma(y, e, y);
    rc[j] = fma(y1, e2, y1);
#pragma unroll
    for (int c = j - 2; c >= 0; --c) l[c] = g[c][j] * rc[j];
#pragma unroll
    for (int u = j - 1; u >= 0; --u)
#pragma unroll
      for (int c = u; c >= 0; --c)
        if (c < j - 1) g[c][u] = fma(-l[c], g[u][j], g[c][u]);
#pragma unroll
    for (int c = j - 1; c >= 0; --c) a[c] = fma(-a[j], l[c], a[c]);
  }
  // (Nothing is stored before the end: a store between them holds the loads of G back, 2250 cycles.)
#pragma unroll
  for (int j = 0; j < 8; ++j) vg[8 * j + (lane & 7)] = a[j];
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    *reinterpret_cast<double2*>(rcp + j) = make_double2(rc[j], rc[j + 1]);
    *reinterpret_cast<double2*>(piv + j) = make_double2(g[j][j], g[j + 1][j + 1]);
  }
  return in_range;
}
// The same column by column with rsqrt(), for pivots that are not positive (reported, and replaced by one) or out of the other form's
// range.  Y is T_g itself here, and rcp and piv are ones.
__device__ __noinline__ void eliminate8_by_roots(const double* G, double* vg, double* rcp, double* piv, int lane, int k_global, int* dev_info) {
  double g[8][8], a[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    a[i] = 0.0;
#pragma unroll
    for (int u = i; u < 8; ++u) g[i][u] = G[8 * i + u];
  }
#pragma unroll
  for (int j = 7; j >= 0; --j) {
    double d = g[j][j];
    if (!(d > 0.0)) {
      if (lane == 0) report_error(dev_info, GPTQ_ERR_NOT_PD, k_global + j);
      d = 1.0;
    }
    const double rp = rsqrt(d);
    const bool own = (lane & 7) == j;
    double x[8];
#pragma unroll
    for (int c = 0; c < j; ++c) x[c] = g[c][j] * rp;
    a[j] = own ? rp : a[j] * rp;
#pragma unroll
    for (int c = j - 1; c >= 0; --c) {
#pragma unroll
      for (int i = c; i >= 0; --i) g[i][c] = fma(-x[i], x[c], g[i][c]);
      a[c] = fma(-a[j], x[c], own ? 0.0 : a[c]);
    }
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 8; ++j) vg[8 * j + (lane & 7)] = j <= (lane & 7) ? a[j] : 0.0;
  rcp[lane & 7] = piv[lane & 7] = 1.0;
}

__device__ __forceinline__ void wait_phase(uint64_t* bar, int phase, const Args& a) {
  if (!umma::mbar_wait(bar, (uint32_t)phase & 1u)) report_error(a.dev_info, GPTQ_ERR_TIMEOUT, 63);
}
// The chain's warp: the last column of eight first, its elimination, and what the next one needs: Y = A V_g^T of the piece left of the next
// diagonal one (A, as the owner of that row leaves it in s.next) and the next diagonal piece minus Y (1 / piv) Y^T.
__device__ __forceinline__ void factor_chain(const Args& a, ChainSmem& s, bool first, int k, int lane) {
  const int r = lane >> 2, q = lane & 3;
  {
    const float2 m = *reinterpret_cast<const float2*>(&s.Md[56 + r][56 + 2 * q]);
    double g[2] = {(double)m.x, (double)m.y};
    __syncwarp();
    bar_arrive(kBarRead, 32 + kRows + kFetch);
    if (!first) {                                        // minus the last row of pieces of T, squared
      double d[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
      for (int kb = 0; kb < 8; ++kb) {
        const double2 x = *reinterpret_cast<const double2*>(&s.T[56 + r][8 * kb + 2 * q]);
        dmma(d[0], x.x, x.x);
        dmma(d[1], x.y, x.y);
      }
      g[0] -= d[0][0] + d[1][0]; g[1] -= d[0][1] + d[1][1];
    }
    *reinterpret_cast<double2*>(s.G + 8 * r + 2 * q) = make_double2(g[0], g[1]);
  }
#pragma unroll 1
  for (int jb = 7; jb >= 0; --jb) {
    const int h = jb & 1, threads = 32 * jb;             // (the chain and rows 0 .. jb - 2)
    __syncwarp();
    if (!eliminate8(s.G, s.vg[jb], s.rcp[jb], s.piv[jb], lane)) {
      __syncwarp();
      eliminate8_by_roots(s.G, s.vg[jb], s.rcp[jb], s.piv[jb], lane, a.k_global + TB * k + 8 * jb, a.dev_info);
    }
    __syncwarp();
    if (jb > 1) bar_arrive(kBarV + h, threads);
    if (jb == 0) break;
    const double2 v = *reinterpret_cast<const double2*>(s.vg[jb] + 8 * r + 2 * q), rc = *reinterpret_cast<const double2*>(s.rcp[jb] + 2 * q);
    bar_sync(kBarNext, 64);
    const double2 n = *reinterpret_cast<const double2*>(s.next[h][0] + 8 * r + 2 * q);
    const double2 d = *reinterpret_cast<const double2*>(s.next[h][1] + 8 * r + 2 * q);
    double x[2] = {0.0, 0.0}, g[2] = {d.x, d.y};
    dmma8(x, n.x, n.y, v);
    dmma8(g, -x[0] * rc.x, -x[1] * rc.y, make_double2(x[0], x[1]));
    *reinterpret_cast<double2*>(&s.D[8 * jb + r][8 * (jb - 1) + 2 * q]) = make_double2(x[0], x[1]);
    *reinterpret_cast<double2*>(s.G + 8 * r + 2 * q) = make_double2(g[0], g[1]);
    __syncwarp();
    if (jb > 1) bar_arrive(kBarY, threads);
    if (lane == 0) umma::mbar_arrive(&s.solved[jb]);
  }
  if (lane == 0) umma::mbar_arrive(&s.solved[0]);
  if (lane < 8) s.root[lane] = rsqrt(s.piv[0][lane]);
}

// acc[i] += x b of pieces (jb, jb - i), i = 1 .. n, of s.D.  (One jump into each run of pieces: a branch around every product, and what the
// compiler puts beside it, cost half of the time.)
__device__ __forceinline__ void update_pieces(const ChainSmem& s, int jb, int n, int r, int q, double x0, double x1, double (&acc)[8][2]) {
  double2 b[7];
#define GPTQ_PIECES_DOWN(DO) \
  switch (n) { case 7: DO(7) case 6: DO(6) case 5: DO(5) case 4: DO(4) case 3: DO(3) case 2: DO(2) case 1: DO(1) default:; }
#define GPTQ_LOAD(i) b[i - 1] = *reinterpret_cast<const double2*>(&s.D[8 * jb + r][8 * (jb - i) + 2 * q]);
#define GPTQ_EVEN(i) dmma(acc[i], x0, b[i - 1].x);
#define GPTQ_ODD(i) dmma(acc[i], x1, b[i - 1].y);
  GPTQ_PIECES_DOWN(GPTQ_LOAD)
  GPTQ_PIECES_DOWN(GPTQ_EVEN)
  GPTQ_PIECES_DOWN(GPTQ_ODD)
#undef GPTQ_PIECES_DOWN
#undef GPTQ_LOAD
#undef GPTQ_EVEN
#undef GPTQ_ODD
}

// A warp that owns a row rt of 8 x 8 pieces of the tile, in its registers: acc[i] is piece (rt, jb - i) at panel jb.  Down to panel rt + 2
// they are upper pieces, in step with the chain; from panel rt on pieces of the transposed inverse, which nothing waits for before the end.
// S: pieces of T T^T.
__device__ __forceinline__ void factor_row(const Args& a, ChainSmem& s, const double (*S)[LDD], bool first, int k, int rt, int lane) {
  const int r = lane >> 2, q = lane & 3, phase = a.nt - 1 - k;
  double acc[8][2];
  {
    float* z = a.A + (int64_t)(TB * k + 8 * rt + r) * a.ld + TB * k + 2 * q;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int ct = 7 - i;
      float2 m = make_float2(0.f, 0.f);
      if (rt <= ct) m = *reinterpret_cast<const float2*>(&s.Md[8 * rt + r][8 * ct + 2 * q]);
      else if (TB * k + 8 * rt < a.w) *reinterpret_cast<float2*>(z + 8 * ct) = m;      // below the diagonal the finished tile is zero
      acc[i][0] = (double)m.x; acc[i][1] = (double)m.y;
    }
  }
  __syncwarp();
  bar_arrive(kBarRead, 32 + kRows + kFetch);
  auto minus_ttt = [&](int ct, double (&c)[2]) {
    const double2 v = *reinterpret_cast<const double2*>(&S[8 * rt + r][8 * ct + 2 * q]);
    c[0] -= v.x; c[1] -= v.y;
  };
  // the row's piece of column rt + 1 and its diagonal one, to the chain, which needs them at panel rt + 1
  auto publish = [&](double (&p)[2], double (&d)[2]) {
    if (!first) {
      wait_phase(&s.ttt[rt + 1], phase - 1, a);
      minus_ttt(rt + 1, p);
      minus_ttt(rt, d);
    }
    *reinterpret_cast<double2*>(s.next[(rt + 1) & 1][0] + 8 * r + 2 * q) = make_double2(p[0], p[1]);
    *reinterpret_cast<double2*>(s.next[(rt + 1) & 1][1] + 8 * r + 2 * q) = make_double2(d[0], d[1]);
    __syncwarp();
    bar_arrive(kBarNext, 64);
  };
  if (rt == 6) publish(acc[0], acc[1]);
#pragma unroll 1
  for (int jb = 7; jb >= rt + 2; --jb) {
    const int h = jb & 1;
    if (!first) {
      wait_phase(&s.ttt[jb], phase - 1, a);
      minus_ttt(jb, acc[0]);
    }
    bar_sync(kBarV + h, 32 * jb);
    // Y = (piece of column jb) V_g^T, unscaled, kept for everybody's updates in piece (jb, rt) of s.D
    double x[2] = {0.0, 0.0};
    dmma8(x, acc[0][0], acc[0][1], *reinterpret_cast<const double2*>(s.vg[jb] + 8 * r + 2 * q));
    const double2 rc = *reinterpret_cast<const double2*>(s.rcp[jb] + 2 * q);
    *reinterpret_cast<double2*>(&s.D[8 * jb + r][8 * rt + 2 * q]) = make_double2(x[0], x[1]);
    __syncwarp();
    if (lane == 0) umma::mbar_arrive(&s.solved[jb]);
    bar_sync(kBarY, 32 * jb);
    update_pieces(s, jb, jb - rt, r, q, -x[0] * rc.x, -x[1] * rc.y, acc);
    if (rt == jb - 2) publish(acc[1], acc[2]);
#pragma unroll
    for (int i = 0; i < 7; ++i) { acc[i][0] = acc[i + 1][0]; acc[i][1] = acc[i + 1][1]; }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = 0.0;
#pragma unroll 1
  for (int jb = rt; jb >= 0; --jb) {
    wait_phase(&s.solved[jb], phase, a);
    double x[2] = {0.0, 0.0};
    if (rt == jb) {
      x[0] = s.vg[jb][16 * q + r]; x[1] = s.vg[jb][16 * q + 8 + r];
    } else {
      dmma8(x, acc[0][0], acc[0][1], *reinterpret_cast<const double2*>(s.vg[jb] + 8 * r + 2 * q));
    }
    const double2 rc = *reinterpret_cast<const double2*>(s.rcp[jb] + 2 * q);
    s.D[8 * jb + 2 * q][8 * rt + r] = x[0];
    s.D[8 * jb + 2 * q + 1][8 * rt + r] = x[1];
    __syncwarp();
    if (lane == 0) umma::mbar_arrive(&s.inverse[jb]);
    update_pieces(s, jb, jb, r, q, -x[0] * rc.x, -x[1] * rc.y, acc);
#pragma unroll
    for (int i = 0; i < 7; ++i) { acc[i][0] = acc[i + 1][0]; acc[i][1] = acc[i + 1][1]; }
  }
}

// Four warps (w: 0 .. 3): the pieces of T T^T, two at a time, so that they share an operand, column by column in the order in which the
// rows need them: for column c the two that the chain takes with it, (c - 1, c) and (c - 1, c - 1), then rows c - 2 .. 0.
__host__ __device__ __forceinline__ constexpr int ttt_jobs(int c) { return 1 + c / 2; }
__device__ __forceinline__ void make_ttt(ChainSmem& s, double (*S)[LDD], int w, int lane) {
  const int r = lane >> 2, q = lane & 3;
  int c = 7, i = w;                                      // job i of column c
#pragma unroll 1
  for (;;) {
    while (c > 0 && i >= ttt_jobs(c)) { i -= ttt_jobs(c); --c; }
    if (c == 0) return;
    // pieces (u, c) and (v, c), or (u, c) and (u, u), u = c - 1
    const int u = i == 0 ? c - 1 : c - 2 * i, v = i == 0 ? c - 1 : u - 1, shared = i == 0 ? c - 1 : c, other = i == 0 ? c : u;
    double d[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    const double* ps = &s.T[8 * shared + r][2 * q];
    const double* po = &s.T[8 * other + r][2 * q];
    const double* pv = &s.T[8 * (v < 0 ? 0 : v) + r][2 * q];
#pragma unroll
    for (int kb = 0; kb < 8; ++kb) {
      const double2 y = *reinterpret_cast<const double2*>(ps + 8 * kb), x = *reinterpret_cast<const double2*>(po + 8 * kb);
      const double2 z = *reinterpret_cast<const double2*>(pv + 8 * kb);
      const double2 fa = i == 0 ? y : x, fb = i == 0 ? x : y;
      dmma(d[0], fa.x, fb.x);
      dmma(d[1], z.x, y.x);
      dmma(d[0], fa.y, fb.y);
      dmma(d[1], z.y, y.y);
    }
    *reinterpret_cast<double2*>(&S[8 * u + r][8 * c + 2 * q]) = make_double2(d[0][0], d[0][1]);
    if (v >= 0) *reinterpret_cast<double2*>(&S[8 * v + r][8 * (i == 0 ? c - 1 : c) + 2 * q]) = make_double2(d[1][0], d[1][1]);
    __syncwarp();
    if (lane == 0) umma::mbar_arrive(&s.ttt[c]);
    i += 4;
  }
}
// Rows 8 jb .. 8 jb + 7 of V by warps w, w + n ..: scaled, to the matrix and, in 64 bits, to the pair's tile.
__device__ __forceinline__ void store_inverse(const Args& a, const ChainSmem& s, int k, int jb, int w, int n, double* pair, int lane) {
  if (2 * lane < 8 * jb) return;                         // (pieces left of the diagonal one: zero since the step began)
#pragma unroll 3
  for (int e = w; e < 8; e += n) {
    const int row = 8 * jb + e;
    const double rt = s.root[row];
    double2 v = *reinterpret_cast<const double2*>(&s.D[row][2 * lane]);
    v.x *= rt; v.y *= rt;
    if (TB * k + 2 * lane < a.w) *reinterpret_cast<float2*>(a.A + (int64_t)(TB * k + row) * a.ld + TB * k + 2 * lane) = make_float2((float)v.x, (float)v.y);
    if (pair != nullptr) *reinterpret_cast<double2*>(pair + row * TB + 2 * lane) = v;
  }
}
// The four warps of make_ttt, when that is done: rows of V as they are finished, all but the first eight.
__device__ __forceinline__ void store_inverses(const Args& a, ChainSmem& s, int k, int w, double* pair, int lane) {
#pragma unroll 1
  for (int jb = 7; jb > 0; --jb) {
    wait_phase(&s.inverse[jb], a.nt - 1 - k, a);
    const double rt = rsqrt(s.piv[jb][lane & 7]);
    if (w == 0 && lane < 8) s.root[8 * jb + lane] = rt;
    bar_sync(kBarRoot, 128);
    store_inverse(a, s, k, jb, w, 4, pair, lane);
  }
}

// ---- the chain ----------------------------------------------------------------------------------------------
// 256 threads: waits until tiles (k, k) and (k, k + 1) have seen n updates.  If nobody has taken the entries of the list that
// lead there (no other CTA of this launch is resident), this CTA runs them itself: entries below `limit` depend only on
// steps that the chain has already passed.
__device__ __forceinline__ bool chain_wait(const Args& a, TaskSmem& s, int k, int n, int limit, int t) {
  const int* p = &a.fl->updated[k * kMaxTiles + k];
  uint64_t t0 = 0;
  for (;;) {
    if (t == 0) {
      int m = 0;
      if (ld_acquire(p) >= 2 * n && ld_acquire(p + 1) >= 2 * n) {
        m = 1;
      } else {
        const uint64_t now = umma::global_timer_ns();
        if (t0 == 0) t0 = now;
        if (ld_acquire(&a.fl->abort)) m = 3;
        else if (now - t0 > umma::g_wait_limit_ns) {
          report_error(a.dev_info, GPTQ_ERR_TIMEOUT, 62);
          st_release(&a.fl->abort, 1);
          m = 3;
        } else if (now - t0 > 20000) {
          int cur = ld_acquire(&a.fl->ticket);
          while (cur < 2 * limit) {
            const int seen = atomicCAS(&a.fl->ticket, cur, cur + 1);
            if (seen == cur) { m = 2; s.msg[1] = cur; break; }
            cur = seen;
          }
        }
      }
      s.msg[0] = m;
    }
    bar_sync(kBarGroup, kGroup);
    const int m = s.msg[0], ticket = s.msg[1];
    bar_sync(kBarGroup, kGroup);
    if (m == 1) return true;
    if (m == 3) return false;
    if (m == 2 && !run_task(a, s, task_of(a.nt, ticket >> 1), ticket & 1, t)) return false;
  }
}

// T[k][k + 1] = M[k][k + 1] V^T in 64 bits, V = the inverse in s.D and s.root that the last step left there, to s.T and to the matrix; one
// row of pieces a warp.
__device__ __forceinline__ void chain_solve(const Args& a, ChainSmem& s, int k, int rt, int lane) {
  const int r = lane >> 2, q = lane & 3;
  double y[8][2];
#pragma unroll
  for (int ct = 0; ct < 8; ++ct) y[ct][0] = y[ct][1] = 0.0;
#pragma unroll
  for (int kb = 0; kb < 8; ++kb) {
    const float2 m = *reinterpret_cast<const float2*>(&s.Mx[8 * rt + r][8 * kb + 2 * q]);
    double2 b[8];
#pragma unroll
    for (int ct = 0; ct <= kb; ++ct) b[ct] = *reinterpret_cast<const double2*>(&s.D[8 * ct + r][8 * kb + 2 * q]);
#pragma unroll
    for (int ct = 0; ct <= kb; ++ct) dmma(y[ct], (double)m.x, b[ct].x);
#pragma unroll
    for (int ct = 0; ct <= kb; ++ct) dmma(y[ct], (double)m.y, b[ct].y);
  }
  float* out = a.A + (int64_t)(TB * k + 8 * rt + r) * a.ld + TB * (k + 1) + 2 * q;
#pragma unroll
  for (int ct = 0; ct < 8; ++ct) {
    const double2 rt2 = *reinterpret_cast<const double2*>(&s.root[8 * ct + 2 * q]);
    y[ct][0] *= rt2.x; y[ct][1] *= rt2.y;
    *reinterpret_cast<double2*>(&s.T[8 * rt + r][8 * ct + 2 * q]) = make_double2(y[ct][0], y[ct][1]);
    if (TB * (k + 1) + 8 * ct < a.w) *reinterpret_cast<float2*>(out + 8 * ct) = make_float2((float)y[ct][0], (float)y[ct][1]);
  }
}
// Tiles (k, k) and, unless k is the last column, (k, k + 1) to s.Md and s.Mx by n threads (a multiple of 16): asynchronous copies, zeros
// beyond the block, whose last rows of s.Md are those of the identity.  The caller waits for the copies.
__device__ __forceinline__ void load_chain_tiles(const Args& a, ChainSmem& s, int k, int t, int n) {
  const int c = 4 * (t & 15), step = n >> 4;
  const bool next = k + 1 < a.nt, in0 = TB * k + c < a.w, in1 = next && TB * (k + 1) + c < a.w;
  const float* src = a.A + (int64_t)(TB * k + (t >> 4)) * a.ld + TB * k + c;
#pragma unroll 4
  for (int row = t >> 4; row < TB; row += step, src += step * a.ld) {
    if (in0 && TB * k + row < a.w) copy_async_16(&s.Md[row][c], src);
    else *reinterpret_cast<float4*>(&s.Md[row][c]) = make_float4(row == c ? 1.f : 0.f, row == c + 1 ? 1.f : 0.f, row == c + 2 ? 1.f : 0.f, row == c + 3 ? 1.f : 0.f);
    if (in1) copy_async_16(&s.Mx[row][c], src + TB);
    else if (next) *reinterpret_cast<float4*>(&s.Mx[row][c]) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}
// Three warps beside the factorisation of tile k: they hand out T[k][k + 1] (in 64 bits to the pair's tile), then fetch the next step's
// tiles, if they are ready before the chain is.  (t: 0 .. 95)
__device__ __forceinline__ void chain_fetch(const Args& a, ChainSmem& s, int k, int t) {
  const int nt = a.nt, warp = t >> 5, lane = t & 31;
  if (k + 1 < nt) {
    if (t == 0) st_release(&a.fl->solved[k * kMaxTiles + k + 1], 2);
    if (!(k & 1)) {
      double* pair = pair_tile(a, k, kPairT);
#pragma unroll 1
      for (int row = warp; row < TB; row += 12) {
        double2 v[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) if (row + 3 * p < TB) v[p] = *reinterpret_cast<const double2*>(&s.T[row + 3 * p][2 * lane]);
#pragma unroll
        for (int p = 0; p < 4; ++p) if (row + 3 * p < TB) *reinterpret_cast<double2*>(pair + (row + 3 * p) * TB + 2 * lane) = v[p];
      }
    }
  }
  bar_sync(kBarRead, 32 + kRows + kFetch);
  if (k == 0) return;
  if (warp == 0) {
    const int* p = &a.fl->updated[(k - 1) * kMaxTiles + k - 1];
    bool ready = false;
    while (!(ready = __all_sync(0xffffffffu, lane > 1 || ld_relaxed(p + lane) >= 2 * (nt - 1 - k))))
      if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&s.done) == k)) break;       // (then all threads fetch, see run_chain)
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    if (t == 0 && ready) s.got = k - 1;
  }
  bar_sync(kBarFetch, kFetch);
  if (s.got == k - 1) load_chain_tiles(a, s, k - 1, t, kFetch);
  // (a bulk copy per row into an mbarrier instead of 16-byte copies: 1024 columns 195 us against 182)
}

// All threads.  Warps by role: T[k][k + 1] is made by warps 0 - 3 and 8 - 11, while 13 - 15 hand the last rows of the step before out; then
// warp 0 runs the chain, with a quarter of the SM's fp64 units to itself; rows of pieces belong to eight warps of the other three
// quarters (rows 0 5 6, 1 4 7, 2 3: equal shares of products with the four warps there that make T T^T and store the inverse); and
// warps 4, 8, 12 fetch the next step's tiles.
__device__ __forceinline__ bool run_chain(const Args& a, Smem& sm, int t) {
  ChainSmem& s = sm.c;
  const int nt = a.nt, lane = t & 31, warp = __shfl_sync(0xffffffffu, t >> 5, 0);    // (a value that the compiler sees to be the warp's)
  if (t == 0) {
    s.got = -1; s.done = -1;
    for (int i = 0; i < 8; ++i) {
      umma::mbar_init(&s.ttt[i], ttt_jobs(i)); umma::mbar_init(&s.solved[i], i > 0 ? i : 1); umma::mbar_init(&s.inverse[i], 8 - i);
    }
    umma::fence_barrier_init();
  }
  __syncthreads();
  auto pair_of = [&](int k) { return (k & 1) ? pair_tile(a, k, kPairV1) : k + 1 < nt ? pair_tile(a, k, kPairV0) : nullptr; };
  auto hand_out = [&](int k) {                           // the first rows of V, and word of the whole step
    if (warp < 13) return;
    store_inverse(a, s, k, 0, warp - 13, 3, pair_of(k), lane);
    bar_sync(kBarOut, kOut);
    if (t == 13 * 32) {
      st_release(&a.fl->factored, nt - k);
      if (!(k & 1) && k + 1 < nt) st_release(&a.fl->paired[k >> 1], 1);
    }
  };
  for (int k = nt - 1; k >= 0; --k) {
    const bool first = k == nt - 1;
    if (k == 0 && t == 0) pdl_next();                     // (the other CTAs' leaving counts as theirs)
    if (!first) hand_out(k + 1);
    if (s.got == k) {                                    // (the word goes out before the last tiles are in)
      if ((warp & 3) == 0 && warp > 0) copy_async_wait();
      if ((warp & 4) == 0 || (warp & 3) == 0) bar_sync(kBarTiles, 10 * 32);
    } else {
      if (!first) {
        if (t < kGroup) {
          const bool go = chain_wait(a, sm.task, k, nt - 2 - k, tasks_before_step(nt, k + 1), t);
          if (t == 0) s.go = go;
        }
        __syncthreads();
        if (!s.go) return false;
      }
      load_chain_tiles(a, s, k, t, kThreads);
      copy_async_wait();
      __syncthreads();
    }
    if (!first) {
      if ((warp & 4) == 0) chain_solve(a, s, k, (warp & 3) + (warp >> 3) * 4, lane);
      __syncthreads();
    }
    const int rt = warp == 1 ? 0 : warp == 5 ? 5 : warp == 9 ? 6 : warp == 2 ? 1 : warp == 6 ? 4 : warp == 10 ? 7 : warp == 3 ? 2 : warp == 7 ? 3 : -1;
    if (rt >= 0) {
      factor_row(a, s, sm.task.E, first, k, rt, lane);
    } else if (warp == 0) {
      factor_chain(a, s, first, k, lane);
      if (lane == 0) *reinterpret_cast<volatile int*>(&s.done) = k;
    } else if ((warp & 3) == 0) {
      chain_fetch(a, s, k, t - 128 - (warp / 4 - 1) * 96);
    } else {
      const int w = warp == 11 ? 3 : warp - 13;
      if (!first) make_ttt(s, sm.task.E, w, lane);
      store_inverses(a, s, k, w, pair_of(k), lane);
    }
    __syncthreads();
  }
  hand_out(0);
  return true;
}

__global__ void __launch_bounds__(kThreads, 1) panel_factor_kernel(const Args a) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char panel_smem[];
  Smem& s = *reinterpret_cast<Smem*>(panel_smem);
  const int t = threadIdx.x;
  if (t == 0) s.role = atomicAdd(&a.fl->role, 1);
  __syncthreads();
  const bool chain = s.role == 0;
  if (!chain && umma::g_skip_loads_of_item == umma::kPanelChainAlone) return;       // (test knob)
  if (chain && !run_chain(a, s, t)) return;
  if (t >= kGroup) return;
  for (;;) {
    if (t == 0) s.task.msg[0] = atomicAdd(&a.fl->ticket, 1);
    bar_sync(kBarGroup, kGroup);
    const int ticket = s.task.msg[0];
    const Task k = task_of(a.nt, ticket >> 1);
    bar_sync(kBarGroup, kGroup);
    if (k.kind < 0 || !run_task(a, s.task, k, ticket & 1, t)) return;
  }
}

// Second launch: the transposed inverse moves from the lower tiles to its place above the diagonal, zeros below it, and the
// progress words are cleared for the next panel.  32 x 32 pieces, grid (w / 32, w / 32), block (32, 8).
__global__ void __launch_bounds__(256) panel_place_inverse_kernel(float* __restrict__ A, int64_t ld, Flags* fl) {
  pdl_begin();
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

static_assert(sizeof(Smem) <= 227 * 1024, "a CTA's shared memory");
// Factors and inverts the w x w block at A (leading dimension ld) on stream s: its upper triangle holds V = T^-1
// afterwards, zeros below.  `fl` must be all zero and is left so; `pairs`: pair_doubles(w) of scratch.  max_ctas: how many CTAs
// may be spent on it.
inline gptq_status_t launch(float* A, int64_t ld, int w, int k_global, Flags* fl, double* pairs, int* dev_info, int max_ctas, cudaStream_t s) {
  Args a{A, ld, w, ceil_div(w, TB), k_global, fl, pairs, dev_info};
  const int products = 2 * tasks_before_step(a.nt, -1);
  // no more CTAs than the widest step has halves of products
  int widest = 1;
  for (int k = 0; k < a.nt; ++k) widest = 2 * step_updates(a.nt, k) + 1 > widest ? 2 * step_updates(a.nt, k) + 1 : widest;
  int ctas = widest < max_ctas ? widest : max_ctas;
  if (ctas > products + 1) ctas = products + 1;
  // ... and half a CTA per tile: launches of several layers then run side by side (a CTA takes an SM), and alone nothing is slower from
  // 384 columns on (125M-shaped block, four factors at once: 2168 us without this, 2034 with, 2033 with 3/8; 768-wide layer 340, 340, 350).
  if (a.nt >= 6 && ctas > a.nt * a.nt / 2) ctas = a.nt * a.nt / 2;
  GPTQ_CUDA_TRY(cudaFuncSetAttribute(panel_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem)));
  GPTQ_LAUNCH_NEXT(panel_factor_kernel, ctas, kThreads, sizeof(Smem), s, a);
  dim3 grid(w / 32, w / 32), blk(32, 8);
  GPTQ_LAUNCH_NEXT(panel_place_inverse_kernel, grid, blk, 0, s, A, ld, fl);
  return GPTQ_OK;
}

}  // namespace panel
}  // namespace
}  // namespace gptq
