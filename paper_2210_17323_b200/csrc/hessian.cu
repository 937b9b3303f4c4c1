// Stage 1: H += 2 * sum_t x_t x_t^T  (Section 2, "Optimal Brain Quantization": H = 2 X X^T;
// Algorithm 1 caption).  X arrives token-major (n_tokens x C, bf16).
//
// Only tiles that touch the upper triangle are computed; a mirror pass copies the strict
// upper triangle onto the lower one so both are valid (and exactly symmetric) on return.
#include "common.cuh"
#include "gemm_simt.cuh"
#include "hessian_umma.cuh"

namespace gptq {

namespace {

// A(m, k) = X[k][m]  (the paper's X is C x tokens; memory holds its transpose)
struct XtAsA {
  static constexpr bool kInnerContig = false;
  const __nv_bfloat16* x; int64_t C;
  __device__ __forceinline__ float operator()(int m, int k) const {
    return __bfloat162float(x[(int64_t)k * C + m]);
  }
};
struct XtAsB {
  static constexpr bool kInnerContig = true;
  const __nv_bfloat16* x; int64_t C;
  __device__ __forceinline__ float operator()(int k, int n) const {
    return __bfloat162float(x[(int64_t)k * C + n]);
  }
};
// Tiles strictly below the diagonal are skipped; tokens are split over blockIdx.z.
struct UpperTilesSplitK {
  int64_t n_tokens;
  __device__ __forceinline__ bool operator()(int m0, int n0, int z, int nz, int& k0, int& k1) const {
    if (m0 > n0 + kSimtBN - 1) return false;
    int64_t per = ((n_tokens + nz - 1) / nz + kSimtBK - 1) / kSimtBK * kSimtBK;
    int64_t a = (int64_t)z * per, b = a + per < n_tokens ? a + per : n_tokens;
    k0 = (int)a; k1 = (int)b;
    return a < b;
  }
};
struct AddTwiceUpper {
  float* H; int64_t C;
  __device__ __forceinline__ void operator()(int m, int n, float acc) const {
    if (m <= n) atomicAdd(&H[(int64_t)m * C + n], 2.f * acc);
  }
};

// 64 x 64 tiles on or above the diagonal, one CTA each (a triangular grid: no CTA without work), through shared memory so that
// both the reads and the writes are 256-byte rows; a thread has four 16-byte loads in flight.  Bound by memory: 4096
// channels (67 MB in and out) 12.6 us, 12288 channels 104 us = 5.8 TB/s; one CTA of 1024 threads per 32 x 32 tile, half of
// them below the diagonal without work, took 34.7 and 512 us.
constexpr int kMirrorTile = 64;
__global__ void __launch_bounds__(256) mirror_upper_to_lower_kernel(float* __restrict__ H, int C) {
  __shared__ float t[kMirrorTile][kMirrorTile + 1];
  pdl_wait();
  // linear index -> (bi <= bj): column bj holds the tiles bj (bj + 1) / 2 ...
  const int idx = blockIdx.x;
  int bj = (int)((sqrtf(8.f * (float)idx + 1.f) - 1.f) * 0.5f);
  while ((int64_t)(bj + 1) * (bj + 2) / 2 <= idx) ++bj;
  while ((int64_t)bj * (bj + 1) / 2 > idx) --bj;
  const int bi = idx - (int)((int64_t)bj * (bj + 1) / 2);
  const int r0 = bi * kMirrorTile, c0 = bj * kMirrorTile, q = threadIdx.x & 15, y = threadIdx.x >> 4;
  float4 v[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int r = r0 + y + 16 * p, c = c0 + 4 * q;
    v[p] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < C && c < C) v[p] = *reinterpret_cast<const float4*>(H + (int64_t)r * C + c);
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    t[y + 16 * p][4 * q] = v[p].x; t[y + 16 * p][4 * q + 1] = v[p].y; t[y + 16 * p][4 * q + 2] = v[p].z; t[y + 16 * p][4 * q + 3] = v[p].w;
  }
  __syncthreads();
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int r = c0 + y + 16 * p, c = r0 + 4 * q;        // four elements of the mirrored tile: H[r][c ..] = H[c ..][r]
    if (r >= C || c >= C) continue;
    float* d = H + (int64_t)r * C + c;
    const float x0 = t[4 * q][y + 16 * p], x1 = t[4 * q + 1][y + 16 * p], x2 = t[4 * q + 2][y + 16 * p], x3 = t[4 * q + 3][y + 16 * p];
    if (bi < bj) {
      *reinterpret_cast<float4*>(d) = make_float4(x0, x1, x2, x3);
    } else {                                              // diagonal tile: the part below the diagonal only
      if (r > c) d[0] = x0;
      if (r > c + 1) d[1] = x1;
      if (r > c + 2) d[2] = x2;
      if (r > c + 3) d[3] = x3;
    }
  }
}

}  // namespace

cudaError_t launch_mirror_upper_to_lower(float* H, int C, cudaStream_t stream, bool next) {
  const int64_t n = ceil_div(C, kMirrorTile), tiles = n * (n + 1) / 2;
  if (next) {
    count_launch();
    return launch_next(mirror_upper_to_lower_kernel, (unsigned)tiles, 256, 0, stream, H, C);
  }
  mirror_upper_to_lower_kernel<<<(unsigned)tiles, 256, 0, stream>>>(H, C);
  count_launch();
  return cudaGetLastError();
}

static gptq_status_t hessian_simt(float* H, const __nv_bfloat16* X, int64_t n_tokens, int C,
                                  cudaStream_t stream, bool mirror) {
  const int64_t kMaxTokensPerLaunch = 1 << 30;  // K indices are 32-bit inside the tile kernel
  for (int64_t t0 = 0; t0 < n_tokens; t0 += kMaxTokensPerLaunch) {
    int64_t nt = n_tokens - t0 < kMaxTokensPerLaunch ? n_tokens - t0 : kMaxTokensPerLaunch;
    const __nv_bfloat16* x = X + t0 * C;
    int tiles = ceil_div(C, kSimtBM);
    int upper = tiles * (tiles + 1) / 2;
    int nz = 1;
    while (upper * nz < 2 * 148 && nz * 2 * 512 <= nt) nz *= 2;
    GPTQ_CUDA_TRY(launch_gemm_simt(C, C, nz, XtAsA{x, C}, XtAsB{x, C}, UpperTilesSplitK{nt},
                                   AddTwiceUpper{H, C}, stream));
  }
  if (mirror) GPTQ_CUDA_TRY(launch_mirror_upper_to_lower(H, C, stream, false));
  return GPTQ_OK;
}

}  // namespace gptq

extern "C" size_t gptq_hessian_workspace_bytes(int C, int64_t n_tokens) {
  (void)C; (void)n_tokens;
  return 0;
}

static gptq_status_t hessian_accumulate_impl(float* H, const void* X_bf16, int64_t n_tokens, int C, int* dev_info,
                                             void* stream, bool mirror) {
  using namespace gptq;
  if (!H || C <= 0 || C % 32 != 0 || n_tokens < 0) return GPTQ_ERR_INVALID_ARG;
  if (n_tokens == 0) return GPTQ_OK;
  if (!X_bf16 || !aligned_to(X_bf16, 16) || !aligned_to(H, 16)) return GPTQ_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const __nv_bfloat16* X = static_cast<const __nv_bfloat16*>(X_bf16);
  if (dev_info) GPTQ_CUDA_TRY(cudaMemsetAsync(dev_info, 0, 2 * sizeof(int), s));
  if (hessian_umma_supported(C, n_tokens)) return hessian_umma(H, X, n_tokens, C, dev_info, s, mirror);
  return hessian_simt(H, X, n_tokens, C, s, mirror);
}

extern "C" gptq_status_t gptq_hessian_accumulate(float* H, const void* X_bf16, int64_t n_tokens, int C,
                                                 void* ws, size_t ws_bytes, int* dev_info, void* stream) {
  (void)ws; (void)ws_bytes;
  return hessian_accumulate_impl(H, X_bf16, n_tokens, C, dev_info, stream, true);
}

extern "C" gptq_status_t gptq_hessian_accumulate_upper(float* H, const void* X_bf16, int64_t n_tokens, int C,
                                                       void* ws, size_t ws_bytes, int* dev_info, void* stream) {
  (void)ws; (void)ws_bytes;
  return hessian_accumulate_impl(H, X_bf16, n_tokens, C, dev_info, stream, false);
}

extern "C" gptq_status_t gptq_hessian_symmetrize(float* H, int C, void* stream) {
  using namespace gptq;
  if (!H || C <= 0 || C % 32 != 0 || !aligned_to(H, 16)) return GPTQ_ERR_INVALID_ARG;
  GPTQ_CUDA_TRY(launch_mirror_upper_to_lower(H, C, static_cast<cudaStream_t>(stream), false));
  return GPTQ_OK;
}
