// SIMT kernels of the rolling step: weight packing, conditioning embedding,
// adaRMSNorm, action in-projection, generic projection GEMM (fp32 FFMA; the
// exact path of fp32 mode), GeGLU, grouped-query attention, and the rolling
// tail (Euler update, release, shift, Philox append).
#include <algorithm>

#include "common.cuh"
#include "cond_cache.cuh"
#include "kernels.h"
#include "launch.h"
#include "noise.cuh"

namespace ravel {

// ============================================================================ packing

template <typename T>
__global__ void pack_transpose_kernel(const float* __restrict__ src, int K, int N, T* __restrict__ dst,
                                      int interleave64, int off) {
  __shared__ float tile[32][33];
  const int n0 = blockIdx.x * 32, k0 = blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int k = k0 + i, n = n0 + threadIdx.x;
    tile[i][threadIdx.x] = (k < K && n < N) ? src[(size_t)k * N + n] : 0.f;
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int n = n0 + i, k = k0 + threadIdx.x;
    if (n < N && k < K) {
      const size_t row = interleave64 ? (size_t)(n / 64) * 128 + off + (n % 64) : (size_t)n;
      dst[row * K + k] = from_f32<T>(tile[threadIdx.x][i]);
    }
  }
}

cudaError_t launch_pack_transpose(const float* src, int K, int N, void* dst, Dtype dt, int interleave64, int off,
                                  cudaStream_t st) {
  dim3 grid((N + 31) / 32, (K + 31) / 32), block(32, 8);
  if (dt == DT_BF16)
    pack_transpose_kernel<bf16><<<grid, block, 0, st>>>(src, K, N, (bf16*)dst, interleave64, off);
  else
    pack_transpose_kernel<float><<<grid, block, 0, st>>>(src, K, N, (float*)dst, interleave64, off);
  return cudaGetLastError();
}

template <typename T>
__global__ void convert_kernel(const float* __restrict__ src, size_t n, T* __restrict__ dst) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = from_f32<T>(src[i]);
}

cudaError_t launch_convert(const float* src, size_t n, void* dst, Dtype dt, cudaStream_t st) {
  const int blocks = (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  if (n == 0) return cudaSuccess;
  if (dt == DT_BF16)
    convert_kernel<bf16><<<blocks, 256, 0, st>>>(src, n, (bf16*)dst);
  else
    convert_kernel<float><<<blocks, 256, 0, st>>>(src, n, (float*)dst);
  return cudaGetLastError();
}

// ============================================================================ conditioning: cache check, embedding

// Sinusoidal embedding of a scalar (flow time or context offset): component
// i < D/2 is sin(x w_i), i >= D/2 is cos(x w_{i-D/2}), w_i = 2 pi / p_i with
// periods p_i geometric from 4e-3 to 4 (w_i precomputed in fp64).  x w
// reaches ~1.6e3 rad, where a float32 product would already be off by ~1e-4:
// the angle is formed and reduced modulo 2 pi in fp64, then sin / cos of the
// reduced angle (|a| <= pi) in fp32.  The first block checks the cache; the
// others, a row each, don't wait for its answer: a launch of its own behind the
// check cost more than rows that nobody reads (3 of a batch-1 step's 582 us).
template <typename T>
__global__ void __launch_bounds__(256) cond_embed_kernel(CondArgs a, int D, const double* __restrict__ omega,
                                                         T* __restrict__ E) {
  pdl_trigger();
  pdl_wait();
  if (blockIdx.x == 0) {
    cond_check(a);
    return;
  }
  const int r = blockIdx.x - 1, half = D / 2;
  const double x = r < a.H ? (double)a.slot_times[r] : (double)a.delta[r - a.H];
  for (int i = threadIdx.x; i < half; i += blockDim.x) {
    const double ang = x * omega[i];
    const double red = ang - 6.283185307179586 * rint(ang * 0.15915494309189535);
    float s, c;
    sincosf((float)red, &s, &c);
    E[(size_t)r * D + i] = from_f32<T>(s);
    E[(size_t)r * D + half + i] = from_f32<T>(c);
  }
}

cudaError_t launch_cond_embed(const CondArgs& a, int D, const double* omega, void* E, Dtype dt, cudaStream_t st) {
  const dim3 grid(1 + a.H + a.B);
  if (dt == DT_BF16)
    return launch_kernel(cond_embed_kernel<bf16>, grid, dim3(256), 0, st, 1, a, D, omega, (bf16*)E);
  return launch_kernel(cond_embed_kernel<float>, grid, dim3(256), 0, st, 1, a, D, omega, (float*)E);
}

// Copies the rows that cond_check listed (this step's fresh offset rows) into
// their cache slots.
__global__ void cond_commit_kernel(CondArgs a) {
  pdl_trigger();
  pdl_wait();
  const int n = a.cc->n_commit;
  for (int i = 0; i < n; ++i) {
    const float4* src = (const float4*)(a.modv + (size_t)a.commit[2 * i] * a.mod_ld);
    float4* dst = (float4*)(a.modv + (size_t)a.commit[2 * i + 1] * a.mod_ld);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < a.mod_ld / 4; c += gridDim.x * blockDim.x) dst[c] = src[c];
  }
}

cudaError_t launch_cond_commit(const CondArgs& a, cudaStream_t st) {
  return launch_kernel(cond_commit_kernel, dim3(64), dim3(256), 0, st, 1, a);
}

// four consecutive values as fp32 (16- / 8-byte aligned)
__device__ __forceinline__ float4 ld4(const float* p) { return *(const float4*)p; }
__device__ __forceinline__ float4 ld4(const bf16* p) {
  const uint2 u = *(const uint2*)p;
  const __nv_bfloat162 lo = *(const __nv_bfloat162*)&u.x, hi = *(const __nv_bfloat162*)&u.y;
  return make_float4(__low2float(lo), __high2float(lo), __low2float(hi), __high2float(hi));
}

// ============================================================================ GEMM (SIMT)

// 64x64 output tile, K step 32, 256 threads, 4x4 outputs per thread spread
// with stride 16 so that shared-memory reads are broadcast-friendly.
template <typename T, int EPI, typename TO>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const T* __restrict__ A, int lda, const T* __restrict__ W,
                                                        int ldw, int M, int N, int K, TO* __restrict__ out, int ldo,
                                                        const float* __restrict__ bias, const int* __restrict__ skip) {
  pdl_trigger();
  pdl_wait();
  if (skip && *skip) return;
  __shared__ float As[32][64 + 4];
  __shared__ float Ws[32][64 + 4];
  const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += 32) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int idx = threadIdx.x + 256 * i;
      const int r = idx >> 5, kk = idx & 31;
      const int m = m0 + r, n = n0 + r, k = k0 + kk;
      As[kk][r] = (m < M && k < K) ? to_f32(A[(size_t)m * lda + k]) : 0.f;
      Ws[kk][r] = (n < N && k < K) ? to_f32(W[(size_t)n * ldw + k]) : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < 32; ++kk) {
      float a[4], w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) w[j] = Ws[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], w[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty + 16 * i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx + 16 * j;
      if (n >= N) continue;
      float v = acc[i][j] + (bias ? bias[n] : 0.f);
      if (EPI == EPI_STORE_SILU) v = silu_f(v);
      if (EPI == EPI_ADD_F32)
        ((float*)out)[(size_t)m * ldo + n] += v;
      else
        out[(size_t)m * ldo + n] = from_f32<TO>(v);
    }
  }
}

// Few rows (the fp32 mode's small experts): a warp owns 8 rows x 2 columns, its
// lanes split K in float4 steps, so W streams once per 8 rows in 512-byte
// requests and the rows come from L1 (the 8 warps of a block read the same
// ones); the 16 sums then halve across the lanes.  Bound by load latency and
// the L1: at M 10, N 256, K 1024 the tile kernel above, whose only CTAs walk K in
// serial 32-wide steps with two barriers each, takes 75 us, this one 8.  The
// row loads of two steps go out together, and no branch on the row count stands
// between them: with one, each load waited for the one before (14 us; a tiny
// step 125 instead of 87).  EPI_GEGLU: a warp's two columns are a feature's gate and
// up, W rows in groups of 64 gates and their 64 ups (the separate launch and its
// fp32 round trip took a two-layer tiny step 4 of 69 us).
constexpr int RG_M = 8, RG_N = 2, RG_WARPS = 8;

template <int EPI, typename TO, int KS>
__global__ void __launch_bounds__(RG_WARPS * 32) gemm_rows_kernel(const float* __restrict__ A, int lda,
                                                                  const float* __restrict__ W, int ldw, int M, int N,
                                                                  int K, TO* __restrict__ out, int ldo,
                                                                  const float* __restrict__ bias,
                                                                  const int* __restrict__ skip) {
  pdl_trigger();
  const int warp = (threadIdx.x >> 5) / KS, part = (threadIdx.x >> 5) % KS, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * RG_M, n0 = (blockIdx.x * (RG_WARPS / KS) + warp) * RG_N;
  const int mr = min(RG_M, M - m0);
  // GeGLU: a gate row and its up row, 64 below it (N = 2 mlp, n0 / 2 the feature)
  const int f = min(n0, N - 1) / 2;
  const int nw = EPI == EPI_GEGLU ? f / 64 * 128 + f % 64 : min(n0, N - 1);
  const float* w0 = W + (size_t)nw * ldw;
  const float* w1 = W + (size_t)(EPI == EPI_GEGLU ? nw + 64 : min(n0 + 1, N - 1)) * ldw;
  const float* x[RG_M];   // rows past M repeat the last one; their sums are not stored
#pragma unroll
  for (int r = 0; r < RG_M; ++r) x[r] = A + (size_t)min(m0 + r, M - 1) * lda;
  pdl_wait();
  if (skip && *skip) return;
  float acc[RG_M][RG_N] = {};
#pragma unroll 2
  for (int k = 4 * (lane + 32 * part); k < K; k += 128 * KS) {
    const float4 wa = ld4(w0 + k), wb = ld4(w1 + k);
    float4 xr[RG_M];
#pragma unroll
    for (int r = 0; r < RG_M; ++r) xr[r] = ld4(x[r] + k);
#pragma unroll
    for (int r = 0; r < RG_M; ++r) {
      acc[r][0] = fmaf(xr[r].x, wa.x, fmaf(xr[r].y, wa.y, fmaf(xr[r].z, wa.z, fmaf(xr[r].w, wa.w, acc[r][0]))));
      acc[r][1] = fmaf(xr[r].x, wb.x, fmaf(xr[r].y, wb.y, fmaf(xr[r].z, wb.z, fmaf(xr[r].w, wb.w, acc[r][1]))));
    }
  }
  // lanes 2i and 2i + 1 end with the warp's sum i (row i / 2, column i % 2):
  // each step keeps half of the sums and adds the partner's half
  float v[RG_M * RG_N];
#pragma unroll
  for (int i = 0; i < RG_M * RG_N; ++i) v[i] = acc[i / RG_N][i % RG_N];
#pragma unroll
  for (int off = 16; off >= 2; off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < off / 2; ++i) {
      const float send = up ? v[i] : v[i + off / 2];
      const float keep = up ? v[i + off / 2] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  float t = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
  if (KS > 1) {
    __shared__ float sums[RG_WARPS / KS][KS][32];
    sums[warp][part][lane] = t;
    __syncthreads();
    if (part) return;
#pragma unroll
    for (int i = 1; i < KS; ++i) t += sums[warp][i][lane];
  }
  if (EPI == EPI_GEGLU) {
    const float up = __shfl_xor_sync(0xffffffffu, t, 2);
    if ((lane & 3) == 0 && (lane >> 2) < mr && n0 < N)
      out[(size_t)(m0 + (lane >> 2)) * ldo + n0 / 2] = from_f32<TO>(gelu_tanh_f(t) * up);
    return;
  }
  const int m = m0 + (lane >> 2), n = n0 + ((lane >> 1) & 1);
  if ((lane & 1) || (lane >> 2) >= mr || n >= N) return;
  t += bias ? bias[n] : 0.f;
  if (EPI == EPI_STORE_SILU) t = silu_f(t);
  TO* o = out + (size_t)m * ldo + n;
  if (EPI == EPI_ADD_F32) *(float*)o += t;
  else *o = from_f32<TO>(t);
}

// Four warps share a column pair's K (an interleaved quarter each, summed through
// shared memory) where that many more blocks still fit the SMs about twice and a
// quarter is at least one step of a warp: M 10, N 256, K 1024 takes 4.1 us instead of
// 8.2.
constexpr int RG_KS = 4, RG_SPLIT_COLS = 1024;

// The row kernel re-reads W for every 8 rows (from L2), the tile kernel pads rows
// to 64 and takes K x 72 ns however few its tiles are: rows while the products
// are few or the tile kernel's rows mostly padding.  Measured per call, rows and
// tiles: M 64 x N 2560 x K 1024 29 and 76 us, 192 x 2560 x 1024 72 and 77, 192 x 3000
// x 1024 84 and 77, 128 x 8192 x 1024 125 and 106; 96 x 4096 x 4096 352 and 450, 192 x 4096 x 4096 605 and 457; at K
// 256, 192 x 2048 23 and 26, 256 x 2048 29 and 26; 24 x 75776 x 1024 306 and 394, 32 x
// 75776 x 1024 406 and 394.  GeGLU saves a launch and its fp32 round trip on top:
// steps of four 1024-wide layers, 100 rows 1239 and 1493 us, 200 rows 2169 and 1951;
// of two 256-wide ones, 250 rows 252 and 277.
bool rows_gemm_supported(const GemmArgs& g) {
  const bool glu = g.epi == EPI_GEGLU;
  const int limit = g.K < 512 ? (glu ? 18 : 13) : glu && g.K < 2048 ? 26 : 16;   // in 2^15 products
  return (g.M <= 24 || (g.M <= 256 && (int64_t)g.M * g.N < limit << 15)) && g.K % 4 == 0 && g.lda % 4 == 0 &&
         g.ldw % 4 == 0 && (((uintptr_t)g.A | (uintptr_t)g.W) & 15u) == 0;
}

template <int EPI, typename TO>
static cudaError_t launch_gemm_rows(const GemmArgs& g, cudaStream_t st) {
  const bool split = g.K >= 512 && (int64_t)g.N * ((g.M + RG_M - 1) / RG_M) <= RG_SPLIT_COLS;
  const int cols = RG_WARPS * RG_N / (split ? RG_KS : 1);
  const dim3 grid((g.N + cols - 1) / cols, (g.M + RG_M - 1) / RG_M);
  return launch_kernel(split ? gemm_rows_kernel<EPI, TO, RG_KS> : gemm_rows_kernel<EPI, TO, 1>, grid, dim3(RG_WARPS * 32),
                       0, st, 1, (const float*)g.A, g.lda, (const float*)g.W, g.ldw, g.M, g.N, g.K, (TO*)g.out, g.ldo,
                       g.bias, g.skip);
}

static cudaError_t gemm_rows_dispatch(const GemmArgs& g, cudaStream_t st) {
  if (g.epi == EPI_ADD_F32) return launch_gemm_rows<EPI_ADD_F32, float>(g, st);
  if (g.epi == EPI_GEGLU) return launch_gemm_rows<EPI_GEGLU, float>(g, st);
  if (g.out_dt == DT_BF16)
    return g.epi == EPI_STORE_SILU ? launch_gemm_rows<EPI_STORE_SILU, bf16>(g, st) : launch_gemm_rows<EPI_STORE, bf16>(g, st);
  return g.epi == EPI_STORE_SILU ? launch_gemm_rows<EPI_STORE_SILU, float>(g, st) : launch_gemm_rows<EPI_STORE, float>(g, st);
}

template <typename T>
static cudaError_t gemm_simt_dispatch(const GemmArgs& g, cudaStream_t st) {
  dim3 grid((g.N + 63) / 64, (g.M + 63) / 64);
  const T* A = (const T*)g.A;
  const T* W = (const T*)g.W;
  if (g.epi == EPI_ADD_F32) {
    launch_kernel(gemm_simt_kernel<T, EPI_ADD_F32, float>, grid, dim3(256), 0, st, 1, A, g.lda, W, g.ldw, g.M, g.N, g.K, (float*)g.out,
                                                                 g.ldo, g.bias, g.skip);
  } else if (g.out_dt == DT_BF16) {
    if (g.epi == EPI_STORE_SILU)
      launch_kernel(gemm_simt_kernel<T, EPI_STORE_SILU, bf16>, grid, dim3(256), 0, st, 1, A, g.lda, W, g.ldw, g.M, g.N, g.K,
                                                                     (bf16*)g.out, g.ldo, g.bias, g.skip);
    else
      launch_kernel(gemm_simt_kernel<T, EPI_STORE, bf16>, grid, dim3(256), 0, st, 1, A, g.lda, W, g.ldw, g.M, g.N, g.K, (bf16*)g.out,
                                                                g.ldo, g.bias, g.skip);
  } else {
    if (g.epi == EPI_STORE_SILU)
      launch_kernel(gemm_simt_kernel<T, EPI_STORE_SILU, float>, grid, dim3(256), 0, st, 1, A, g.lda, W, g.ldw, g.M, g.N, g.K,
                                                                      (float*)g.out, g.ldo, g.bias, g.skip);
    else
      launch_kernel(gemm_simt_kernel<T, EPI_STORE, float>, grid, dim3(256), 0, st, 1, A, g.lda, W, g.ldw, g.M, g.N, g.K, (float*)g.out,
                                                                 g.ldo, g.bias, g.skip);
  }
  return cudaGetLastError();
}

cudaError_t launch_gemm_simt(const GemmArgs& g, Dtype dt, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  if (dt == DT_F32 && rows_gemm_supported(g)) return gemm_rows_dispatch(g, st);
  return dt == DT_BF16 ? gemm_simt_dispatch<bf16>(g, st) : gemm_simt_dispatch<float>(g, st);
}

// ============================================================================ adaRMSNorm

// (t_stride as in NormArgs)
__device__ __forceinline__ int time_row(int t_stride, int b, int j) {
  return t_stride < 0 ? ~t_stride : b * t_stride + j;
}

__device__ __forceinline__ float4 add3(float4 a, float4 b, float4 c) {
  return make_float4(a.x + b.x + c.x, a.y + b.y + c.y, a.z + b.z + c.z, a.w + b.w + c.w);
}
__device__ __forceinline__ void st4(float* p, float4 v) { *(float4*)p = v; }
__device__ __forceinline__ void st4(bf16* p, float4 v) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  uint2 u;
  u.x = *(uint32_t*)&lo;
  u.y = *(uint32_t*)&hi;
  *(uint2*)p = u;
}

__device__ __forceinline__ float4 add2(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// adaRMSNorm over a block of rows of one robot (Sec. 3.1, Eq. 2):
//   action row (b, j):  y = x * rsqrt(mean(x^2) + eps) * (1 + scale) + shift,
//                       (scale, shift) = M_t[j] + M_delta[b] + bias  (the
//                       modulation is linear in the two embeddings)
//   FOP row (b, f):     y = z * rsqrt(mean(z^2) + eps) * (1 + gamma)
// A thread owns columns 4*tid + 1024*g (g < G) of every row of the block, so
// the per-robot part M_delta[b] + bias (or gamma) is read once per block and
// kept in registers; rows go through one at a time with one barrier each
// (the row sums are reduced through a double-buffered table).  Few rows per
// block: the row's loads are the block's critical path, and spreading the
// rows over more blocks (one each when they fit the SMs) beat batching four
// rows per round trip.  ONE: one time row for all slots (a select at run time
// cost a tiny fp32 step 1.8 of 64 us, a batch-1 step 1.1 of 577).
template <typename T, int G, bool ONE>
__global__ void __launch_bounds__(256) ada_norm_kernel(NormArgs a, int rb_act, int nb_act, int rb_fop, int nb_fop) {
  constexpr int R = 1;
  __shared__ float red[2][R][8];
  pdl_trigger();
  const int D = a.D, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int blk = blockIdx.x;
  const bool act = blk < a.B * nb_act;
  int b, j0, j1;
  if (act) {
    b = blk / nb_act;
    j0 = (blk % nb_act) * rb_act;
    j1 = min(a.H, j0 + rb_act);
  } else {
    blk -= a.B * nb_act;
    b = blk / nb_fop;
    j0 = (blk % nb_fop) * rb_fop;
    j1 = min(a.F, j0 + rb_fop);
  }
  float4 csc[G], csh[G];   // action: bias (+ M_delta[b] after the wait); FOP: gamma
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int c = 4 * threadIdx.x + 1024 * g;
    csc[g] = csh[g] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c < D) {   // weights: independent of the earlier kernels
      if (act && !a.act_gain) {
        csc[g] = ld4(a.mod_b + a.off + c);
        csh[g] = ld4(a.mod_b + a.off + D + c);
      } else {
        csc[g] = ld4(act ? a.act_gain + c : a.gamma + c);
      }
    }
  }
  pdl_wait();
  const bool modulated = act && !a.act_gain;   // action rows with adaLN modulation
  const float* md = modulated ? a.modv + (size_t)(a.drow ? a.drow[b] : a.H + b) * a.mod_ld + a.off : nullptr;
  int buf = 0;
  for (int j = j0; j < j1; j += R, buf ^= 1) {
    float4 xv[R][G], ts[R][G], th[R][G], dsc[G], dsh[G];
    float ss[R];
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
      ss[rr] = 0.f;
      const int jj = j + rr;
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const int c = 4 * threadIdx.x + 1024 * g;
        xv[rr][g] = ts[rr][g] = th[rr][g] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (jj < j1 && c < D) {
          if (act) {
            xv[rr][g] = ld4(a.x + (size_t)(b * a.H + jj) * D + c);
            if (modulated) {
              const float* mt = a.modv + (size_t)(ONE ? ~a.t_stride : b * a.t_stride + jj) * a.mod_ld + a.off;
              ts[rr][g] = ld4(mt + c);
              th[rr][g] = ld4(mt + D + c);
            }
          } else {
            xv[rr][g] = ld4((const T*)a.fop + (size_t)(b * a.F + jj) * D + c);
          }
        }
      }
    }
    // M_delta[b] after the row's own loads: its address waits for drow[b], and a
    // warp issues in order (before them, the row waited for two round trips:
    // 36 to 47 launches of a step, 6 us at batch 1, 17 on the wide expert)
    const bool first = modulated && j == j0;
    if (first) {
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const int c = 4 * threadIdx.x + 1024 * g;
        if (c < D) {
          dsc[g] = ld4(md + c);
          dsh[g] = ld4(md + D + c);
        }
      }
    }
#pragma unroll
    for (int rr = 0; rr < R; ++rr)
#pragma unroll
      for (int g = 0; g < G; ++g)
        ss[rr] += xv[rr][g].x * xv[rr][g].x + xv[rr][g].y * xv[rr][g].y + xv[rr][g].z * xv[rr][g].z +
                  xv[rr][g].w * xv[rr][g].w;
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ss[rr] += __shfl_xor_sync(0xffffffffu, ss[rr], o);
      if (lane == 0) red[buf][rr][warp] = ss[rr];
    }
    __syncthreads();
    if (first) {
#pragma unroll
      for (int g = 0; g < G; ++g)
        if (4 * (int)threadIdx.x + 1024 * g < D) {
          csc[g] = add2(csc[g], dsc[g]);
          csh[g] = add2(csh[g], dsh[g]);
        }
    }
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
      const int jj = j + rr;
      float tot = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) tot += red[buf][rr][w];
      const float inv = rsqrtf(tot / (float)D + 1e-6f);
      if (jj >= j1) continue;
      T* Y = (T*)a.Y + ((size_t)b * a.row_pitch + (act ? jj : a.H + jj)) * D;
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const int c = 4 * threadIdx.x + 1024 * g;
        if (c >= D) continue;
        const float4 x = xv[rr][g];
        if (modulated) {
          const float4 sc = add2(csc[g], ts[rr][g]), sh = add2(csh[g], th[rr][g]);
          st4(Y + c, make_float4(x.x * inv * (1.f + sc.x) + sh.x, x.y * inv * (1.f + sc.y) + sh.y,
                                 x.z * inv * (1.f + sc.z) + sh.z, x.w * inv * (1.f + sc.w) + sh.w));
        } else {
          const float4 gm = csc[g];
          st4(Y + c, make_float4(x.x * inv * (1.f + gm.x), x.y * inv * (1.f + gm.y), x.z * inv * (1.f + gm.z),
                                 x.w * inv * (1.f + gm.w)));
        }
      }
    }
  }
}

// The same for rows in numbers: a block takes RB robots x RJ slots (RB RJ = 4), so
// that each modulation row it reads serves several rows: a row then costs 14
// KB of L2 traffic at width 1024 (its own 6 KB, half a slot's and half a
// robot's modulation, a quarter of the bias) instead of 19 to 28, which is
// what bounds the norm once the rows fill the SMs.  Every load is issued
// before the one barrier.  FOP rows go four to a block.  The arithmetic is the
// row kernel's, operation for operation.  (64 robots x 50 slots, width 1024, 35
// launches: step 2701 -> 2682 us; 1056 rows: 1288 -> 1264.)
template <typename T, int RB, int RJ>
__global__ void __launch_bounds__(256) ada_norm_tile_kernel(NormArgs a, int nb_b, int nb_j) {
  constexpr int R = RB * RJ;
  __shared__ float red[R][8];
  pdl_trigger();
  const int D = a.D, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, c = 4 * threadIdx.x;
  const bool on = c < D;
  const bool act = (int)blockIdx.x < nb_b * nb_j;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const int b0 = act ? (blockIdx.x / nb_j) * RB : 0, j0 = act ? (blockIdx.x % nb_j) * RJ : 0;
  const int f0 = act ? 0 : (blockIdx.x - nb_b * nb_j) * R;   // first FOP row (of B F)
  float4 bsc = zero, bsh = zero;   // weights: independent of the earlier kernels
  if (on) {
    bsc = ld4(act ? a.mod_b + a.off + c : a.gamma + c);
    if (act) bsh = ld4(a.mod_b + a.off + D + c);
  }
  pdl_wait();
  float4 x[R], dsc[RB], dsh[RB], tsc[RJ], tsh[RJ];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    x[r] = zero;
    if (!on) continue;
    if (act) {
      const int b = b0 + r / RJ, j = j0 + r % RJ;
      if (b < a.B && j < a.H) x[r] = ld4(a.x + (size_t)(b * a.H + j) * D + c);
    } else if (f0 + r < a.B * a.F) {
      x[r] = ld4((const T*)a.fop + (size_t)(f0 + r) * D + c);
    }
  }
  if (act && on) {
#pragma unroll
    for (int i = 0; i < RJ; ++i) {
      const float* mt = a.modv + (size_t)time_row(a.t_stride, b0, min(j0 + i, a.H - 1)) * a.mod_ld + a.off;
      tsc[i] = ld4(mt + c);
      tsh[i] = ld4(mt + D + c);
    }
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int b = min(b0 + i, a.B - 1);
      const float* md = a.modv + (size_t)(a.drow ? a.drow[b] : a.H + b) * a.mod_ld + a.off;
      dsc[i] = ld4(md + c);
      dsh[i] = ld4(md + D + c);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float ss = warp_sum(x[r].x * x[r].x + x[r].y * x[r].y + x[r].z * x[r].z + x[r].w * x[r].w);
    if (lane == 0) red[r][warp] = ss;
  }
  __syncthreads();
  if (!on) return;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += red[r][w];
    const float inv = rsqrtf(tot / (float)D + 1e-6f);
    const float4 v = x[r];
    if (act) {
      const int b = b0 + r / RJ, j = j0 + r % RJ;
      if (b >= a.B || j >= a.H) continue;
      const float4 sc = add2(add2(bsc, dsc[r / RJ]), tsc[r % RJ]), sh = add2(add2(bsh, dsh[r / RJ]), tsh[r % RJ]);
      st4((T*)a.Y + ((size_t)b * a.row_pitch + j) * D + c,
          make_float4(v.x * inv * (1.f + sc.x) + sh.x, v.y * inv * (1.f + sc.y) + sh.y,
                      v.z * inv * (1.f + sc.z) + sh.z, v.w * inv * (1.f + sc.w) + sh.w));
    } else if (f0 + r < a.B * a.F) {
      const int b = (f0 + r) / a.F, f = (f0 + r) % a.F;
      st4((T*)a.Y + ((size_t)b * a.row_pitch + a.H + f) * D + c,
          make_float4(v.x * inv * (1.f + bsc.x), v.y * inv * (1.f + bsc.y), v.z * inv * (1.f + bsc.z),
                      v.w * inv * (1.f + bsc.w)));
    }
  }
}

namespace {
int g_norm_sms = 0;
}

template <typename T>
cudaError_t launch_ada_norm_t(const NormArgs& a, cudaStream_t st) {
  if (!g_norm_sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&g_norm_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || g_norm_sms < 1)
      g_norm_sms = 132;
  }
  const int G = (a.D + 1023) / 1024;
  const int R = 1;
  // rows per block: as few as fill up to 8 resident blocks of 256 threads per
  // SM (one row each when the rows fit)
  const int nf = a.fop ? a.F : 0;
  const int total = a.B * (a.H + nf);
  // modulated rows of up to 1024 features, from where the row kernel's blocks no
  // longer fit the SMs at once (five each)
  if (a.D <= 1024 && !a.act_gain && a.H > 0 && total > 5 * g_norm_sms) {
    NormArgs b = a;
    b.F = nf;
    const int fop_blocks = (a.B * nf + 3) / 4;
    if (a.t_stride <= 0) {
      const int nb = (a.B + 1) / 2, nj = (a.H + 1) / 2;
      return launch_kernel(ada_norm_tile_kernel<T, 2, 2>, dim3(nb * nj + fop_blocks), dim3(256), 0, st, 1, b, nb, nj);
    }
    const int nj = (a.H + 3) / 4;   // a schedule per robot: slots of one robot
    return launch_kernel(ada_norm_tile_kernel<T, 1, 4>, dim3(a.B * nj + fop_blocks), dim3(256), 0, st, 1, b, a.B, nj);
  }
  int rb_all = (total + 8 * g_norm_sms - 1) / (8 * g_norm_sms);
  rb_all = (rb_all + R - 1) / R * R;
  auto rows_per_block = [&](int rows_per_robot) { return std::max(R, std::min(rb_all, rows_per_robot)); };
  const int rb_act = rows_per_block(a.H), nb_act = (a.H + rb_act - 1) / rb_act;
  const int rb_fop = nf ? rows_per_block(nf) : 1, nb_fop = nf ? (nf + rb_fop - 1) / rb_fop : 0;
  const int blocks = a.B * (nb_act + nb_fop);
  if (blocks <= 0) return cudaSuccess;
  NormArgs b = a;
  b.F = nf;
#define RAVEL_NORM(G)                                                                                            \
  return launch_kernel(a.t_stride < 0 ? ada_norm_kernel<T, G, true> : ada_norm_kernel<T, G, false>, dim3(blocks), \
                       dim3(256), 0, st, 1, b, rb_act, nb_act, rb_fop, nb_fop)
  switch (G) {
    case 1: RAVEL_NORM(1);
    case 2: RAVEL_NORM(2);
    case 3: RAVEL_NORM(3);
    default: RAVEL_NORM(4);
  }
#undef RAVEL_NORM
}

cudaError_t launch_ada_norm(const NormArgs& a, Dtype dt, cudaStream_t st) {
  if (a.D <= 0 || a.D > 4096 || a.D % 4) return cudaErrorInvalidValue;
  return dt == DT_BF16 ? launch_ada_norm_t<bf16>(a, st) : launch_ada_norm_t<float>(a, st);
}

// ============================================================================ in-proj

// The in-projection reads what the step starts from (buffer, slot times, state,
// weights) and x's last readers were the step before, while the launches in
// front of it, back to the step's first one, which waits for all earlier work,
// are the conditioning: it runs beside them, and waits for them only where it
// needs the modulation (or at its end, for the kernels that follow).
__global__ void in_proj_kernel(const float* __restrict__ buf, int A, int D, const float* __restrict__ in_w,
                               const float* __restrict__ in_b, float* __restrict__ x, const float* __restrict__ state,
                               const float* __restrict__ rel_mask, const float* __restrict__ slot_times, int H,
                               int t_stride) {
  pdl_trigger();
  extern __shared__ float arow[];   // the action row of this slot
  const int r = blockIdx.y;
  for (int i = threadIdx.x; i < A; i += blockDim.x) {
    float a = buf[(size_t)r * A + i];
    if (state) {   // relative coordinates of the expert: a - (1 - t_j) m s_b
      const int b = r / H, j = r % H;
      a = __fsub_rn(a, __fmul_rn(__fsub_rn(1.f, slot_times[b * t_stride + j]),
                                 __fmul_rn(rel_mask[i], state[(size_t)b * A + i])));
    }
    arow[i] = a;
  }
  __syncthreads();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < D) {
    float acc = in_b[c];
    for (int i = 0; i < A; ++i) acc = fmaf(arow[i], in_w[(size_t)i * D + c], acc);
    x[(size_t)r * D + c] = acc;
  }
  pdl_wait();   // (the kernels after this one wait for it alone)
}

cudaError_t launch_in_proj(const float* buf, int BH, int A, int D, const float* in_w, const float* in_b, float* x,
                           cudaStream_t st, const float* state, const float* rel_mask, const float* slot_times, int H,
                           int t_stride) {
  if (BH <= 0) return cudaSuccess;
  return launch_kernel(in_proj_kernel, dim3((D + 255) / 256, BH), dim3(256), A * sizeof(float), st, 1, buf, A, D,
                       in_w, in_b, x, state, rel_mask, slot_times, H, t_stride);
}

// The in-projection of whole rows with the first layer's adaRMSNorm: a block
// takes R consecutive slots of one robot (projected into x, fp32, then
// normalised with their modulation into Y) or R FOP rows (normalised with their
// gain).  A thread owns features 4 tid + 1024 g, so a row of W_in is one
// 16-byte load per thread that serves R slots, eight of them in flight: one
// slot per block and a load per feature re-read the 128 KB of W_in for every
// slot (64 robots x 50 slots: step 2682 -> 2662 us) and waited for 32 loads in
// turn (4 robots: 900 -> 891 us).  All but the modulation runs before the wait
// (see above; where the modulation GEMM runs in front of it: four robots on
// schedules of their own 999 -> 992 us, ten denoising passes 6068 -> 6029).
template <typename T, int R, int G>
__global__ void __launch_bounds__(256) in_proj_norm_kernel(const float* __restrict__ buf, int A, int D,
                                                           const float* __restrict__ in_w,
                                                           const float* __restrict__ in_b, float* __restrict__ x,
                                                           const float* __restrict__ state,
                                                           const float* __restrict__ rel_mask,
                                                           const float* __restrict__ slot_times, RowNorm rn, int nj) {
  extern __shared__ float arow[];   // [R][A] the action rows of these slots
  __shared__ float red[R][8];
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool act = (int)blockIdx.x < rn.B * nj;
  const int b = act ? blockIdx.x / nj : 0, j0 = act ? (blockIdx.x % nj) * R : 0;
  const int f0 = act ? 0 : (blockIdx.x - rn.B * nj) * R;   // first FOP row (of B F)
  float4 v[R][G];
  if (act) {
    for (int i = threadIdx.x; i < R * A; i += 256) {
      const int j = j0 + i / A, d = i % A;
      float a = 0.f;
      if (j < rn.H) {
        a = buf[(size_t)(b * rn.H + j) * A + d];
        if (state)   // relative coordinates of the expert: a - (1 - t_j) m s_b
          a = __fsub_rn(a, __fmul_rn(__fsub_rn(1.f, slot_times[b * rn.t_stride + j]),
                                     __fmul_rn(rel_mask[d], state[(size_t)b * A + d])));
      }
      arow[i] = a;
    }
    __syncthreads();
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int c = 4 * threadIdx.x + 1024 * g;
      const float4 bias = c < D ? ld4(in_b + c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int r = 0; r < R; ++r) v[r][g] = bias;
      if (c >= D) continue;
#pragma unroll 8
      for (int i = 0; i < A; ++i) {
        const float4 w = ld4(in_w + (size_t)i * D + c);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const float a = arow[r * A + i];
          v[r][g] = make_float4(fmaf(a, w.x, v[r][g].x), fmaf(a, w.y, v[r][g].y), fmaf(a, w.z, v[r][g].z),
                                fmaf(a, w.w, v[r][g].w));
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (j0 + r < rn.H) st4(x + (size_t)(b * rn.H + j0 + r) * D + c, v[r][g]);
    }
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const int c = 4 * threadIdx.x + 1024 * g;
        v[r][g] = (c < D && f0 + r < rn.B * rn.F) ? ld4((const T*)rn.fop + (size_t)(f0 + r) * D + c)
                                                  : make_float4(0.f, 0.f, 0.f, 0.f);
      }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float ss = 0.f;
#pragma unroll
    for (int g = 0; g < G; ++g)
      ss += v[r][g].x * v[r][g].x + v[r][g].y * v[r][g].y + v[r][g].z * v[r][g].z + v[r][g].w * v[r][g].w;
    ss = warp_sum(ss);
    if (lane == 0) red[r][warp] = ss;
  }
  __syncthreads();
  pdl_wait();   // the modulation
  const float* md = rn.modv + (size_t)(act ? (rn.drow ? rn.drow[b] : rn.H + b) : 0) * rn.mod_ld + rn.off;
  const float* mb = rn.mod_b + rn.off;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int c = 4 * threadIdx.x + 1024 * g;
    if (c >= D) continue;
    float4 dsc, dsh, bsc, bsh;
    if (act) {
      dsc = ld4(md + c);
      dsh = ld4(md + D + c);
      bsc = ld4(mb + c);
      bsh = ld4(mb + D + c);
    } else {
      bsc = ld4(rn.gamma + c);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float tot = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) tot += red[r][w];
      const float inv = rsqrtf(tot / (float)D + 1e-6f);
      const float4 q = v[r][g];
      if (act) {
        if (j0 + r >= rn.H) continue;
        const float* mt = rn.modv + (size_t)time_row(rn.t_stride, b, j0 + r) * rn.mod_ld + rn.off;
        const float4 sc = add3(ld4(mt + c), dsc, bsc), sh = add3(ld4(mt + D + c), dsh, bsh);
        st4((T*)rn.Y + ((size_t)b * rn.row_pitch + j0 + r) * D + c,
            make_float4(q.x * inv * (1.f + sc.x) + sh.x, q.y * inv * (1.f + sc.y) + sh.y,
                        q.z * inv * (1.f + sc.z) + sh.z, q.w * inv * (1.f + sc.w) + sh.w));
      } else if (f0 + r < rn.B * rn.F) {
        const int fb = (f0 + r) / rn.F, f = (f0 + r) % rn.F;
        st4((T*)rn.Y + ((size_t)fb * rn.row_pitch + rn.H + f) * D + c,
            make_float4(q.x * inv * (1.f + bsc.x), q.y * inv * (1.f + bsc.y), q.z * inv * (1.f + bsc.z),
                        q.w * inv * (1.f + bsc.w)));
      }
    }
  }
}

template <typename T, int R, int G>
static cudaError_t launch_in_proj_norm_t(const float* buf, int A, int D, const float* in_w, const float* in_b,
                                         float* x, const float* state, const float* rel_mask, const float* slot_times,
                                         const RowNorm& rn, cudaStream_t st) {
  const int nj = (rn.H + R - 1) / R, blocks = rn.B * nj + (rn.fop ? (rn.B * rn.F + R - 1) / R : 0);
  return launch_kernel(in_proj_norm_kernel<T, R, G>, dim3(blocks), dim3(256), (size_t)R * A * sizeof(float), st, 1,
                       buf, A, D, in_w, in_b, x, state, rel_mask, slot_times, rn, nj);
}

cudaError_t launch_in_proj_norm(const float* buf, int A, int D, const float* in_w, const float* in_b, float* x,
                                const float* state, const float* rel_mask, const float* slot_times, const RowNorm& rn,
                                Dtype dt, int num_sms, cudaStream_t st) {
  const int rows = rn.B * rn.H + (rn.fop ? rn.B * rn.F : 0);
  if (D > 4096 || D % 4) return cudaErrorInvalidValue;
  if (rows <= 0) return cudaSuccess;
  if (dt != DT_BF16) return cudaErrorNotSupported;   // (the fp32 step runs the two kernels)
#define RAVEL_IPN(R, G) \
  return launch_in_proj_norm_t<bf16, R, G>(buf, A, D, in_w, in_b, x, state, rel_mask, slot_times, rn, st)
  if (D > 2048) RAVEL_IPN(1, 4);
  if (D > 1024) RAVEL_IPN(1, 2);
  // one slot per block while they leave SMs idle, then four, or eight (whose
  // actions must fit the block's shared memory)
  if (rows <= 2 * num_sms || A > 1024) RAVEL_IPN(1, 1);
  if (rows <= 8 * num_sms) RAVEL_IPN(4, 1);
  RAVEL_IPN(8, 1);
#undef RAVEL_IPN
}

__global__ void noop_kernel() {}

cudaError_t launch_noop(cudaStream_t st) { return launch_kernel(noop_kernel, dim3(1), dim3(1), 0, st, 1); }

// ============================================================================ GeGLU

template <typename T>
__global__ void geglu_kernel(const float* __restrict__ GU, int M, int Fm, T* __restrict__ Hm) {
  pdl_trigger();
  pdl_wait();
  const size_t total = (size_t)M * Fm;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(i / Fm), f = (int)(i % Fm);
    const size_t base = (size_t)m * 2 * Fm + (size_t)(f / 64) * 128 + (f % 64);
    Hm[i] = from_f32<T>(gelu_tanh_f(GU[base]) * GU[base + 64]);
  }
}

cudaError_t launch_geglu(const float* GU, int M, int Fm, void* Hm, Dtype dt, cudaStream_t st) {
  const size_t total = (size_t)M * Fm;
  if (!total) return cudaSuccess;
  const int blocks = (int)((total + 255) / 256 < 8192 ? (total + 255) / 256 : 8192);
  if (dt == DT_BF16) return launch_kernel(geglu_kernel<bf16>, dim3(blocks), dim3(256), 0, st, 1, GU, M, Fm, (bf16*)Hm);
  return launch_kernel(geglu_kernel<float>, dim3(blocks), dim3(256), 0, st, 1, GU, M, Fm, (float*)Hm);
}

// ============================================================================ attention (SIMT)

// One CTA per (robot b, KV head g, tile of QT query rows).  Query row r of a
// (b, g) pair is slot j = r / G of query head g*G + r % G.  Keys are visited
// in chunks of KT: [0, P) the active context's prefix, [P, P+F) the FOP
// tokens, [P+F, P+F+H) the action slots; online softmax in fp32.  Eight
// threads copy a key's K and V row in float4 steps, into registers while the
// chunk before is worked on; rows of Q and K are padded by four floats, so that
// the 16-byte reads of a score (8 keys per phase) fall into distinct banks.
// Bound by a few blocks' shared-memory reads, hence 16-byte ones throughout: 40
// query rows, 78 keys and head dim 64 take 6 us; with scalar reads of the
// probabilities and V, and each chunk's loads in front of its work, 10; with
// unpadded rows (16 keys of a request in one bank) and an integer division for
// every element's row, 40.  NC: 32-column groups of the head dim, rounded up to
// 2, 4 or 8.
constexpr int ATT_QT = 16, ATT_KT = 32, ATT_THREADS = 256;

__device__ __forceinline__ void fma4(float4& d, float p, float4 v) {
  d = make_float4(fmaf(p, v.x, d.x), fmaf(p, v.y, d.y), fmaf(p, v.z, d.z), fmaf(p, v.w, d.w));
}

template <typename T, int NC>
__global__ void __launch_bounds__(ATT_THREADS, 2) attention_simt_kernel(AttnArgs a) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ float sm[];
  const int hd = a.hd, ld = hd + 4;
  float* Qs = sm;                      // [QT][hd + 4]
  float* Ks = Qs + ATT_QT * ld;        // [KT][hd + 4]
  float* Vs = Ks + ATT_KT * ld;        // [KT][hd]
  float* Ss = Vs + ATT_KT * hd;        // [QT][KT]
  const int bg = blockIdx.x;
  const int b = bg / a.Hkv, g = bg % a.Hkv;
  const int G = a.Hq / a.Hkv;
  const int nrows = a.H * G;
  const int r0 = blockIdx.y * ATT_QT;
  const int slot = a.ctx_state[2 * b];       // this robot's active context
  const int P = a.ctx_state[2 * b + 1];
  if (P < 0 || P > a.Pmax) {
    if (threadIdx.x == 0) raise_error(a.err, ERR_PREFIX_LEN);
    return;
  }
  const T* qkv = (const T*)a.qkv;
  const size_t ctx_off = ((((size_t)a.layer * a.Bmax + b) * a.Hkv + g) * (size_t)a.Pmax) * hd;
  const T* pk = (const T*)(slot ? a.ctx_k1 : a.ctx_k0) + ctx_off;
  const T* pv = (const T*)(slot ? a.ctx_v1 : a.ctx_v0) + ctx_off;
  const int kofs = a.Hq * hd + g * hd, vofs = (a.Hq + a.Hkv) * hd + g * hd;
  const int nk = P + a.F + a.H;
  const int rpr = a.H + a.F;   // QKV rows per robot: H action slots, then F FOP tokens
  const float scale = rsqrtf((float)hd);
  // 16 threads per query row: its Q, its scores (keys qlane, qlane + 16), its
  // softmax and its output columns 4 qlane + 64 i (four each)
  const int qrow = threadIdx.x >> 4, qlane = threadIdx.x & 15;
  const int r = r0 + qrow, j = r < nrows ? r / G : -1, h = g * G + r % G;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int c = 4 * qlane; c < hd; c += 64) {
    float4 v = zero;
    if (r < nrows) v = ld4(qkv + (size_t)(b * rpr + j) * a.ld_qkv + h * hd + c);
    st4(Qs + qrow * ld + c, make_float4(v.x * scale, v.y * scale, v.z * scale, v.w * scale));
  }
  // the K and V row of key k0 + threadIdx.x / 8: columns 4 (threadIdx.x % 8) + 32 i
  const int kk = threadIdx.x >> 3, kc = 4 * (threadIdx.x & 7);
  float4 kv[NC], vv[NC];
  auto fetch = [&](int key) {
    const T *kr = nullptr, *vr = nullptr;
    if (key < P) {
      kr = pk + (size_t)key * hd;
      vr = pv + (size_t)key * hd;
    } else if (key < nk) {   // the step's own rows: FOP tokens, then slots
      const int row = key < P + a.F ? a.H + (key - P) : key - P - a.F;
      kr = qkv + (size_t)(b * rpr + row) * a.ld_qkv + kofs;
      vr = qkv + (size_t)(b * rpr + row) * a.ld_qkv + vofs;
    }
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      kv[i] = vv[i] = zero;
      if (kr && kc + 32 * i < hd) {
        kv[i] = ld4(kr + kc + 32 * i);
        vv[i] = ld4(vr + kc + 32 * i);
      }
    }
  };
  float m_run = -INFINITY, l_run = 0.f;
  float4 acc[NC / 2];
#pragma unroll
  for (int i = 0; i < NC / 2; ++i) acc[i] = zero;

  fetch(kk);
  for (int k0 = 0; k0 < nk; k0 += ATT_KT) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      if (kc + 32 * i < hd) {
        st4(Ks + kk * ld + kc + 32 * i, kv[i]);
        st4(Vs + kk * hd + kc + 32 * i, vv[i]);
      }
    }
    __syncthreads();
    fetch(k0 + ATT_KT + kk);
    float4 d[2] = {zero, zero};
#pragma unroll 4
    for (int c = 0; c < hd; c += 4) {
      const float4 q = ld4(Qs + qrow * ld + c);
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const float4 k = ld4(Ks + (qlane + 16 * t) * ld + c);
        d[t].x = fmaf(q.x, k.x, d[t].x);
        d[t].y = fmaf(q.y, k.y, d[t].y);
        d[t].z = fmaf(q.z, k.z, d[t].z);
        d[t].w = fmaf(q.w, k.w, d[t].w);
      }
    }
    float s[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int key = k0 + qlane + 16 * t;
      bool vis = key < nk;
      if (a.mask_mode == 1 && key >= P + a.F && key < nk) vis = vis && (key - P - a.F == j);
      s[t] = vis ? (d[t].x + d[t].y) + (d[t].z + d[t].w) : -INFINITY;
    }
    float cmax = fmaxf(s[0], s[1]);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) cmax = fmaxf(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
    const float m_new = fmaxf(m_run, cmax);
    const float corr = (m_new == -INFINITY) ? 1.f : __expf(m_run - m_new);
    float psum = 0.f;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const float p = (s[t] == -INFINITY) ? 0.f : __expf(s[t] - m_new);
      Ss[qrow * ATT_KT + qlane + 16 * t] = p;
      psum += p;
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) psum += __shfl_xor_sync(0xffffffffu, psum, o);
    l_run = l_run * corr + psum;
    m_run = m_new;
    __syncwarp();   // a row's 16 threads are half a warp
#pragma unroll
    for (int i = 0; i < NC / 2; ++i) {
      const int c = 4 * qlane + 64 * i;
      if (c < hd) {
        float4 v0 = make_float4(acc[i].x * corr, acc[i].y * corr, acc[i].z * corr, acc[i].w * corr), v1 = zero;
#pragma unroll(NC <= 4 ? 8 : 2)
        for (int q = 0; q < ATT_KT; q += 4) {
          const float4 p = ld4(Ss + qrow * ATT_KT + q);
          const float* vs = Vs + q * hd + c;
          fma4(v0, p.x, ld4(vs));
          fma4(v1, p.y, ld4(vs + hd));
          fma4(v0, p.z, ld4(vs + 2 * hd));
          fma4(v1, p.w, ld4(vs + 3 * hd));
        }
        acc[i] = make_float4(v0.x + v1.x, v0.y + v1.y, v0.z + v1.z, v0.w + v1.w);
      }
    }
  }
  if (r < nrows) {
    T* o = (T*)a.out + (size_t)(b * a.H + j) * a.ld_out + h * hd;
    const float inv = 1.f / l_run;
#pragma unroll
    for (int i = 0; i < NC / 2; ++i) {
      const int c = 4 * qlane + 64 * i;
      if (c < hd) st4(o + c, make_float4(acc[i].x * inv, acc[i].y * inv, acc[i].z * inv, acc[i].w * inv));
    }
  }
}

static size_t att_smem(int hd) {
  return (size_t)((ATT_QT + ATT_KT) * (hd + 4) + ATT_KT * hd + ATT_QT * ATT_KT) * sizeof(float);
}

cudaError_t launch_attention_simt(const AttnArgs& a, Dtype dt, cudaStream_t st) {
  if (a.hd > 256 || a.hd % 8) return cudaErrorInvalidValue;
  const int G = a.Hq / a.Hkv;
  dim3 grid(a.B * a.Hkv, (a.H * G + ATT_QT - 1) / ATT_QT);
  const size_t smem = att_smem(a.hd);
  const bool bf = dt == DT_BF16;
  if (a.hd <= 64)
    return launch_kernel(bf ? attention_simt_kernel<bf16, 2> : attention_simt_kernel<float, 2>, grid, dim3(ATT_THREADS), smem, st, 1, a);
  if (a.hd <= 128)
    return launch_kernel(bf ? attention_simt_kernel<bf16, 4> : attention_simt_kernel<float, 4>, grid, dim3(ATT_THREADS), smem, st, 1, a);
  return launch_kernel(bf ? attention_simt_kernel<bf16, 8> : attention_simt_kernel<float, 8>, grid, dim3(ATT_THREADS), smem, st, 1, a);
}

// ============================================================================ FOP adapter cross-attention

// One CTA per (robot b, query head h) and half of the slots; warp w takes slots w,
// w + 8, ... of them.  Lane f scores FOP keys f and f + 32 (K rows padded by four
// floats, so that 16-byte reads of eight keys hit distinct banks), the softmax
// runs once across the lanes, then the lanes split the head dim over the
// weighted values.  (Lanes over the head dim with a warp reduction per key, and
// every lane's own exponentials: 96 us more per adapter at 4 robots x 30 slots x
// 16 heads x 32 keys.)
template <typename T>
__global__ void __launch_bounds__(256) fop_xattn_kernel(const T* __restrict__ Q, const T* __restrict__ KV,
                                                        T* __restrict__ out, int H, int F, int Hq, int Hkv, int hd,
                                                        const float* __restrict__ gate) {
  pdl_trigger();
  extern __shared__ float xs[];
  const int ld = hd + 4;
  float* Ks = xs;                 // [F][hd + 4]
  float* Vs = Ks + F * ld;        // [F][hd]
  float* Qs = Vs + F * hd;        // [8 warps][hd]
  float* Ps = Qs + 8 * hd;        // [8 warps][64]
  const int b = blockIdx.x / Hq, h = blockIdx.x % Hq, g = h / (Hq / Hkv);
  const int ldkv = 2 * Hkv * hd, ldq = Hq * hd;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float scale = rsqrtf((float)hd), gt = tanhf(gate[0]);
  pdl_wait();
  for (int f = warp; f < F; f += 8) {
    const T* row = KV + (size_t)(b * F + f) * ldkv + g * hd;
    for (int c = 4 * lane; c < hd; c += 128) {
      st4(Ks + f * ld + c, ld4(row + c));
      st4(Vs + f * hd + c, ld4(row + Hkv * hd + c));
    }
  }
  __syncthreads();
  float *q = Qs + warp * hd, *p = Ps + warp * 64;
  const int per = (H + gridDim.y - 1) / gridDim.y, j1 = min(H, (int)(blockIdx.y + 1) * per);
  for (int j = blockIdx.y * per + warp; j < j1; j += 8) {
    const size_t o0 = (size_t)(b * H + j) * ldq + h * hd;
    for (int c = 4 * lane; c < hd; c += 128) st4(q + c, ld4(Q + o0 + c));
    __syncwarp();
    float s[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int f = lane + 32 * t;
      if (f >= F) continue;
      float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int c = 0; c < hd; c += 4) {
        const float4 x = ld4(q + c), k = ld4(Ks + f * ld + c);
        d.x = fmaf(x.x, k.x, d.x);
        d.y = fmaf(x.y, k.y, d.y);
        d.z = fmaf(x.z, k.z, d.z);
        d.w = fmaf(x.w, k.w, d.w);
      }
      s[t] = ((d.x + d.y) + (d.z + d.w)) * scale;
    }
    const float mx = warp_max(fmaxf(s[0], s[1]));
    const float e0 = __expf(s[0] - mx), e1 = __expf(s[1] - mx);   // exp(-inf) = 0 past F
    const float inv = gt / warp_sum(e0 + e1);
    p[lane] = e0;
    p[lane + 32] = e1;
    __syncwarp();
    for (int c = lane; c < hd; c += 32) {
      float a0 = 0.f, a1 = 0.f;
      int f = 0;
      for (; f + 1 < F; f += 2) {
        a0 = fmaf(p[f], Vs[f * hd + c], a0);
        a1 = fmaf(p[f + 1], Vs[(f + 1) * hd + c], a1);
      }
      if (f < F) a0 = fmaf(p[f], Vs[f * hd + c], a0);
      out[o0 + c] = from_f32<T>((a0 + a1) * inv);
    }
    __syncwarp();
  }
}

static size_t xattn_smem(int F, int hd) {
  return ((size_t)F * (2 * hd + 4) + 8 * hd + 8 * 64) * sizeof(float);
}

cudaError_t launch_fop_xattn(const void* Q, const void* KV, void* out, int B, int H, int F, int Hq, int Hkv, int hd,
                             const float* gate, Dtype dt, cudaStream_t st) {
  if (B <= 0 || H <= 0) return cudaSuccess;
  if (F < 1 || F > 64 || hd > 256) return cudaErrorInvalidValue;
  const dim3 grid(B * Hq, H > 8 ? 2 : 1);
  if (dt == DT_BF16)
    return launch_kernel(fop_xattn_kernel<bf16>, grid, dim3(256), xattn_smem(F, hd), st, 1, (const bf16*)Q,
                         (const bf16*)KV, (bf16*)out, H, F, Hq, Hkv, hd, gate);
  return launch_kernel(fop_xattn_kernel<float>, grid, dim3(256), xattn_smem(F, hd), st, 1, (const float*)Q,
                       (const float*)KV, (float*)out, H, F, Hq, Hkv, hd, gate);
}

// ============================================================================ tail

// One CTA per robot: a'_j = a_j + dt_j v_j (Eq. 3), released = a'_0, buffer
// slots shift forward, the last slot receives the Gaussian action of index
// counters[b], and the counter advances.
// (Bound by load latency: a thread's elements load four at a time; one at a time
// the launch took 7 us instead of 4.5 at 50 slots of 32 actions.)
__global__ void tail_kernel(TailArgs a) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ float sa[];   // [H][A]
  const int b = blockIdx.x;
  const int H = a.H, A = a.A;
  float* buf = a.buffer + (size_t)b * H * A;
  const float* v = a.vel + (size_t)b * H * A;
  const float* tb = a.slot_times + (size_t)b * a.t_stride;   // robot b's schedule
  constexpr int U = 4;   // elements whose loads a thread issues together
  for (int i0 = threadIdx.x; i0 < H * A; i0 += U * blockDim.x) {
    float vi[U], old[U], dt[U], rm[U], sv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = min(i0 + u * (int)blockDim.x, H * A - 1), j = i / A, o = i - j * A;
      vi[u] = v[i];
      old[u] = buf[i];
      dt[u] = __fsub_rn(tb[j], j ? tb[j - 1] : 0.f);
      rm[u] = a.state ? a.rel_mask[o] : 0.f;
      sv[u] = a.state ? a.state[(size_t)b * A + o] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * (int)blockDim.x;
      if (i >= H * A) break;
      // absolute buffer, relative expert: the slot also moves by dt m s as its
      // flow time drops from t_j to t_{j-1}
      sa[i] = fmaf(dt[u], a.state ? fmaf(rm[u], sv[u], vi[u]) : vi[u], old[u]);
      if (a.vel_out) a.vel_out[(size_t)b * H * A + i] = vi[u];
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < H * A; i += blockDim.x) {
    if (i < A) a.released[(size_t)b * A + i] = sa[i];
    if (i < (H - 1) * A) buf[i] = sa[i + A];
  }
  const uint64_t n = a.counters[b];
  const uint64_t seed = a.seeds[b];
  for (int g = threadIdx.x; g < (A + 3) / 4; g += blockDim.x) {
    float z[4];
    action_noise4(seed, n, (uint32_t)g, z);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (4 * g + i < A) buf[(size_t)(H - 1) * A + 4 * g + i] = z[i];
  }
  __syncthreads();
  if (threadIdx.x == 0) a.counters[b] = n + 1;
}

cudaError_t launch_tail(const TailArgs& a, cudaStream_t st) {
  if (a.B <= 0) return cudaSuccess;
  const size_t smem = (size_t)a.H * a.A * sizeof(float);
  return launch_kernel(tail_kernel, dim3(a.B), dim3(256), smem, st, 1, a);
}

// The step's last three stages in one launch (bf16 mode, A <= 32), one CTA per R
// consecutive slots of a robot: the final adaRMSNorm of an action row (Eq. 2's
// modulation, offset off), the velocity head v = Y W_out^T + b_out on the
// bf16-rounded normed row (as the separate norm + GEMM compute it) and the slot's
// Euler step; slot 0 is released, the last slot's row takes the new noise, and the
// robot's CTA that finishes last shifts the others forward.  (The CTAs count
// themselves on cnt[b], reset by the last one, so it is zero between launches: the
// classic last-block pattern, no CTA waits for another.)
// Bound by the latency of its loads, so they go out together: W_out and the
// bias, which no earlier kernel writes, before the wait for those kernels, the
// rest right after it, without a branch on A between them (outputs past A
// repeat the last row and are dropped).  (50 rows, A 32, D 1024: 6 us, 10 with
// the loads behind the norm and the whole tail in the last CTA; 120 rows, A 20: 6,
// and 17.)  R > 1, for more than two rows per SM: the CTA keeps its share of W_out
// (64 KB in all) in registers for its rows, the next row's loads in flight behind
// this one's sums.  (Whole steps of 3200 and 800 rows: 2642 and 1253 us with one
// row per CTA, 2615 and 1249 with four, 2612 and 1248 with eight, 2633 and 1262
// with eight in 128 registers, two CTAs per SM.)
template <int R>
__global__ void __launch_bounds__(256) head_tail_kernel(HeadArgs h, TailArgs a) {
  pdl_trigger();
  __shared__ float red[2][8][33];   // per-warp sums: [warp][output] (+ the norm's row sum in [w][32])
  __shared__ int last;
  const int H = a.H, A = a.A, D = h.D, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, o = threadIdx.x;
  const int nc = (H + R - 1) / R;   // CTAs per robot
  const int b = blockIdx.x / nc, j0 = blockIdx.x % nc * R, j1 = min(H, j0 + R), f0 = 4 * threadIdx.x;
  const float* mb = h.mod_b + h.off;
  uint2 wq[32];   // 4 bf16 of every W_out row
  float4 x, b0, b1, t0, t1, d0, d1;
  auto weights = [&](int f) {
#pragma unroll
    for (int i = 0; i < 32; ++i) wq[i] = *(const uint2*)((const bf16*)h.w + (size_t)min(i, A - 1) * D + f);
    b0 = ld4(mb + f);
    b1 = ld4(mb + D + f);
  };
  if (f0 < D) weights(f0);
  pdl_wait();
  const float* md = h.modv + (size_t)(h.drow ? h.drow[b] : H + b) * h.mod_ld + h.off;
  auto row = [&](int j, int f) {
    const float* mt = h.modv + (size_t)(b * h.t_stride + j) * h.mod_ld + h.off;
    x = ld4(h.x + (size_t)(b * H + j) * D + f);
    t0 = ld4(mt + f);
    t1 = ld4(mt + D + f);
  };
  auto offset = [&](int f) {
    d0 = ld4(md + f);
    d1 = ld4(md + D + f);
  };
  if (f0 < D) {
    row(j0, f0);
    offset(f0);
  }
  // a slot's Euler step (threads o < A): its flow times, old value and, with an
  // absolute buffer and a relative expert, the state it also moves by
  float* buf = a.buffer + (size_t)b * H * A;
  const float* tb = a.slot_times + (size_t)b * a.t_stride;   // robot b's schedule
  float dt = 0.f, old = 0.f, rm = 0.f, sv = 0.f, bias = 0.f;
  auto euler = [&](int j) {
    dt = __fsub_rn(tb[j], j ? tb[j - 1] : 0.f);
    old = buf[j * A + o];
  };
  if (o < A) {
    euler(j0);
    bias = h.b[o];
    if (a.state) {
      rm = a.rel_mask[o];
      sv = a.state[(size_t)b * A + o];
    }
  }
  const uint64_t n = a.counters[b];
  for (int j = j0; j < j1; ++j) {
    float(*rd)[33] = red[(j - j0) & 1];
    // sum of squares of the row (4 features per thread per pass)
    float ss = 0.f;
    if (f0 < D) ss = x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
    for (int f = f0 + 4 * blockDim.x; f < D; f += 4 * blockDim.x) {
      const float4 xv = ld4(h.x + (size_t)(b * H + j) * D + f);
      ss += xv.x * xv.x + xv.y * xv.y + xv.z * xv.z + xv.w * xv.w;
    }
    ss = warp_sum(ss);
    if (lane == 0) rd[warp][32] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += rd[w][32];
    const float inv = rsqrtf(tot / (float)D + 1e-6f);
    // this thread's partial products for all 32 outputs
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.f;
    for (int f = f0; f < D; f += 4 * blockDim.x) {
      if (f != f0) {
        weights(f);
        row(j, f);
        offset(f);
      }
      const float xs[4] = {x.x, x.y, x.z, x.w};
      const float sc[4] = {t0.x + d0.x + b0.x, t0.y + d0.y + b0.y, t0.z + d0.z + b0.z, t0.w + d0.w + b0.w};
      const float sh[4] = {t1.x + d1.x + b1.x, t1.y + d1.y + b1.y, t1.z + d1.z + b1.z, t1.w + d1.w + b1.w};
      float y[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) y[e] = __bfloat162float(__float2bfloat16_rn(xs[e] * inv * (1.f + sc[e]) + sh[e]));
      if (R > 1 && f + 4 * blockDim.x >= D && j + 1 < j1) row(j + 1, f0);   // (D <= 1024: one pass)
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        acc[i] = fmaf(y[0], __uint_as_float(wq[i].x << 16), acc[i]);
        acc[i] = fmaf(y[1], __uint_as_float(wq[i].x & 0xFFFF0000u), acc[i]);
        acc[i] = fmaf(y[2], __uint_as_float(wq[i].y << 16), acc[i]);
        acc[i] = fmaf(y[3], __uint_as_float(wq[i].y & 0xFFFF0000u), acc[i]);
      }
    }
    // warp: lane o ends with the warp's sum of output o (each step keeps half
    // of the outputs and adds the partner's half)
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
      const bool up = (lane & off) != 0;
#pragma unroll
      for (int i = 0; i < off; ++i) {
        const float send = up ? acc[i] : acc[i + off];
        const float keep = up ? acc[i + off] : acc[i];
        acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
      }
    }
    rd[warp][lane] = acc[0];
    __syncthreads();
    if (o < A) {
      float v = bias;
#pragma unroll
      for (int w = 0; w < 8; ++w) v += rd[w][o];
      if (a.vel_out) a.vel_out[((size_t)b * H + j) * A + o] = v;
      const float next = fmaf(dt, a.state ? fmaf(rm, sv, v) : v, old);
      if (j == 0) a.released[(size_t)b * A + o] = next;
      else h.v[((size_t)b * H + j) * A + o] = next;
      if (R > 1 && j + 1 < j1) euler(j + 1);
    }
  }
  if (j1 == H) {   // (the last slot's old value has been read)
    const int g = (int)blockDim.x - 1 - (int)threadIdx.x;
    if (4 * g < A) {
      float z[4];
      action_noise4(a.seeds[b], n, (uint32_t)g, z);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (4 * g + i < A) buf[(size_t)(H - 1) * A + 4 * g + i] = z[i];
    }
  }
  // the robot's last CTA to finish shifts the slots
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const int done = atomicAdd(h.cnt + b, 1);
    last = done == nc - 1;
    if (last) h.cnt[b] = 0;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const float* next = h.v + ((size_t)b * H + 1) * A;
  const int m = (H - 1) * A;
  for (int i0 = threadIdx.x; i0 < m; i0 += 8 * blockDim.x) {
    float q[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) q[k] = i0 + k * 256 < m ? __ldcg(next + i0 + k * 256) : 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (i0 + k * 256 < m) buf[i0 + k * 256] = q[k];
  }
  if (threadIdx.x == 0) a.counters[b] = n + 1;
}

cudaError_t launch_head_tail(const HeadArgs& h, const TailArgs& a, int num_sms, cudaStream_t st) {
  if (a.B <= 0) return cudaSuccess;
  if (a.A > 32 || h.D % 4) return cudaErrorNotSupported;
  // (rows of up to 1024 features: one pass, whose weights stay in registers)
  if (a.B * a.H > 2 * num_sms && h.D <= 1024)
    return launch_kernel(head_tail_kernel<8>, dim3(a.B * ((a.H + 7) / 8)), dim3(256), 0, st, 1, h, a);
  return launch_kernel(head_tail_kernel<1>, dim3(a.B * a.H), dim3(256), 0, st, 1, h, a);
}

// Full-horizon denoising (the synchronous baseline): every slot takes the
// same Euler step a += dt v with dt = t_now - t_next (float32, read off the
// time grid like the rolling step's dt_j); nothing is released or shifted.
__global__ void denoise_tail_kernel(float* __restrict__ buffer, const float* __restrict__ vel, float* __restrict__ vel_out,
                                    int n, float t_now, float t_next) {
  pdl_trigger();
  pdl_wait();
  const float dt = __fsub_rn(t_now, t_next);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float v = vel[i];
    buffer[i] = fmaf(dt, v, buffer[i]);
    if (vel_out) vel_out[i] = v;
  }
}

cudaError_t launch_denoise_tail(float* buffer, const float* vel, float* vel_out, int B, int H, int A, float t_now,
                                float t_next, cudaStream_t st) {
  const int n = B * H * A;
  if (n <= 0) return cudaSuccess;
  const int blocks = std::min((n + 255) / 256, 1024);
  return launch_kernel(denoise_tail_kernel, dim3(blocks), dim3(256), 0, st, 1, buffer, vel, vel_out, n, t_now, t_next);
}

// The flow times of up to H synchronous denoising passes from pass n0 on (the
// last one's repeated): rows of one conditioning for all of them.
__global__ void fill_times_kernel(float* __restrict__ times, int H, PassTimes t, int n0, int n_steps) {
  pdl_trigger();
  pdl_wait();
  for (int i = threadIdx.x; i < H; i += blockDim.x) times[i] = t.t[min(n0 + i, n_steps - 1)];
}

cudaError_t launch_fill_times(float* times, int H, const PassTimes& t, int n0, int n_steps, cudaStream_t st) {
  return launch_kernel(fill_times_kernel, dim3(1), dim3(128), 0, st, 1, times, H, t, n0, n_steps);
}

// A fresh chunk: slot j of robot b receives the Gaussian action of index
// counters[b] + j, and the counter advances by H.
__global__ void chunk_noise_kernel(float* __restrict__ buffer, const uint64_t* __restrict__ seeds,
                                   uint64_t* __restrict__ counters, int H, int A) {
  pdl_trigger();
  pdl_wait();
  const int b = blockIdx.x;
  const int groups = (A + 3) / 4;
  const uint64_t n0 = counters[b];
  for (int i = threadIdx.x; i < H * groups; i += blockDim.x) {
    const int j = i / groups, g = i % groups;
    float z[4];
    action_noise4(seeds[b], n0 + (uint64_t)j, (uint32_t)g, z);
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (4 * g + t < A) buffer[((size_t)b * H + j) * A + 4 * g + t] = z[t];
  }
  __syncthreads();
  if (threadIdx.x == 0) counters[b] = n0 + (uint64_t)H;
}

cudaError_t launch_chunk_noise(float* buffer, const uint64_t* seeds, uint64_t* counters, int B, int H, int A,
                               cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  return launch_kernel(chunk_noise_kernel, dim3(B), dim3(128), 0, st, 1, buffer, seeds, counters, H, A);
}

cudaError_t init_simt_kernels() {
  const int att = (int)att_smem(256);
  cudaError_t e = cudaFuncSetAttribute(attention_simt_kernel<bf16, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, att);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(attention_simt_kernel<float, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, att);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tail_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 16384 * (int)sizeof(float));
  const int xa = (int)xattn_smem(64, 256);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fop_xattn_kernel<bf16>, cudaFuncAttributeMaxDynamicSharedMemorySize, xa);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fop_xattn_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, xa);
  return e;
}

__global__ void reset_kernel(float* __restrict__ buffer, const uint64_t* __restrict__ seeds,
                             uint64_t* __restrict__ counters, int H, int A) {
  const int b = blockIdx.x;
  const int groups = (A + 3) / 4;
  for (int i = threadIdx.x; i < H * groups; i += blockDim.x) {
    const int j = i / groups, g = i % groups;
    float z[4];
    action_noise4(seeds[b], (uint64_t)j, (uint32_t)g, z);
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (4 * g + t < A) buffer[((size_t)b * H + j) * A + 4 * g + t] = z[t];
  }
  if (threadIdx.x == 0) counters[b] = (uint64_t)H;
}

cudaError_t launch_reset(float* buffer, const uint64_t* seeds, uint64_t* counters, int B, int H, int A,
                         cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  reset_kernel<<<B, 128, 0, st>>>(buffer, seeds, counters, H, A);
  return cudaGetLastError();
}

__global__ void copy_list_kernel(CopyList c) {
  const int i = blockIdx.y;
  const size_t bytes = c.bytes[i], t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t step = (size_t)gridDim.x * blockDim.x;
  if ((((uintptr_t)c.dst[i] | (uintptr_t)c.src[i] | bytes) & 15) == 0) {
    for (size_t k = t0; k < bytes / 16; k += step) ((uint4*)c.dst[i])[k] = ((const uint4*)c.src[i])[k];
  } else {
    for (size_t k = t0; k < bytes / 2; k += step) ((uint16_t*)c.dst[i])[k] = ((const uint16_t*)c.src[i])[k];
  }
}

cudaError_t launch_copy_list(const CopyList& c, cudaStream_t st) {
  size_t most = 0;
  for (int i = 0; i < c.n; ++i) most = std::max(most, c.bytes[i]);
  if (most == 0) return cudaSuccess;
  const unsigned blocks = (unsigned)std::min<size_t>((most / 16 + 255) / 256 + 1, 256);
  copy_list_kernel<<<dim3(blocks, c.n), 256, 0, st>>>(c);
  return cudaGetLastError();
}

__global__ void delay_kernel(unsigned long long ns) {
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  do {
    __nanosleep(10000);
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  } while (t - t0 < ns);
}

cudaError_t launch_delay(unsigned long long ns, cudaStream_t st) {
  delay_kernel<<<1, 1, 0, st>>>(ns);
  return cudaGetLastError();
}

__global__ void flip_kernel(int* s, CtxList f) {
  for (int i = threadIdx.x; i < f.n; i += blockDim.x) {
    s[2 * f.robot[i]] = f.slot[i];
    s[2 * f.robot[i] + 1] = f.len[i];
  }
}

cudaError_t launch_flip(int* ctx_state, const CtxList& f, cudaStream_t st) {
  if (f.n <= 0) return cudaSuccess;
  flip_kernel<<<1, 128, 0, st>>>(ctx_state, f);
  return cudaGetLastError();
}

// Context rows of the listed robots into their slots: source [L][src_n][Hkv]
// [P][row] with the list's robots at positions i0 .. i0 + f.n - 1 of each
// layer, destination [slot][L][Bmax][Hkv][Pmax][row] (16-byte words); rows P ..
// Pz - 1 become zeros.
__global__ void ctx_scatter_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst0, uint4* __restrict__ dst1,
                                   int src_n, int i0, int Bmax, int Hkv, int P, int Pz, int Pmax, int row_words,
                                   CtxList f) {
  const int z = blockIdx.y;                  // (l * f.n + i) * Hkv + g
  const int g = z % Hkv, li = z / Hkv;
  const int i = li % f.n, l = li / f.n;
  const size_t words = (size_t)P * row_words, all = (size_t)Pz * row_words;
  const uint4* s = src + ((size_t)(l * src_n + i0 + i) * Hkv + g) * words;
  uint4* d = (f.slot[i] ? dst1 : dst0) + (((size_t)l * Bmax + f.robot[i]) * Hkv + g) * (size_t)Pmax * row_words;
  for (size_t w = (size_t)blockIdx.x * blockDim.x + threadIdx.x; w < all; w += (size_t)gridDim.x * blockDim.x)
    d[w] = w < words ? s[w] : make_uint4(0, 0, 0, 0);
}

cudaError_t launch_ctx_scatter(const void* src, int src_n, int i0, void* dst0, void* dst1, int L, int Bmax, int Hkv,
                               int P, int Pz, int Pmax, size_t row_bytes, const CtxList& f, cudaStream_t st) {
  if (f.n <= 0 || P <= 0) return cudaSuccess;
  if (row_bytes % 16 || ((uintptr_t)src | (uintptr_t)dst0 | (uintptr_t)dst1) % 16) return cudaErrorMisalignedAddress;
  const int row_words = (int)(row_bytes / 16);
  const size_t words = (size_t)P * row_words;
  dim3 grid((unsigned)std::min<size_t>((words + 255) / 256, 64), (unsigned)(L * f.n * Hkv));
  ctx_scatter_kernel<<<grid, 256, 0, st>>>((const uint4*)src, (uint4*)dst0, (uint4*)dst1, src_n, i0, Bmax, Hkv, P,
                                           Pz, Pmax, row_words, f);
  return cudaGetLastError();
}

}  // namespace ravel

// 1 if an fp32 GEMM of these sizes (16-byte aligned rows) takes the row kernel, for tests.
extern "C" int ravel_debug_rows_gemm(int M, int N, int K, int epi) {
  using namespace ravel;
  return rows_gemm_supported(GemmArgs{nullptr, K, nullptr, K, M, N, K, (Epi)epi, nullptr, N, DT_F32, nullptr}) ? 1 : 0;
}
