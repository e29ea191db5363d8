// Projection GEMM on the 5th-generation tensor cores (tcgen05 + TMEM + TMA).
//
//   out[m][n] (op)= sum_k X[m][k] * W[n][k]       X: activations [M][K] bf16
//                                                  W: weights     [N][K] bf16 (K-major)
//
// Swap-AB tiling: a tile is 128 weight rows (the MMA's M = 128 TMEM lanes) by
// BN tokens (the MMA's N, 32..256): with 50-66 tokens per robot the weights
// are the large operand, and one kernel covers both the bandwidth-bound
// batch-1 case (few tiles, split-K over the grid) and the compute-bound
// large-batch case (many 128 x 256 tiles).
//
// Warp roles (192 threads): warp 0 = TMA producer, warp 1 = TMEM allocator +
// MMA issuer (both stay converged: every lane waits, the elected one's
// instruction is predicated), warps 2..5 = epilogue (warp w reads TMEM lanes
// 32*(w%4)..+31).  Operand tiles are 64 K-elements wide (one 128-byte
// swizzle row) in an S-stage shared-memory ring guarded by mbarriers.  Every
// wait is bounded: on timeout the kernel raises ERR_TIMEOUT in the device
// error word and unwinds instead of hanging.
//
// Work distribution:
//  * no split: CTAs walk the tiles (persistent when there are more tiles than
//    SMs) with two TMEM accumulators, so the epilogue of one tile overlaps the
//    MMAs of the next; where the tiles are many, pairs of CTAs run 256-row
//    tiles with the two-SM MMA instead (tc_gemm_pair_kernel, below);
//  * few tiles: the K dimension is split over grid.z.  The splits of a tile
//    form a thread-block cluster and rank q sums a token slice over the splits
//    in order (deterministic) and applies the epilogue.  The partials travel
//    by st.async straight into rank q's shared memory, completing on an
//    mbarrier there, or, where the output is not 16-byte aligned, through L2
//    and the cluster barrier.
// Epilogue: a chunk of tokens is written into a shared-memory box in the
// output layout and leaves through one TMA store (or a TMA reduce-add for the
// residual-stream epilogue), double-buffered so that the epilogue threads
// never wait on global memory; unaligned outputs are stored by the threads
// instead.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "kernels.h"
#include "launch.h"
#include "tc_common.cuh"

namespace ravel {
namespace {

constexpr int TC_BM = 128;
constexpr int TC_BK = 64;
constexpr int TC_THREADS = 192;
constexpr int TC_PAIR_THREADS = 320;   // pair kernel: TMA, MMA and two sets of four epilogue warps
constexpr uint32_t TC_A_BYTES = TC_BM * TC_BK * 2;
constexpr int TC_SMEM_BUDGET = 200 * 1024;   // operand ring
constexpr int TC_SMEM_MAX = 227 * 1024;
constexpr size_t TC_SMEM_SM = 228 * 1024;
constexpr int TC_RING_SPLIT = 128 * 1024;    // operand ring of a split-K launch
constexpr int STG_LD = 132;                  // SIMT staging pitch (floats): 16 tokens x 128 tile rows
constexpr uint32_t STG_BYTES = 16 * STG_LD * 4;
constexpr uint32_t XCH_BYTES = 32 * STG_LD * 4;  // GeGLU transpose tile (TMA epilogue): <= 32 tokens x 128 rows

enum { RED_NONE = 0, RED_L2_CLUSTER = 1, RED_DSMEM = 2, RED_DSMEM32 = 3 };
// Epilogue kind of an instantiation: outputs through TMA boxes as fp32, bf16,
// a reduce-add into the fp32 residual stream or the GeGLU pair -- fixed, so
// that a long persistent launch carries only the code of its own epilogue --
// or stored by the threads: a split rank's slice (EK_SLICE: any epilogue, so
// that the short split-K launches of one step all run one binary, whose code
// the previous launch has left in the SM's instruction cache), or any tile
// (EK_GENERIC: unaligned outputs).
enum { EK_F32 = 0, EK_BF16 = 1, EK_ADD = 2, EK_GEGLU = 3, EK_GENERIC = 4, EK_SLICE = 5 };


struct TcParams {
  int M, N;
  int bn, stages, splits, num_kb;
  uint32_t ncols;       // TMEM columns of the launch
  uint32_t acc_cols;    // TMEM columns of one accumulator
  int accs;             // accumulators that an item's K range is cut into, at most one per k-tile (sum_accumulators)
  int tiles_n, tiles_m, num_tiles;
  int epi;              // Epi
  int out_bf16;
  void* out;
  int ldo;
  const float* bias;
  float* ws;
  int* err;
  int oneshot;          // split launch whose whole K range fits the ring: tmW / tmX are 3-D maps
                        // (64, rows, K / 64) and one box each brings all of its k-tiles
  int box_m;            // tokens per epilogue chunk (= rows of a TMA output box)
  uint32_t box_bytes;   // bytes of one TMA output box (1024-aligned)
  uint32_t stg_off;     // SIMT transpose tile, or two TMA output boxes
  uint32_t xch_off;     // GeGLU exchange
  uint32_t rcv_off;     // RED_DSMEM*: the partials received from the splits, [split][cpr / 4][128 rows]
                        // float4 (bf16: two rows per 16 bytes)
  uint32_t bar_off;     // mbarriers, TMEM slot, flags
  unsigned long long wait_ns;   // limit of every bounded wait (ERR_TIMEOUT after it)
  int withhold;         // fault injection (tests): the MMA thread first waits for an arrival that
                        // nobody makes, so the launch gives up after wait_ns and unwinds
  const int* skip;      // optional device flag read after the dependency wait: nonzero -> the launch
                        // completes the copies it started and exits without computing
  uint32_t set_bytes;   // pair kernel: bytes from epilogue set 0's boxes / exchange to set 1's
};

// The i-th work item of this CTA: a tile (tn, tm) and split sp.  With splits
// the grid is (tiles_n, tiles_m, splits) and every CTA has one item; without,
// the grid is 1-D and CTA c takes tiles c, c + gridDim.x, ... (token tiles of
// one weight tile are adjacent, so concurrently running CTAs share it in L2).
__device__ __forceinline__ bool work_item(const TcParams& p, int i, int& tn, int& tm, int& sp) {
  if (p.splits > 1) {
    if (i) return false;
    tn = blockIdx.x;
    tm = blockIdx.y;
    sp = blockIdx.z;
    return true;
  }
  const int t = blockIdx.x + i * gridDim.x;
  if (t >= p.num_tiles) return false;
  tm = t % p.tiles_m;
  tn = t / p.tiles_m;
  sp = 0;
  return true;
}

__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 1, 128;" ::: "memory"); }
// the 128 threads of epilogue warp set `set` (the pair kernel runs two sets)
__device__ __forceinline__ void epi_bar_set(int set) {
  if (set) asm volatile("bar.sync 2, 128;" ::: "memory");
  else asm volatile("bar.sync 1, 128;" ::: "memory");
}

// v[4g + e] += sum over splits s = 0..S-1 (in order) of the partial of this
// thread's row at column group g (g < NG); b0 points at split 0, group 0;
// splits are sstride floats apart, groups 512.  Up to 16 float4 loads are in
// flight per batch; splits past S add exact zeros.
template <int NG>
__device__ __forceinline__ void reduce_splits_l2(const float* b0, int S, size_t sstride, float v[16]) {
  constexpr int GB = 16 / NG;
  for (int s0 = 0; s0 < S; s0 += GB) {
    float4 x[GB][NG];
#pragma unroll
    for (int u = 0; u < GB; ++u)
#pragma unroll
      for (int g = 0; g < NG; ++g)
        x[u][g] = (s0 + u < S) ? __ldcg((const float4*)(b0 + (size_t)(s0 + u) * sstride + (size_t)g * 512))
                               : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < GB; ++u)
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        v[4 * g] += x[u][g].x;
        v[4 * g + 1] += x[u][g].y;
        v[4 * g + 2] += x[u][g].z;
        v[4 * g + 3] += x[u][g].w;
      }
  }
}

// v[4g + e] (g < NG <= 8) = sum over splits s = 0..S-1 (in order) of the
// received bf16 partials: b0 points at this thread's four tokens of split 0,
// group 0 (half of a two-row message); group g of split s is (s * NG + g) *
// 128 uint2 further.
template <int NG>
__device__ __forceinline__ void reduce_slice_smem(const uint2* b0, int S, float v[32]) {
  #pragma unroll 1
  for (int s = 0; s < S; ++s) {
    uint2 x[NG];
#pragma unroll
    for (int g = 0; g < NG; ++g) x[g] = b0[(size_t)(s * NG + g) * TC_BM];
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      v[4 * g] += __uint_as_float(x[g].x << 16);
      v[4 * g + 1] += __uint_as_float(x[g].x & 0xFFFF0000u);
      v[4 * g + 2] += __uint_as_float(x[g].y << 16);
      v[4 * g + 3] += __uint_as_float(x[g].y & 0xFFFF0000u);
    }
  }
}

// As above for fp32 partials: b0 points at this thread's row of split 0,
// group 0; group g of split s is (s * NG + g) * 128 float4 further.
template <int NG>
__device__ __forceinline__ void reduce_slice_smem(const float4* b0, int S, float v[32]) {
  #pragma unroll 1
  for (int s = 0; s < S; ++s) {
    float4 x[NG];
#pragma unroll
    for (int g = 0; g < NG; ++g) x[g] = b0[(size_t)(s * NG + g) * TC_BM];
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      v[4 * g] += x[g].x;
      v[4 * g + 1] += x[g].y;
      v[4 * g + 2] += x[g].z;
      v[4 * g + 3] += x[g].w;
    }
  }
}

// v[k] += the item's other accumulators (in K order) at this thread's row,
// columns taddr + k of the first one.
__device__ __forceinline__ void add_accumulators(uint32_t taddr, uint32_t acc_cols, int accs, uint32_t v[16]) {
  #pragma unroll 1
  for (int j = 1; j < accs; j += 3) {   // up to three loads in flight
    const int n = accs - j;
    uint32_t x[3][16];
#pragma unroll
    for (int u = 0; u < 3; ++u)
      if (u < n) tmem_ld16_async(taddr + (uint32_t)(j + u) * acc_cols, x[u]);
    tmem_wait_ld();
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      tmem_reg_fence16(x[u]);
      if (u >= n) break;
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = __float_as_uint(__uint_as_float(v[k]) + __uint_as_float(x[u][k]));
    }
  }
}

// Epilogue of tokens m0 .. m0+nc-1 (nc <= 16) of tile row block tile_n: v[i]
// is this thread's tile row r at token m0+i.  All 128 epilogue threads call it
// together.  The chunk is transposed through `stage` so that each thread then
// writes one token's 16 (or, for GeGLU, 8) consecutive outputs as 16-byte
// stores.
__device__ __forceinline__ void epilogue_chunk(const TcParams& p, int tile_n, int m0, int nc, int r,
                                               const float v[16], float* stage) {
#pragma unroll
  for (int i = 0; i < 16; ++i) stage[i * STG_LD + r] = v[i];
  epi_bar();
  const int c = r >> 3, fg = r & 7;
  const int m = m0 + c;
  if (c < nc && m < p.M) {
    const float* srow = stage + c * STG_LD;
    if (p.epi == EPI_GEGLU) {
      // rows 0..63 of the tile are gate features, rows 64..127 the matching up features
      const int f0 = tile_n * 64 + fg * 8, nf = p.N / 2;
      float o[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int ng = tile_n * TC_BM + fg * 8 + q;   // gate row; its up row is ng + 64
        const float bg = p.bias ? p.bias[ng] : 0.f, bu = p.bias ? p.bias[ng + 64] : 0.f;
        o[q] = gelu_tanh_bf16out(srow[fg * 8 + q] + bg) * (srow[64 + fg * 8 + q] + bu);
      }
      bf16* dst = (bf16*)p.out + (size_t)m * p.ldo + f0;
      if (f0 + 8 <= nf && ((uintptr_t)dst & 15) == 0) {
        *(uint4*)dst = make_uint4(pack_bf16x2(o[0], o[1]), pack_bf16x2(o[2], o[3]), pack_bf16x2(o[4], o[5]),
                                  pack_bf16x2(o[6], o[7]));
      } else {
        for (int q = 0; q < 8; ++q)
          if (f0 + q < nf) dst[q] = __float2bfloat16_rn(o[q]);
      }
    } else {
      const int n0 = tile_n * TC_BM + fg * 16;
      const bool full = n0 + 16 <= p.N;
      float x[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        x[q] = srow[fg * 16 + q] + ((p.bias && n0 + q < p.N) ? p.bias[n0 + q] : 0.f);
        if (p.epi == EPI_STORE_SILU) x[q] = silu_f(x[q]);
      }
      if (p.epi == EPI_ADD_F32) {
        float* dst = (float*)p.out + (size_t)m * p.ldo + n0;
        if (full && ((uintptr_t)dst & 15) == 0) {
          float4 a[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) a[k] = *(const float4*)(dst + 4 * k);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            *(float4*)(dst + 4 * k) =
                make_float4(a[k].x + x[4 * k], a[k].y + x[4 * k + 1], a[k].z + x[4 * k + 2], a[k].w + x[4 * k + 3]);
        } else {
          for (int q = 0; q < 16; ++q)
            if (n0 + q < p.N) dst[q] += x[q];
        }
      } else if (p.out_bf16) {
        bf16* dst = (bf16*)p.out + (size_t)m * p.ldo + n0;
        if (full && ((uintptr_t)dst & 15) == 0) {
          *(uint4*)dst = make_uint4(pack_bf16x2(x[0], x[1]), pack_bf16x2(x[2], x[3]), pack_bf16x2(x[4], x[5]),
                                    pack_bf16x2(x[6], x[7]));
          *(uint4*)(dst + 8) = make_uint4(pack_bf16x2(x[8], x[9]), pack_bf16x2(x[10], x[11]),
                                          pack_bf16x2(x[12], x[13]), pack_bf16x2(x[14], x[15]));
        } else {
          for (int q = 0; q < 16; ++q)
            if (n0 + q < p.N) dst[q] = __float2bfloat16_rn(x[q]);
        }
      } else {
        float* dst = (float*)p.out + (size_t)m * p.ldo + n0;
        if (full && ((uintptr_t)dst & 15) == 0) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            *(float4*)(dst + 4 * k) = make_float4(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3]);
        } else {
          for (int q = 0; q < 16; ++q)
            if (n0 + q < p.N) dst[q] = x[q];
        }
      }
    }
  }
  epi_bar();
}


// TMA epilogue of tokens m0 .. m0+box_m-1 of tile row block tile_n: v[i] is
// this thread's tile row r at token m0+i, brow its bias.  All 128 epilogue
// threads call it together.  The chunk is written into output box `ebuf` in
// shared memory (token-major, as the output), and thread 64 sends the box
// with one TMA store (EPI_ADD_F32: TMA reduce-add into the residual stream);
// rows past M and columns past N are clipped by the tensor map.
// f(i) for i < n (n <= NV, a multiple of G), unrolled: without a bound
// check when n == NV, else one per group of G (the epilogue warps run one per
// scheduler, so every compare and branch in these loops is exposed latency)
template <int NV, int G = 4, typename F>
__device__ __forceinline__ void for_upto(int n, F&& f) {
  static_assert(NV % G == 0, "whole groups");
  if (n == NV) {
#pragma unroll
    for (int i = 0; i < NV; ++i) f(i);
  } else {
#pragma unroll
    for (int g = 0; g < NV; g += G) {
      if (g >= n) break;
#pragma unroll
      for (int i = g; i < g + G; ++i) f(i);
    }
  }
}

template <int EK, int NV = 16>
__device__ __forceinline__ void epilogue_tma(const TcParams& p, const CUtensorMap* tmO, int tile_n, int m0, int r,
                                             const float* v, float brow, uint8_t* boxes, float* xch, int& ebuf) {
  const int bm = p.box_m;   // <= NV
  // epilogue warp set (threads 64..191: 0; 192..319: 1, pair kernel only) and
  // the thread of the set that issues and waits for its TMA stores
  const int set = threadIdx.x >= 192 ? 1 : 0;
  const bool issuer = threadIdx.x == 64 + 128 * set;
  // the box written two chunks ago must have been read by its TMA store
  if (issuer) bulk_wait_read<1>();
  epi_bar_set(set);
  uint8_t* box = boxes + (size_t)ebuf * p.box_bytes;
  constexpr int kind = EK;
  if (kind == EK_GEGLU) {
    // tile rows 0..63 are gate features, 64..127 the matching up features:
    // transpose through xch so that every thread then forms 8 outputs of one
    // token (the GELUs spread over all 128 threads)
    for_upto<NV>(bm, [&](int i) { xch[i * STG_LD + r] = v[i] + brow; });
    epi_bar_set(set);
#pragma unroll
    for (int h = 0; h < NV / 16; ++h) {
      const int c = (r >> 3) + 16 * h, fg = r & 7;
      if (c < bm) {
        const float4* g4 = (const float4*)(xch + c * STG_LD + fg * 8);
        const float4* u4 = (const float4*)(xch + c * STG_LD + 64 + fg * 8);
        const float4 ga = g4[0], gb = g4[1], ua = u4[0], ub = u4[1];
        *(uint4*)((bf16*)box + c * 64 + fg * 8) =
            make_uint4(pack_bf16x2(gelu_tanh_bf16out(ga.x) * ua.x, gelu_tanh_bf16out(ga.y) * ua.y),
                       pack_bf16x2(gelu_tanh_bf16out(ga.z) * ua.z, gelu_tanh_bf16out(ga.w) * ua.w),
                       pack_bf16x2(gelu_tanh_bf16out(gb.x) * ub.x, gelu_tanh_bf16out(gb.y) * ub.y),
                       pack_bf16x2(gelu_tanh_bf16out(gb.z) * ub.z, gelu_tanh_bf16out(gb.w) * ub.w));
      }
    }
  } else if (kind == EK_BF16) {
    bf16* o = (bf16*)box;
    if (p.epi == EPI_STORE_SILU)
      for_upto<NV>(bm, [&](int i) { o[i * TC_BM + r] = __float2bfloat16_rn(silu_f(v[i] + brow)); });
    else
      for_upto<NV>(bm, [&](int i) { o[i * TC_BM + r] = __float2bfloat16_rn(v[i] + brow); });
  } else {
    float* o = (float*)box;
    if (kind == EK_F32 && p.epi == EPI_STORE_SILU)
      for_upto<NV>(bm, [&](int i) { o[i * TC_BM + r] = silu_f(v[i] + brow); });
    else
      for_upto<NV>(bm, [&](int i) { o[i * TC_BM + r] = v[i] + brow; });
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  epi_bar_set(set);
  if (issuer) {
    if (kind == EK_ADD) tma_reduce_add_2d(tmO, box, tile_n * TC_BM, m0);
    else tma_store_2d(tmO, box, kind == EK_GEGLU ? tile_n * 64 : tile_n * TC_BM, m0);
    bulk_commit();
  }
  ebuf ^= 1;
}

// The outputs of a split rank's slice: v[i] is this thread's tile row r at token
// m0+i (i < cpr <= 32), brow its bias; all 128 epilogue threads call it
// together.  Stored (or added) by the threads, a warp 128 bytes of one token per
// instruction: the slice is 4 to 16 KB, and a box in shared memory with its
// proxy fence, barriers and TMA store took 1100 to 1900 cycles of the launch's
// critical path.  xch: the idle operand ring (GeGLU's transpose).
__device__ __forceinline__ void store_slice(const TcParams& p, int tile_n, int m0, int cpr, int r, const float* v,
                                            float brow, float* xch) {
  const int lim = min(cpr, p.M - m0);   // tokens that exist (may be <= 0)
  const int n = tile_n * TC_BM + r;
  if (p.epi == EPI_GEGLU) {
    // rows 0..63 are gate features, 64..127 the matching up features: through
    // xch, every thread then forms 8 outputs of one token
#pragma unroll
    for (int g = 0; g < 32; g += 4) {
      if (g >= cpr) break;
#pragma unroll
      for (int i = g; i < g + 4; ++i) xch[i * STG_LD + r] = v[i] + brow;
    }
    epi_bar();
    #pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      const int c = (r >> 3) + 16 * h, fg = r & 7;
      if (c < lim) {
        const float4* g4 = (const float4*)(xch + c * STG_LD + fg * 8);
        const float4* u4 = (const float4*)(xch + c * STG_LD + 64 + fg * 8);
        const float4 ga = g4[0], gb = g4[1], ua = u4[0], ub = u4[1];
        *(uint4*)((bf16*)p.out + (size_t)(m0 + c) * p.ldo + tile_n * 64 + fg * 8) =
            make_uint4(pack_bf16x2(gelu_tanh_bf16out(ga.x) * ua.x, gelu_tanh_bf16out(ga.y) * ua.y),
                       pack_bf16x2(gelu_tanh_bf16out(ga.z) * ua.z, gelu_tanh_bf16out(ga.w) * ua.w),
                       pack_bf16x2(gelu_tanh_bf16out(gb.x) * ub.x, gelu_tanh_bf16out(gb.y) * ub.y),
                       pack_bf16x2(gelu_tanh_bf16out(gb.z) * ub.z, gelu_tanh_bf16out(gb.w) * ub.w));
      }
    }
  } else if (p.epi == EPI_ADD_F32) {
    float* o = (float*)p.out + (size_t)m0 * p.ldo + n;
    const bool in = n < p.N;
#pragma unroll
    for (int g = 0; g < 32; g += 4) {
      if (g >= lim) break;
#pragma unroll
      for (int i = g; i < g + 4; ++i)   // one add per element: the result does not depend on an order
        if (in && i < lim) atomicAdd(o + (size_t)i * p.ldo, v[i] + brow);
    }
  } else {
    const bool silu = p.epi == EPI_STORE_SILU;
    auto value = [&](int i) { return silu ? silu_f(v[i] + brow) : v[i] + brow; };
    if (p.out_bf16) {
      // lanes of rows r and r + 1 swap tokens i + 1 and i: each then stores both
      // rows of one token
      const bool odd = r & 1;
      bf16* o = (bf16*)p.out + (size_t)(m0 + (odd ? 1 : 0)) * p.ldo + (n & ~1);
      const bool both = (n | 1) < p.N, one = (n & ~1) < p.N;
#pragma unroll
      for (int g = 0; g < 32; g += 4) {
        if (g >= lim) break;
#pragma unroll
        for (int i = g; i < g + 4; i += 2) {
          const float a = value(i), b = value(i + 1);
          const float got = __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
          const uint32_t w = odd ? pack_bf16x2(got, b) : pack_bf16x2(a, got);
          if (i + (odd ? 1 : 0) < lim) {
            if (both) *(uint32_t*)(o + (size_t)i * p.ldo) = w;
            else if (one) *(uint16_t*)(o + (size_t)i * p.ldo) = (uint16_t)w;
          }
        }
      }
    } else {
      float* o = (float*)p.out + (size_t)m0 * p.ldo + n;
      const bool in = n < p.N;
#pragma unroll
      for (int g = 0; g < 32; g += 4) {
        if (g >= lim) break;
#pragma unroll
        for (int i = g; i < g + 4; ++i)
          if (in && i < lim) o[(size_t)i * p.ldo] = value(i);
      }
    }
  }
}

// RED, how the splits of a tile are combined, and EK, the epilogue kind, are
// fixed per instantiation, so that each reduction mode gets its own register
// allocation and each launch only the code it runs.
template <int RED, int EK>
__global__ void __launch_bounds__(TC_THREADS, 2)
    tc_gemm_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                   const __grid_constant__ CUtensorMap tmO, TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte aligned; derived from smem_raw by pointer arithmetic so that the
  // compiler keeps it (and everything indexed from it) in the shared window
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int BN = p.bn, S = p.stages;
  const uint32_t b_bytes = (uint32_t)BN * TC_BK * 2;
  uint8_t* a_s = smem;
  uint8_t* b_s = smem + (size_t)S * TC_A_BYTES;
  uint8_t* stg_raw = smem + p.stg_off;
  float* stage = (float*)stg_raw;
  float* xch = (float*)(smem + p.xch_off);
  uint64_t* full = (uint64_t*)(smem + p.bar_off);
  uint64_t* empty = full + S;
  uint64_t* acc_full = empty + S;      // [2]
  uint64_t* acc_empty = acc_full + 2;  // [2]
  uint64_t* rcv_bar = acc_empty + 2;    // RED_DSMEM*: every split's slice of this rank has arrived
  uint32_t* tmem_slot = (uint32_t*)(rcv_bar + 1);
  int* flags = (int*)(tmem_slot + 1);   // [0] abort, [2] issued, [3] consumed

  // (through a shuffle, so that the compiler knows it is uniform in the warp)
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  int tn0 = 0, tm0 = 0, sp0 = 0;
  const bool has_work = work_item(p, 0, tn0, tm0, sp0);
  const int kb0_first = (int)((long)sp0 * p.num_kb / p.splits);
  const int kb1_first = (int)((long)(sp0 + 1) * p.num_kb / p.splits);
  const int npre = has_work ? min(S, kb1_first - kb0_first) : 0;
  // the K range of an item in several accumulators, summed in the epilogue
  // (every item of a launch without splits has the same range)
  constexpr bool MULTI = RED != RED_DSMEM;
  const int accs = MULTI ? min(p.accs, kb1_first - kb0_first) : 1;
  const uint32_t item_cols = p.acc_cols * (uint32_t)p.accs;
  const int cpr = BN / p.splits;   // tokens of the slice each split rank owns (a multiple of 4)
  constexpr bool TMA_OUT = EK < EK_GENERIC;
  // partials exchanged through distributed shared memory: RED_DSMEM in bf16
  // (two rows per message), RED_DSMEM32 in fp32
  constexpr bool DSM = RED == RED_DSMEM || RED == RED_DSMEM32;

  pdl_trigger();
  uint64_t pol_w = 0, pol_x = 0;
  uint32_t el = 0;   // the issuing lane of warps 0 (TMA) and 1 (MMA)
  const uint32_t full0 = smem_u32(full), a0 = smem_u32(a_s), b0 = smem_u32(b_s);
  if (warp == 0) {
    el = elect_one();
    if (el) {
      for (int s = 0; s < S; ++s) {
        mbar_init(&full[s], 1);
        mbar_init(&empty[s], 1);
      }
      for (int b = 0; b < 2; ++b) {
        mbar_init(&acc_full[b], 1);
        mbar_init(&acc_empty[b], 128);
      }
      mbar_init(rcv_bar, 1);   // RED_DSMEM*: the partials' arrival; otherwise armed by nobody
      flags[0] = flags[2] = flags[3] = 0;
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      // the slices of all splits (this one's included): 128 rows x cpr tokens each
      if constexpr (DSM) mbar_expect_tx(rcv_bar, (uint32_t)(BN * TC_BM * (RED == RED_DSMEM ? 2 : 4)));
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      // Weights never depend on earlier kernels: stream the first stages' weight
      // tiles while the previous kernel is still finishing.
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmW) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmX) : "memory");
      if (TMA_OUT) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmO) : "memory");
    }
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol_w));
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_x));
    __syncwarp();
  }
  // A launch that may be skipped at run time (p.skip) issues nothing before
  // it has read its flag after the wait; every other launch streams its first
  // weight tiles now, while the previous kernel is still finishing.
  auto issue_weight_prologue = [&]() {   // warp 0
    if (p.oneshot) {
      // every weight k-tile of this CTA in one box; the token k-tiles follow
      // after the wait into the same barrier
      // (the boxes are S = the largest split's k-tile count deep; a shorter
      // split ignores the extra tile)
      mbar_expect_tx_el(&full[0], (uint32_t)S * (TC_A_BYTES + b_bytes), el);
      tma_load_3d_el(&tmW, full0, a0, 0, tn0 * TC_BM, kb0_first, pol_w, el);
    } else {
      #pragma unroll 1
      for (int i = 0; i < npre; ++i) {
        mbar_expect_tx_el(&full[i], TC_A_BYTES + b_bytes, el);
        tma_load_2d_el(&tmW, full0 + 8u * (uint32_t)i, a0 + (uint32_t)i * TC_A_BYTES, (kb0_first + i) * TC_BK,
                       tn0 * TC_BM, pol_w, el);
      }
      // a split CTA has one short K range: the rest of its weight slice goes
      // to L2 now, so that after the wait every operand load is an L2 hit
      if (p.splits > 1) {
        #pragma unroll 1
        for (int kb = kb0_first + npre; kb < kb1_first; ++kb) prefetch_l2_2d_el(&tmW, kb * TC_BK, tn0 * TC_BM, el);
      }
    }
  };
  if (warp == 0 && !p.skip) issue_weight_prologue();
  // RED_DSMEM*: this CTA's receive barrier is armed; the epilogue warps wait for
  // the whole cluster's before they send
  if constexpr (DSM) cluster_arrive_release();
  // everything below may read what earlier kernels wrote; TMEM is taken only
  // now, so a CTA waiting here never holds columns its predecessor needs
  pdl_wait();
  if (p.skip) {
    // nothing is in flight yet; the flag is the same for every CTA
    if (*p.skip) return;
    if (warp == 0) issue_weight_prologue();
  }
  if (warp == 0) {
    // the tokens of the stages whose weights are on their way: before the
    // TMEM set-up, which they do not need
    if (p.oneshot) {
      tma_load_3d_el(&tmX, full0, b0, 0, tm0 * BN, kb0_first, pol_x, el);
    } else {
      #pragma unroll 1
      for (int i = 0; i < npre; ++i)
        tma_load_2d_el(&tmX, full0 + 8u * (uint32_t)i, b0 + (uint32_t)i * b_bytes, (kb0_first + i) * TC_BK, tm0 * BN,
                       pol_x, el);
    }
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(p.ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cta_sync();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    int it = p.oneshot ? 1 : npre;   // stages issued, across all work items
    if (!p.oneshot && has_work) {
      int s = npre == S ? 0 : npre;          // ring position and the parity its `empty` wait takes
      uint32_t ph = npre == S ? 0u : 1u;
      bool ok = true;
      int tn = tn0, tm = tm0, sp = sp0, i = 0;
      int kb = kb0_first + npre, kb1 = kb1_first;
      while (true) {
        #pragma unroll 1
        for (; kb < kb1; ++kb, ++it) {
          ok = mbar_wait_warp(&empty[s], ph, p.wait_ns);
          if (!ok) break;
          mbar_expect_tx_el(&full[s], TC_A_BYTES + b_bytes, el);
          tma_load_2d_el(&tmW, full0 + 8u * (uint32_t)s, a0 + (uint32_t)s * TC_A_BYTES, kb * TC_BK, tn * TC_BM, pol_w,
                         el);
          tma_load_2d_el(&tmX, full0 + 8u * (uint32_t)s, b0 + (uint32_t)s * b_bytes, kb * TC_BK, tm * BN, pol_x, el);
          if (++s == S) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!ok || !work_item(p, ++i, tn, tm, sp)) break;
        kb = (int)((long)sp * p.num_kb / p.splits);
        kb1 = (int)((long)(sp + 1) * p.num_kb / p.splits);
      }
      if (!ok && lane == 0) flags[0] = 1;
    }
    if (lane == 0) flags[2] = it;
    __syncwarp();
  } else if (warp == 1) {
    el = elect_one();
    const uint32_t idesc = idesc_bf16(TC_BM, BN);
    const uint64_t ad0 = sw128_desc(a0), bd0 = sw128_desc(b0);
    // accumulator j takes acc_q k-tiles, the first acc_r of them one more
    const int cnt = kb1_first - kb0_first, acc_q = accs > 1 ? cnt / accs : cnt, acc_r = accs > 1 ? cnt - acc_q * accs : 0;
    int it = 0;
    bool ok = true;
    // fault injection: an arrival that never comes (rcv_bar is armed by
    // nobody outside the RED_DSMEM modes, which the host never combines with this)
    if (p.withhold) ok = mbar_wait_warp(rcv_bar, 0, p.wait_ns);
    if (ok && p.oneshot) {   // one item, every k-tile behind one barrier
      ok = mbar_wait_warp(&full[0], 0, p.wait_ns);
      if (ok) {
        tc_fence_after();
        uint64_t ad = ad0, bd = bd0;
        int j = 0, first = 0, next = acc_q + (acc_r > 0 ? 1 : 0);   // accumulator j takes k-tiles [first, next)
        uint32_t d = tmem;
        #pragma unroll 1
        for (int kb = 0; kb < cnt; ++kb, ad += TC_A_BYTES >> 4, bd += b_bytes >> 4) {
          if (MULTI && kb == next) {
            first = kb;
            next += acc_q + (++j < acc_r ? 1 : 0);
            d += p.acc_cols;
          }
#pragma unroll
          for (int k = 0; k < TC_BK / 16; ++k)
            umma_bf16(d, ad + 2 * k, bd + 2 * k, idesc, (kb > first || k > 0) ? 1u : 0u, el);
        }
        umma_commit(&acc_full[0], el);
        it = 1;
      }
    }
    int tn, tm, sp, s = 0;
    uint32_t ph = 0, aoff = 0, boff = 0;   // ring position: parity and descriptor offsets of stage s
    for (int i = 0; !p.oneshot && ok && work_item(p, i, tn, tm, sp); ++i) {
      const int b = i & 1;
      // the accumulator of item i - 2 must have been drained by the epilogue
      if (i >= 2) ok = mbar_wait_warp(&acc_empty[b], (uint32_t)((i >> 1) - 1) & 1u, p.wait_ns);
      if (!ok) break;
      tc_fence_after();
      uint32_t d = tmem + (uint32_t)b * item_cols;
      const int kb0 = (int)((long)sp * p.num_kb / p.splits), kb1 = (int)((long)(sp + 1) * p.num_kb / p.splits);
      int j = 0, first = kb0, next = kb0 + acc_q + (acc_r > 0 ? 1 : 0);   // as above
      #pragma unroll 1
      for (int kb = kb0; kb < kb1; ++kb, ++it) {
        if (MULTI && kb == next) {
          first = kb;
          next += acc_q + (++j < acc_r ? 1 : 0);
          d += p.acc_cols;
        }
        ok = mbar_wait_warp(&full[s], ph, p.wait_ns);
        if (!ok) break;
        tc_fence_after();
        const uint64_t ad = ad0 + aoff, bd = bd0 + boff;
#pragma unroll
        for (int k = 0; k < TC_BK / 16; ++k)
          umma_bf16(d, ad + 2 * k, bd + 2 * k, idesc, (kb > first || k > 0) ? 1u : 0u, el);
        umma_commit(&empty[s], el);
        aoff += TC_A_BYTES >> 4;
        boff += b_bytes >> 4;
        if (++s == S) {
          s = 0;
          ph ^= 1u;
          aoff = boff = 0;
        }
      }
      if (!ok) break;
      umma_commit(&acc_full[b], el);   // arrives once every MMA issued above has completed
    }
    if (lane == 0) {
      if (!ok) flags[0] = 1;
      flags[3] = it;
    }
    __syncwarp();
  } else {
    // epilogue warps 2..5: TMEM lane quarter q = warp % 4, tile row r
    const int q = warp & 3;
    const int r = q * 32 + lane;
    int ebuf = 0;   // TMA output box in use
    int tn, tm, sp;
    for (int i = 0; work_item(p, i, tn, tm, sp); ++i) {
      const int b = i & 1;
      const bool ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[b], (uint32_t)(i >> 1) & 1u, p.wait_ns));
      if constexpr (DSM) cluster_wait_acquire();   // every CTA of the cluster has armed its receive barrier
      if (!ok) {
        if (lane == 0) flags[0] = 1;
        break;
      }
      tc_fence_after();
      const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)b * item_cols;
      const int m_base = tm * BN;
      const int n = tn * TC_BM + r;
      const float brow = (p.bias && n < p.N) ? p.bias[n] : 0.f;
      if constexpr (RED == RED_NONE) {
        // 16-token chunks; the TMEM load of chunk c+1 is in flight while chunk
        // c goes out
        uint32_t nxt[16];
        tmem_ld16_async(trow, nxt);
        tmem_wait_ld();
        tmem_reg_fence16(nxt);
        #pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 16) {
          float v[16];
          add_accumulators(trow + c0, p.acc_cols, accs, nxt);
#pragma unroll
          for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(nxt[k]);
          const bool more = c0 + 16 < BN;
          if (more) {
            tmem_ld16_async(trow + c0 + 16, nxt);
          } else {   // accumulator drained: the MMA warp may reuse it
            tc_fence_before();
            mbar_arrive(&acc_empty[b]);
          }
          if constexpr (TMA_OUT) epilogue_tma<EK>(p, &tmO, tn, m_base + c0, r, v, brow, stg_raw, xch, ebuf);
          else epilogue_chunk(p, tn, m_base + c0, 16, r, v, stage);
          if (more) {
            tmem_wait_ld();
            tmem_reg_fence16(nxt);
          }
        }
      } else if constexpr (RED == RED_DSMEM) {
        // token slice q of this split's partial goes to rank q (= split q) of
        // the cluster in bf16, two rows per 16-byte message: the lanes of rows
        // r and r+1 swap halves of their packed 4-token groups 2k and 2k+1,
        // so that the even lane sends group 2k of both rows and the odd lane
        // group 2k+1; group g of the slice for row pair r/2 lands at
        // [sp][g][r/2] there
        const int ngs = cpr / 4;
        const bool odd = lane & 1;
        const uint32_t rcv0 = smem_u32(smem + p.rcv_off) + (uint32_t)(sp * ngs * 64 + (r >> 1)) * 16u;
        const uint32_t bar0 = smem_u32(rcv_bar);
        // destination rank and group of this lane's next message (group 2k + odd)
        int dst = (odd && ngs == 1) ? 1 : 0, gl = (odd && ngs > 1) ? 1 : 0;
        #pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 64) {   // up to four TMEM loads in flight, one wait
          const int nq = min(4, (BN - c0) / 16);   // BN is a multiple of 16
          uint32_t raw[64];
#pragma unroll
          for (int qq = 0; qq < 4; ++qq)
            if (qq < nq) tmem_ld16_async(trow + c0 + 16 * qq, raw + 16 * qq);
          tmem_wait_ld();
#pragma unroll
          for (int qq = 0; qq < 4; ++qq) tmem_reg_fence16(raw + 16 * qq);
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            if (k >= 2 * nq) break;
            const uint32_t* a = raw + 8 * k;
            const uint32_t p0 = pack_bf16x2(__uint_as_float(a[0]), __uint_as_float(a[1]));
            const uint32_t p1 = pack_bf16x2(__uint_as_float(a[2]), __uint_as_float(a[3]));
            const uint32_t p2 = pack_bf16x2(__uint_as_float(a[4]), __uint_as_float(a[5]));
            const uint32_t p3 = pack_bf16x2(__uint_as_float(a[6]), __uint_as_float(a[7]));
            const uint32_t got0 = __shfl_xor_sync(0xffffffffu, odd ? p0 : p2, 1);
            const uint32_t got1 = __shfl_xor_sync(0xffffffffu, odd ? p1 : p3, 1);
            const uint4 w = odd ? make_uint4(got0, got1, p2, p3) : make_uint4(p0, p1, got0, got1);
            const uint32_t to = mapa_shared(rcv0, (uint32_t)dst);
            st_async_u4(to + (uint32_t)gl * 1024u, w, to + (bar0 - rcv0));
            // two groups on: a select per rank boundary, not a branch
            gl += 2;
            bool wrap = gl >= ngs;
            gl = wrap ? gl - ngs : gl;
            dst += wrap ? 1 : 0;
            wrap = gl >= ngs;
            gl = wrap ? gl - ngs : gl;
            dst += wrap ? 1 : 0;
          }
        }
      } else if constexpr (RED == RED_DSMEM32) {
        // token slice q of this split's partial goes to rank q (= split q) of
        // the cluster: float4 group g of the slice lands at [sp][g][r] there
        const int ngs = cpr / 4;
        const uint32_t rcv0 = smem_u32(smem + p.rcv_off) + (uint32_t)(sp * ngs * TC_BM + r) * 16u;
        const uint32_t bar0 = smem_u32(rcv_bar);
        int dst = 0, gl = 0;   // destination rank and group of the next float4
        #pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 64) {   // up to four TMEM loads in flight, one wait
          const int nq = min(4, (BN - c0) / 16);   // BN is a multiple of 16
          uint32_t raw[64];
#pragma unroll
          for (int qq = 0; qq < 4; ++qq)
            if (qq < nq) tmem_ld16_async(trow + c0 + 16 * qq, raw + 16 * qq);
          tmem_wait_ld();
#pragma unroll
          for (int qq = 0; qq < 4; ++qq) tmem_reg_fence16(raw + 16 * qq);
#pragma unroll
          for (int qq = 0; qq < 4; ++qq)
            if (qq < nq) add_accumulators(trow + c0 + 16 * qq, p.acc_cols, accs, raw + 16 * qq);
#pragma unroll
          for (int qq = 0; qq < 16; ++qq) {
            if (qq >= 4 * nq) break;
            st_async_f4(mapa_shared(rcv0 + (uint32_t)gl * (TC_BM * 16), (uint32_t)dst),
                        make_float4(__uint_as_float(raw[4 * qq]), __uint_as_float(raw[4 * qq + 1]),
                                    __uint_as_float(raw[4 * qq + 2]), __uint_as_float(raw[4 * qq + 3])),
                        mapa_shared(bar0, (uint32_t)dst));
            const bool wrap = ++gl == ngs;   // next rank: a select, not a branch
            gl = wrap ? 0 : gl;
            dst += wrap ? 1 : 0;
          }
        }
      } else {   // RED_L2_CLUSTER
        // this split's fp32 partial to the workspace as [col/4][row][4]: each
        // thread stores float4 of 4 consecutive columns, a warp one 512-byte run
        const size_t cl = (size_t)tm * gridDim.x + tn;
        float* w = p.ws + ((cl * p.splits + sp) * (size_t)(BN / 4)) * (TC_BM * 4) + (size_t)r * 4;
        #pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 64) {   // up to four TMEM loads in flight, one wait
          const int nq = min(4, (BN - c0) / 16);   // BN is a multiple of 16
          uint32_t raw[64];
#pragma unroll
          for (int qq = 0; qq < 4; ++qq)
            if (qq < nq) tmem_ld16_async(trow + c0 + 16 * qq, raw + 16 * qq);
          tmem_wait_ld();
#pragma unroll
          for (int qq = 0; qq < 4; ++qq) tmem_reg_fence16(raw + 16 * qq);
#pragma unroll
          for (int qq = 0; qq < 4; ++qq)
            if (qq < nq) add_accumulators(trow + c0 + 16 * qq, p.acc_cols, accs, raw + 16 * qq);
#pragma unroll
          for (int qq = 0; qq < 16; ++qq)
            if (qq < 4 * nq)
              __stcg((float4*)(w + (size_t)(c0 / 4 + qq) * (TC_BM * 4)),
                     make_float4(__uint_as_float(raw[4 * qq]), __uint_as_float(raw[4 * qq + 1]),
                                 __uint_as_float(raw[4 * qq + 2]), __uint_as_float(raw[4 * qq + 3])));
        }
        __threadfence();
      }
    }
    // every TMA output box has been read out of shared memory (the grid's
    // completion makes the writes visible to the dependent launch)
    if (TMA_OUT && threadIdx.x == 64) bulk_wait_read<0>();
  }
  tc_fence_before();
  cta_sync();
  if (flags[0]) {
    // unwind: wait (bounded) for the copies this CTA issued but never consumed
    if (threadIdx.x == 0) {
      for (int i = flags[3]; i < flags[2]; ++i) mbar_wait(&full[i % S], (uint32_t)(i / S) & 1u);
      raise_error(p.err, ERR_TIMEOUT);
    }
    cta_sync();
  }
  if constexpr (DSM) {
    // Rank q sums its slice of tokens [q*cpr, (q+1)*cpr) over the splits in
    // order once every split's bytes have arrived (the wait also keeps this
    // CTA alive until no store into its shared memory is in flight), then
    // stores the slice from the threads (store_slice).
    if (warp >= 2) {
      const int r = (warp & 3) * 32 + lane;
      const bool ok = __all_sync(0xffffffffu, mbar_wait_cluster(rcv_bar, 0, p.wait_ns));
      if (!ok) {
        if (lane == 0) raise_error(p.err, ERR_TIMEOUT);
      } else {
        const int n = tn0 * TC_BM + r;
        const float brow = (p.bias && n < p.N) ? p.bias[n] : 0.f;
        float v[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = 0.f;
        if constexpr (RED == RED_DSMEM) {
          const uint2* b0 = (const uint2*)(smem + p.rcv_off) + 2 * (r >> 1) + (r & 1);
          switch (cpr / 4) {
            case 1: reduce_slice_smem<1>(b0, p.splits, v); break;
            case 2: reduce_slice_smem<2>(b0, p.splits, v); break;
            case 3: reduce_slice_smem<3>(b0, p.splits, v); break;
            case 4: reduce_slice_smem<4>(b0, p.splits, v); break;
            case 5: reduce_slice_smem<5>(b0, p.splits, v); break;
            case 6: reduce_slice_smem<6>(b0, p.splits, v); break;
            case 7: reduce_slice_smem<7>(b0, p.splits, v); break;
            default: reduce_slice_smem<8>(b0, p.splits, v); break;
          }
        } else {
          const float4* b0 = (const float4*)(smem + p.rcv_off) + r;
          switch (cpr / 4) {
            case 1: reduce_slice_smem<1>(b0, p.splits, v); break;
            case 2: reduce_slice_smem<2>(b0, p.splits, v); break;
            case 3: reduce_slice_smem<3>(b0, p.splits, v); break;
            case 4: reduce_slice_smem<4>(b0, p.splits, v); break;
            case 5: reduce_slice_smem<5>(b0, p.splits, v); break;
            case 6: reduce_slice_smem<6>(b0, p.splits, v); break;
            case 7: reduce_slice_smem<7>(b0, p.splits, v); break;
            default: reduce_slice_smem<8>(b0, p.splits, v); break;
          }
        }
        store_slice(p, tn0, tm0 * BN + sp0 * cpr, cpr, r, v, brow, (float*)smem);
      }
    }
  }
  if constexpr (RED == RED_L2_CLUSTER) {
    // Every split of this tile has written its partial; the cluster barrier
    // (release / acquire) makes them visible.  Rank q sums columns
    // [q*BN/S, (q+1)*BN/S) over the splits in order and applies the epilogue.
    cluster_sync();
    if (warp >= 2) {
      const int r = (warp & 3) * 32 + lane;
      const int Sp = p.splits;
      const int rank = (int)cluster_ctarank();
      const size_t cl = (size_t)tm0 * gridDim.x + tn0;
      const float* base = p.ws + (cl * Sp * (size_t)(BN / 4) + rank * cpr / 4) * (TC_BM * 4) + (size_t)r * 4;
      const size_t sstride = (size_t)(BN / 4) * (TC_BM * 4);
      #pragma unroll 1
      for (int cc = 0; cc < cpr; cc += p.box_m) {
        const int nc = p.box_m;
        float v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = 0.f;
        const float* b0 = base + (size_t)(cc / 4) * (TC_BM * 4);
        if (nc == 16) reduce_splits_l2<4>(b0, Sp, sstride, v);
        else if (nc == 8) reduce_splits_l2<2>(b0, Sp, sstride, v);
        else reduce_splits_l2<1>(b0, Sp, sstride, v);
        epilogue_chunk(p, tn0, tm0 * BN + rank * cpr + cc, nc, r, v, stage);
      }
    }
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.ncols) : "memory");
  }
}


// ---------------------------------------------------------------------------
// Two-SM GEMM (persistent, many tiles): a pair of CTAs (a cluster of 2) runs
// one M = 256 MMA per K step -- A = 256 weight rows, 128 in each CTA's shared
// memory, B = BN tokens, BN / 2 in each -- and each CTA's TMEM accumulates its
// own 128 rows for all BN tokens.  Per K step an SM then streams 128 + BN/2
// operand rows through TMA and the MMA instead of 128 + BN, which is what
// bounds the one-SM tile's main loop.  The even CTA's thread issues the MMAs
// and owns the stage barriers: both CTAs load their halves into their own
// shared memory and count the bytes on the even CTA's `full` barrier; the
// MMA completion is multicast to both CTAs' `empty` / `acc_full` barriers;
// both CTAs run the epilogue of their own rows, whose drained accumulators
// the even CTA's `acc_empty` counts (512 arrivals, 256 epilogue threads each).
template <int EK>
__global__ void __launch_bounds__(TC_PAIR_THREADS, 1)
    tc_gemm_pair_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                        const __grid_constant__ CUtensorMap tmO, TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte aligned; derived from smem_raw by pointer arithmetic so that the
  // compiler keeps it (and everything indexed from it) in the shared window
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int BN = p.bn, BNh = BN / 2, S = p.stages;
  const uint32_t bh_bytes = (uint32_t)BNh * TC_BK * 2;
  const uint32_t stage_tx = 2u * (TC_A_BYTES + bh_bytes);   // both CTAs' halves of a stage
  uint8_t* a_s = smem;
  uint8_t* b_s = smem + (size_t)S * TC_A_BYTES;
  uint8_t* stg_raw = smem + p.stg_off;
  float* xch = (float*)(smem + p.xch_off);
  uint64_t* full = (uint64_t*)(smem + p.bar_off);   // the even CTA's count both halves
  uint64_t* empty = full + S;
  uint64_t* acc_full = empty + S;      // [2]
  uint64_t* acc_empty = acc_full + 2;  // [2] the even CTA's: 512 arrivals (256 epilogue threads per CTA)
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 2);
  int* flags = (int*)(tmem_slot + 1);  // [0] abort, [2] stages issued, [3] stages consumed

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int pair = (int)(blockIdx.x >> 1), npairs = (int)(gridDim.x >> 1);
  // work item i of this pair: pair tile pair + i * npairs = (256-row block tn2, token tile tm)
  auto item = [&](int i, int& tn2, int& tm) -> bool {
    const int t = pair + i * npairs;
    if (t >= p.num_tiles) return false;
    tm = t % p.tiles_m;
    tn2 = t / p.tiles_m;
    return true;
  };
  int tn0 = 0, tm0 = 0;
  const bool has_work = item(0, tn0, tm0);
  const int npre = has_work ? min(S, p.num_kb) : 0;
  constexpr bool TMA_OUT = EK != EK_GENERIC;
  static_assert(TMA_OUT, "the pair kernel stores through TMA boxes");

  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 512);
    }
    flags[0] = flags[2] = flags[3] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // both CTAs' barriers exist before either signals the other's
  cluster_sync();
  const uint32_t full0 = mapa_shared(smem_u32(full), 0);          // the even CTA's full[0]
  const uint32_t acc_empty0 = mapa_shared(smem_u32(acc_empty), 0);
  uint64_t pol_w = 0, pol_x = 0;
  uint32_t el = 0;   // the issuing lane of warps 0 (TMA) and 1 (MMA)
  const uint32_t a0 = smem_u32(a_s), b0 = smem_u32(b_s);
  if (warp == 0) {
    el = elect_one();
    if (el) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmW) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmX) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmO) : "memory");
    }
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol_w));
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_x));
    __syncwarp();
  }
  const uint32_t el_lead = leader ? el : 0u;   // the even CTA's issuing lane
  // the first stages' weight halves, before the wait on the previous kernel
  // (after it, for a launch that may be skipped at run time)
  auto issue_weight_prologue = [&]() {   // warp 0
    #pragma unroll 1
    for (int i = 0; i < npre; ++i) {
      mbar_expect_tx_el(&full[i], stage_tx, el_lead);
      tma_load_2d_pair_el(&tmW, full0 + 8u * (uint32_t)i, a0 + (uint32_t)i * TC_A_BYTES, i * TC_BK,
                          (2 * tn0 + (int)rank) * TC_BM, pol_w, el);
    }
  };
  if (warp == 0 && !p.skip) issue_weight_prologue();
  pdl_wait();
  if (p.skip) {
    // nothing has been issued yet and the flag is the same for both CTAs of
    // the pair: they leave together, with no copy or arrival in flight
    if (*p.skip) return;
    if (warp == 0) issue_weight_prologue();
  }
  if (warp == 0) {   // their token halves, before the TMEM set-up
    #pragma unroll 1
    for (int i = 0; i < npre; ++i)
      tma_load_2d_pair_el(&tmX, full0 + 8u * (uint32_t)i, b0 + (uint32_t)i * bh_bytes, i * TC_BK,
                          tm0 * BN + (int)rank * BNh, pol_x, el);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(p.ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cta_sync();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {   // producer (both CTAs): this CTA's A rows and B half of each stage
    int it = npre;
    if (has_work) {
      int s = npre == S ? 0 : npre;   // ring position and the parity its `empty` wait takes
      uint32_t ph = npre == S ? 0u : 1u;
      bool ok = true;
      int tn2 = tn0, tm = tm0, i = 0, kb = npre;
      while (true) {
        #pragma unroll 1
        for (; kb < p.num_kb; ++kb, ++it) {
          ok = mbar_wait_warp(&empty[s], ph);
          if (!ok) break;
          const uint32_t fb = full0 + 8u * (uint32_t)s;
          mbar_expect_tx_el(&full[s], stage_tx, el_lead);
          tma_load_2d_pair_el(&tmW, fb, a0 + (uint32_t)s * TC_A_BYTES, kb * TC_BK, (2 * tn2 + (int)rank) * TC_BM,
                              pol_w, el);
          tma_load_2d_pair_el(&tmX, fb, b0 + (uint32_t)s * bh_bytes, kb * TC_BK, tm * BN + (int)rank * BNh, pol_x, el);
          if (++s == S) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!ok || !item(++i, tn2, tm)) break;
        kb = 0;
      }
      if (!ok && lane == 0) flags[0] = 1;
    }
    if (lane == 0) flags[2] = it;
    __syncwarp();
  } else if (warp == 1) {
    if (leader) {   // MMA issuer: the even CTA only
      el = elect_one();
      const uint32_t idesc = idesc_bf16(2 * TC_BM, BN);
      const uint64_t ad0 = sw128_desc(a0), bd0 = sw128_desc(b0);
      int it = 0, s = 0;
      uint32_t ph = 0, aoff = 0, boff = 0;   // ring position: parity and descriptor offsets of stage s
      bool ok = true;
      int tn2, tm;
      for (int i = 0; ok && item(i, tn2, tm); ++i) {
        const int b = i & 1;
        // both CTAs' epilogues must have drained the accumulator of item i - 2
        if (i >= 2) ok = mbar_wait_warp(&acc_empty[b], (uint32_t)((i >> 1) - 1) & 1u);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)b * p.acc_cols;
        #pragma unroll 1
        for (int kb = 0; kb < p.num_kb; ++kb, ++it) {
          ok = mbar_wait_warp(&full[s], ph);
          if (!ok) break;
          tc_fence_after();
          const uint64_t ad = ad0 + aoff, bd = bd0 + boff;
#pragma unroll
          for (int k = 0; k < TC_BK / 16; ++k)
            umma_bf16_pair(d, ad + 2 * k, bd + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u, el);
          umma_commit_pair_mc(&empty[s], 3, el);   // both CTAs' halves of the stage are free
          aoff += TC_A_BYTES >> 4;
          boff += bh_bytes >> 4;
          if (++s == S) {
            s = 0;
            ph ^= 1u;
            aoff = boff = 0;
          }
        }
        if (ok) umma_commit_pair_mc(&acc_full[b], 3, el);
      }
      if (lane == 0) {
        if (!ok) flags[0] = 1;
        flags[3] = it;
      }
    }
    __syncwarp();
  } else {
    // epilogue warps 2..9 of both CTAs: TMEM lane quarter q, this CTA's tile
    // row r; set 0 (warps 2..5) takes the 32-token chunks 0, 2, 4, ..., set 1
    // (warps 6..9) chunks 1, 3, 5, ..., each with its own boxes and barrier
    const int q = warp & 3;
    const int r = q * 32 + lane;
    const int set = warp >= 6 ? 1 : 0;
    uint8_t* sboxes = stg_raw + (size_t)set * p.set_bytes;
    float* sxch = (float*)((uint8_t*)xch + (size_t)set * p.set_bytes);
    int ebuf = 0;
    int tn2, tm;
    for (int i = 0; item(i, tn2, tm); ++i) {
      const int b = i & 1;
      const bool ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[b], (uint32_t)(i >> 1) & 1u));
      if (!ok) {
        if (lane == 0) flags[0] = 1;
        break;
      }
      tc_fence_after();
      const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)b * p.acc_cols;
      const int tile_n = 2 * tn2 + (int)rank;   // this CTA's 128-row block
      const int m_base = tm * BN;
      const int n = tile_n * TC_BM + r;
      const float brow = (p.bias && n < p.N) ? p.bias[n] : 0.f;
      // 32-token chunks (BN is a multiple of 32, at least 64): this set's
      // every other chunk, the next one's TMEM load in flight meanwhile
      uint32_t nxt[32];
      const int cf = 32 * set;
      tmem_ld32_async(trow + cf, nxt);
      tmem_wait_ld();
      tmem_reg_fence16(nxt);
      tmem_reg_fence16(nxt + 16);
      for (int c0 = cf; c0 < BN; c0 += 64) {
        float v[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(nxt[k]);
        const bool more = c0 + 64 < BN;
        if (more) {
          tmem_ld32_async(trow + c0 + 64, nxt);
        } else {   // this thread is done with the accumulator: tell the MMA issuer
          tc_fence_before();
          mbar_arrive_remote(acc_empty0 + 8u * (uint32_t)b);
        }
        epilogue_tma<EK, 32>(p, &tmO, tile_n, m_base + c0, r, v, brow, sboxes, sxch, ebuf);
        if (more) {
          tmem_wait_ld();
          tmem_reg_fence16(nxt);
          tmem_reg_fence16(nxt + 16);
        }
      }
    }
    if (threadIdx.x == 64 + 128 * set) bulk_wait_read<0>();   // this set's boxes have been read out
  }
  tc_fence_before();
  cta_sync();
  if (flags[0]) {
    // unwind: the even CTA waits (bounded) for stages issued but never consumed
    if (threadIdx.x == 0) {
      if (leader)
        for (int i = flags[3]; i < flags[2]; ++i) mbar_wait(&full[i % S], (uint32_t)(i / S) & 1u);
      raise_error(p.err, ERR_TIMEOUT);
    }
    cta_sync();
  }
  // neither CTA leaves while the other may still signal its barriers or
  // (through the MMA) read its shared memory
  cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.ncols) : "memory");
  }
}

using TcKernel = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, TcParams);

TcKernel tc_pair_kernel(int ek) {
  switch (ek) {
    case EK_F32: return tc_gemm_pair_kernel<EK_F32>;
    case EK_BF16: return tc_gemm_pair_kernel<EK_BF16>;
    case EK_ADD: return tc_gemm_pair_kernel<EK_ADD>;
    case EK_GEGLU: return tc_gemm_pair_kernel<EK_GEGLU>;
    default: return nullptr;
  }
}

// The instantiation for a reduction mode and epilogue kind (nullptr where the
// two cannot occur together: the shared-memory exchange needs TMA outputs).
TcKernel tc_kernel(int red, int ek) {
#define RAVEL_TC_K(R, E) \
  if (red == R && ek == E) return tc_gemm_kernel<R, E>;
  RAVEL_TC_K(RED_NONE, EK_F32) RAVEL_TC_K(RED_NONE, EK_BF16) RAVEL_TC_K(RED_NONE, EK_ADD)
  RAVEL_TC_K(RED_NONE, EK_GEGLU) RAVEL_TC_K(RED_NONE, EK_GENERIC)
  RAVEL_TC_K(RED_L2_CLUSTER, EK_GENERIC)
  RAVEL_TC_K(RED_DSMEM, EK_SLICE) RAVEL_TC_K(RED_DSMEM32, EK_SLICE)
#undef RAVEL_TC_K
  return nullptr;
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

cudaError_t get_encoder() {
  if (g_encode) return cudaSuccess;
  cudaDriverEntryPointQueryResult q;
  void* fn = nullptr;
  cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
  if (e != cudaSuccess) return e;
  if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorSymbolNotFound;
  g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
  return cudaSuccess;
}

// 2D bf16 map over a row-major [rows][cols] matrix (row stride ld elements),
// box = box_rows x 64 columns, 128-byte swizzle, zero fill out of bounds.
cudaError_t encode_2d(CUtensorMap* m, const void* base, int rows, int cols, int ld, int box_rows) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)TC_BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// 3D map over a row-major bf16 [rows][cols] matrix (cols a multiple of 64)
// viewed as (64 elements, rows, cols / 64 k-tiles): a box of box_rows x nkb
// lands as nkb consecutive K-major 128-byte-swizzled tiles of box_rows rows.
cudaError_t encode_kt(CUtensorMap* m, const void* base, int rows, int cols, int ld, int box_rows, int nkb) {
  cuuint64_t dims[3] = {(cuuint64_t)TC_BK, (cuuint64_t)rows, (cuuint64_t)(cols / TC_BK)};
  cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)TC_BK * 2};
  cuuint32_t box[3] = {(cuuint32_t)TC_BK, (cuuint32_t)box_rows, (cuuint32_t)nkb};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// 2D map over a row-major output [rows][cols] (row stride ld elements) for
// TMA stores: box = box_cols x box_rows, no swizzle (the box is dense in
// shared memory), writes past the extents clipped.
cudaError_t encode_out(CUtensorMap* m, void* base, int rows, int cols, int ld, bool bf, int box_cols, int box_rows) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * (bf ? 2 : 4)};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(m, bf ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims,
                        strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                        CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

std::atomic<int> g_withhold{0};   // launches left to run with a withheld arrival (fault injection)
constexpr unsigned long long kWithholdWaitNs = 2000000ull;   // their wait limit: 2 ms

// Resident clusters of 2, 4, 8, 16 split CTAs (one CTA per SM; 0: that
// cluster size is not to be had).  The split-K kernels take a whole SM each,
// and clusters stay inside a GPC: 76, 36, 15 and 7 on this part.
struct TcClusters {
  int n[4];
};
TcClusters g_max_clusters = {{0, 0, 0, 0}};

// Whether a step's launch (xbf16) exchanges its splits' shares in bf16: where
// tiles of 64 (M <= 64) or 128 tokens leave so many SMs idle that a split's slice
// is at most 32 tokens, and that many splits have a k-tile each.  Elsewhere
// shares stay fp32, whatever the plan: a share in bf16 costs a sum up to 2^-8 of
// the share, and the estimated time is no reason to take that where it was not taken
// (QKV of 2560 features from 129 tokens on, O and down of 1024 from 513 on).
bool bf16_shares(const GemmArgs& g, int num_sms) {
  const int s = g.M <= 64 ? 2 : 4;
  const long tiles = (long)((g.N + TC_BM - 1) / TC_BM) * ((g.M + 127) / 128);
  return g.xbf16 && tiles * s <= num_sms && (g.K + TC_BK - 1) / TC_BK >= s;
}

// Tokens per chunk of a split's slice of cpr tokens (a multiple of 4).
int split_chunk(int cpr) { return cpr % 16 == 0 ? 16 : cpr % 8 == 0 ? 8 : 4; }

// How a GEMM is cut: token-tile width, K splits (a cluster), or SM pairs.
struct TcPlan {
  bool pair = false;
  int bn = 0, splits = 1;
};

// The plan of least estimated time.  The estimate, in microseconds, was fitted
// to 3,900 measured launches (a chain of dependent launches with weights from
// HBM; N x K of 2560 x 1024, 1024 x 2048, 8192 x 1024, 1024 x 4096, 1536 x
// 1024, 1024 x 1024, 2048 x 1024 and 75776 x 1024, 8 to 4224 tokens, all
// widths and splits): a launch costs a fixed 2.6 (SM pairs: 3.4), its
// epilogue grows with the tile width (GeGLU's more), a k-tile takes as long as
// its operands need to arrive (168 GB/s per SM, 142 in pairs, whose MMA then
// needs 0.295 at 256 tokens), splits add their exchange, and clusters that do
// not fit at once add a wave.  Over the measured shapes the plan chosen is
// 0.7 % slower than the best measured one; the widest-tile-and-most-splits
// rule before it was 19 % slower (M 50 x N 1024 x K 2048: 16 splits, 5.9 us;
// now 4.1 us; M 240 x 1024 x 4096: 12.4, now 7.3 us).  Inside a step (xbf16)
// the neighbours of a launch are other kernels: there the exchange of bf16
// shares, where bf16_shares allows it, weighs less, an unsplit launch 0.3 more
// (its code is another binary's than the split launches'), and split CTAs past
// half the SMs, which the next kernel could have started on, up to 0.7 more.
// Whole steps at 1 to 64 robots, each projection's width and splits varied in
// turn: the rule is 0 to 3.5 % of the step away from the best combination
// (batch 1 at it: 652 us, 685 with the chain's terms alone).
TcPlan plan_gemm(const GemmArgs& g, bool dsmem, size_t ws_bytes, bool pairs, int num_sms, const TcClusters& clusters) {
  const int M = g.M, N = g.N, K = g.K;
  const bool geglu = g.epi == EPI_GEGLU, xbf16 = g.xbf16 != 0, shares_bf16 = bf16_shares(g, num_sms);
  const int tiles_n = (N + TC_BM - 1) / TC_BM, num_kb = (K + TC_BK - 1) / TC_BK;
  TcPlan best;
  float cost = 3.4e38f;
  auto consider = [&](bool pair, int bn, int splits, float t) {
    if (t < cost) {
      cost = t;
      best.pair = pair;
      best.bn = bn;
      best.splits = splits;
    }
  };
  // (tiles wider than the tokens, rounded up to the MMA's step, only pad)
  const int bn_max = std::min(256, std::max(32, (M + 15) / 16 * 16));
  for (int bn = 32; bn <= bn_max; bn += 16) {
    const int tiles = tiles_n * ((M + bn - 1) / bn);
    const float step = (float)((128 + bn) * 128) / 168e3f, epi = 0.0135f * (float)bn * (geglu ? 2.18f : 1.f);
    const int waves = (tiles + num_sms - 1) / num_sms;
    consider(false, bn, 1,
             (xbf16 ? 2.9f : 2.6f) + epi + (float)waves * (float)num_kb * step + (float)(waves - 1) * 0.0067f * (float)bn);
    for (int i = 0; i < 4; ++i) {
      // the splits of a tile form one cluster; each sums a slice of whole
      // 4-token groups, of at most 32 tokens through shared memory, and
      // through L2 the partials have to fit the workspace; there the slice goes
      // out in chunks of 16, 8 or 4 tokens, each a round trip (two with the
      // residual stream's reads: M 200 x N 2049 x K 6216 in seven chunks of 4
      // tokens took 48 us, in two of 16 29, of 64-token tiles in two waves 41)
      const int sp = 2 << i;
      if (sp > num_kb || bn % (4 * sp) || !clusters.n[i] || (long)tiles * sp > 2L * num_sms) break;
      if (dsmem ? bn / sp > 32 : (size_t)sp * tiles * bn * TC_BM * 4 > ws_bytes) continue;
      const int chunks = bn / sp / split_chunk(bn / sp);
      const int w = (tiles + clusters.n[i] - 1) / clusters.n[i];
      consider(false, bn, sp,
               2.6f + epi / (float)sp + (float)w * (float)((num_kb + sp - 1) / sp) * step +
                   (shares_bf16 ? 0.47f : 2.14f) * (float)bn / 64.f + (float)(w - 1) * (dsmem ? 2.5f : 10.f) +
                   (dsmem ? 0.f : (float)(chunks - 1) * (g.epi == EPI_ADD_F32 ? 4.f : 0.8f)) +
                   (xbf16 ? 0.7f * (float)std::max(0, tiles * sp - num_sms / 2) / (float)(num_sms / 2) : 0.f));
    }
  }
  const int tiles_n2 = (N + 2 * TC_BM - 1) / (2 * TC_BM), slots = num_sms / 2;
  for (int bn = 64; pairs && bn <= std::max(64, std::min(256, (M + 31) / 32 * 32)); bn += 32) {
    const int waves = (tiles_n2 * ((M + bn - 1) / bn) + slots - 1) / slots;
    const float step = std::max((float)((128 + bn / 2) * 128) / 142e3f, 0.295f * (float)bn / 256.f);
    consider(true, bn, 1,
             3.4f + 0.0119f * (float)bn * (geglu ? 1.35f : 1.f) + (float)waves * (float)num_kb * step +
                 (float)(waves - 1) * 1.1f);
  }
  return best;
}

bool out_is_bf16(const GemmArgs& g) { return g.epi == EPI_GEGLU || (g.epi != EPI_ADD_F32 && g.out_dt == DT_BF16); }

// outputs through TMA boxes when the output rows are 16-byte aligned
bool out_aligned(const GemmArgs& g) {
  return ((uintptr_t)g.out & 15) == 0 && ((size_t)g.ldo * (out_is_bf16(g) ? 2 : 4)) % 16 == 0;
}

// The tensor cores truncate each fp32 accumulation, so a sum's error grows
// with its length: about 1e-9 of the result per K element (N(0, 1) x N(0,
// 0.02) operands: 1.2e-7 at K = 128, 9.9e-7 at 1024).  Where the result is
// stored in fp32 and no share is rounded to bf16, an item's K range therefore
// goes through an accumulator per k-tile (64 elements), as far as TMEM holds
// them beside the accumulators of the tile before, added in the epilogue.  Past
// 32 k-tiles four take a quarter each (outputs through TMA boxes; the others have
// fewer splits than they had): M 800 x N 1024 x K 4096 errs by 7.9e-7 with
// four, 3.7e-7 with eight, which add 1.6 to its 14.8 us.  A step's projections,
// whose operands are bf16 activations, take two halves where 128-token tiles
// leave half the SMs idle, as a split of those would (800 tokens: 0.3 us per
// launch; 3200: 16 of a step's 2630, and no split to match).  The two-SM kernel sums all of
// K in one (its tiles fill TMEM), as it does for bf16 results, which round at
// 2e-3.
int sum_accumulators(const GemmArgs& g, bool bf16_exchange, int kb_per_item, uint32_t acc_cols, bool two_items,
                     int num_sms) {
  if (bf16_exchange || g.epi == EPI_GEGLU || (g.epi != EPI_ADD_F32 && g.out_dt == DT_BF16)) return 1;
  const int fit = std::max(1, 512 / (int)acc_cols / (two_items ? 2 : 1));
  const long tiles = (long)((g.N + TC_BM - 1) / TC_BM) * ((g.M + 127) / 128);
  return std::min({kb_per_item, fit, g.xbf16 ? (tiles * 2 <= num_sms ? 2 : 1) : kb_per_item > 32 && out_aligned(g) ? 4 : fit});
}

// Sizes of a launch: the operand ring, TMEM and the shared memory around them.
struct TcLayout {
  int stages = 0, accs = 1, reduce = RED_NONE, box_m = 0;
  bool oneshot = false;
  uint32_t acc_cols = 32, ncols = 0, box_bytes = 0, stg_off = 0, xch_off = 0, rcv_off = 0, bar_off = 0, set_bytes = 0;
  size_t ring = 0, smem = 0;   // smem 0: no such launch
};

// Two-SM launch with token tiles of bn (a multiple of 32 in [64, 256]).
TcLayout pair_layout(const GemmArgs& g, int bn) {
  TcLayout l;
  while ((int)l.acc_cols < bn) l.acc_cols <<= 1;
  l.ncols = 2 * l.acc_cols;
  l.box_m = 32;
  l.box_bytes = (uint32_t)(((size_t)l.box_m * (g.epi == EPI_GEGLU ? 64 : TC_BM) * (out_is_bf16(g) ? 2 : 4) + 1023) /
                           1024 * 1024);
  const size_t stg_bytes = 2 * (size_t)l.box_bytes;
  const size_t xch_bytes = g.epi == EPI_GEGLU ? (XCH_BYTES + 1023) / 1024 * 1024 : 0;
  // each of the two epilogue warp sets has its own boxes and exchange tile
  l.set_bytes = (uint32_t)(stg_bytes + xch_bytes);
  const size_t fixed = 1024 + 2 * (size_t)l.set_bytes + 256;
  const int stage_bytes = TC_A_BYTES + (bn / 2) * TC_BK * 2;
  l.stages = std::min(8, (int)((TC_SMEM_MAX - fixed) / stage_bytes));
  if (l.stages < 2) return l;
  l.ring = ((size_t)l.stages * stage_bytes + 1023) / 1024 * 1024;
  l.stg_off = (uint32_t)l.ring;
  l.xch_off = l.stg_off + (uint32_t)stg_bytes;
  l.bar_off = l.stg_off + 2 * l.set_bytes;
  const size_t smem = 1024 + l.bar_off + (size_t)(2 * l.stages + 4) * 8 + 4 + 16 + 64;
  l.smem = smem > (size_t)TC_SMEM_MAX ? 0 : smem;
  return l;
}

// One-SM launch of a plan.
TcLayout one_layout(const GemmArgs& g, const TcPlan& plan, int num_sms) {
  TcLayout l;
  const bool tma_out = out_aligned(g);
  const int bn = plan.bn, splits = plan.splits, es = out_is_bf16(g) ? 2 : 4;
  const int tiles = (g.N + TC_BM - 1) / TC_BM * ((g.M + bn - 1) / bn);
  const int num_kb = (g.K + TC_BK - 1) / TC_BK;
  const int cpr = bn / splits;   // a multiple of 4 whenever the splits form a cluster
  while ((int)l.acc_cols < bn) l.acc_cols <<= 1;
  const int stage_bytes = TC_A_BYTES + bn * TC_BK * 2;
  const int kb_per_item = (num_kb + splits - 1) / splits;
  const int grid_ctas = splits > 1 ? tiles * splits : std::min(tiles, num_sms);
  const int items = splits > 1 ? 1 : (tiles + grid_ctas - 1) / grid_ctas;
  l.stages = std::min(8, TC_SMEM_BUDGET / stage_bytes);
  // a split-K launch is latency-bound: enough stages for its whole (short) K
  // range when that fits, so that no operand load waits for a freed stage
  if (splits > 1) l.stages = std::min(l.stages, std::max(2, TC_RING_SPLIT / stage_bytes));
  l.stages = std::max(2, std::min(l.stages, std::max(2, kb_per_item * items)));
  const bool xbf = bf16_shares(g, num_sms);   // partials exchanged in bf16, else in fp32
  const bool dsmem = splits > 1 && tma_out;
  const size_t rcv_bytes = dsmem ? (size_t)TC_BM * bn * (xbf ? 2 : 4) : 0;
  // a CTA with several items works on two at a time
  l.accs = sum_accumulators(g, dsmem && xbf, kb_per_item, l.acc_cols, items > 1, num_sms);
  l.ncols = 32;
  while (l.ncols < l.acc_cols * (uint32_t)l.accs * (items > 1 ? 2u : 1u)) l.ncols <<= 1;
  // one-shot: a cluster split whose whole K range fits a ring of up to 200 KB
  // takes its weight and token k-tiles in one box each (K a multiple of 64)
  l.oneshot = splits > 1 && g.K % TC_BK == 0 && g.K / TC_BK <= 256 &&
              (size_t)kb_per_item * stage_bytes <=
                  std::min<size_t>(TC_SMEM_BUDGET, TC_SMEM_MAX - 4096 - (rcv_bytes + 1023) / 1024 * 1024);
  if (l.oneshot) l.stages = kb_per_item;   // the ring is exactly one box deep
  l.ring = ((size_t)l.stages * stage_bytes + 1023) / 1024 * 1024;
  l.reduce = splits == 1 ? RED_NONE : !dsmem ? RED_L2_CLUSTER : xbf ? RED_DSMEM : RED_DSMEM32;
  // tokens per output box; a split's slice is stored by the threads, its
  // received partials (all splits' slices of this rank) behind the ring
  l.box_m = splits == 1 ? 16 : split_chunk(cpr);
  l.box_bytes = (uint32_t)(((size_t)l.box_m * (g.epi == EPI_GEGLU ? 64 : TC_BM) * es + 1023) / 1024 * 1024);
  const size_t stg_bytes = dsmem ? rcv_bytes : tma_out ? 2 * (size_t)l.box_bytes : (STG_BYTES + 1023) / 1024 * 1024;
  const size_t xch_bytes = (splits == 1 && tma_out && g.epi == EPI_GEGLU) ? (XCH_BYTES + 1023) / 1024 * 1024 : 0;
  l.stg_off = l.rcv_off = (uint32_t)l.ring;
  l.xch_off = l.stg_off + (uint32_t)stg_bytes;
  l.bar_off = l.xch_off + (uint32_t)xch_bytes;
  size_t smem = 1024 + l.bar_off + (size_t)(2 * l.stages + 5) * 8 + 4 + 16 + 64;
  // The CTAs of a split wait for one another with their TMEM taken.  Beside a
  // CTA of another stream's split launch, one could wait for columns that the
  // other frees only after a peer that waits likewise, until both time out:
  // a launch takes no larger share of the SM's TMEM than of its shared memory
  // (1 KB per CTA is the system's), so that what fits together fits in both.
  if (splits > 1) smem = std::max(smem, (size_t)l.ncols * TC_SMEM_SM / 512 - 1024);
  l.smem = smem > (size_t)TC_SMEM_MAX ? 0 : smem;
  return l;
}

// Two-SM launch of a persistent GEMM (see tc_gemm_pair_kernel) with token
// tiles of bn and the usual TMA epilogue layout.
cudaError_t launch_gemm_pair(const GemmArgs& g, const TcWorkspace& ws, int num_sms, cudaStream_t st, int bn) {
  const TcLayout l = pair_layout(g, bn);
  if (!l.smem) return cudaErrorInvalidConfiguration;
  const bool out_bf = out_is_bf16(g);
  const int ek = g.epi == EPI_GEGLU ? EK_GEGLU : g.epi == EPI_ADD_F32 ? EK_ADD : out_bf ? EK_BF16 : EK_F32;
  const int tiles_n = (g.N + TC_BM - 1) / TC_BM;
  const int tiles_n2 = (g.N + 2 * TC_BM - 1) / (2 * TC_BM);
  const int slots = num_sms / 2;
  const int tiles_m = (g.M + bn - 1) / bn;
  const int num_tiles = tiles_n2 * tiles_m;
  const int num_kb = (g.K + TC_BK - 1) / TC_BK;
  CUtensorMap mw, mx, mo;
  cudaError_t e = encode_2d(&mw, g.W, g.N, g.K, g.ldw, TC_BM);
  if (e == cudaSuccess) e = encode_2d(&mx, g.A, g.M, g.K, g.lda, bn / 2);
  if (e == cudaSuccess)
    e = encode_out(&mo, g.out, g.M, g.epi == EPI_GEGLU ? g.N / 2 : g.N, g.ldo, out_bf,
                   g.epi == EPI_GEGLU ? 64 : TC_BM, l.box_m);
  if (e != cudaSuccess) return e;
  TcParams p{g.M, g.N, bn, l.stages, 1, num_kb, l.ncols, l.acc_cols, 1, tiles_n, tiles_m,
             num_tiles, (int)g.epi, g.out_dt == DT_BF16 ? 1 : 0, g.out, g.ldo, g.bias, ws.ws, ws.err,
             0, l.box_m, l.box_bytes, l.stg_off, l.xch_off, 0, l.bar_off, kTcTimeoutNs, 0, g.skip};
  p.set_bytes = l.set_bytes;
  const int npairs = std::min(num_tiles, slots);
  return launch_kernel_cluster(tc_pair_kernel(ek), dim3(2 * npairs), dim3(TC_PAIR_THREADS), l.smem, st, dim3(2, 1, 1),
                               mw, mx, mo, p);
}

}  // namespace

void debug_withhold_gemm(int launches) { g_withhold.store(launches > 0 ? launches : 0); }

cudaError_t init_tc_gemm() {
  cudaError_t e = get_encoder();
  if (e != cudaSuccess) return e;
  std::vector<const void*> kernels;
  for (int red = 0; red <= RED_DSMEM32; ++red)
    for (int ek = 0; ek <= EK_SLICE; ++ek)
      if (TcKernel k = tc_kernel(red, ek)) kernels.push_back((const void*)k);
  for (int ek = 0; ek < EK_GENERIC; ++ek) kernels.push_back((const void*)tc_pair_kernel(ek));
  for (const void* k : kernels) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM_MAX);
    if (e != cudaSuccess) return e;
  }
  // clusters of 16 are beyond the portable limit: use them only if allowed
  bool big = true;
  for (const void* k : kernels) big = big && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  for (int i = 0; i < (big ? 4 : 3); ++i) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 2u << i;
    cfg.gridDim = dim3(1, 1, 2u << i);
    cfg.blockDim = dim3(TC_THREADS);
    cfg.dynamicSmemBytes = TC_SMEM_MAX;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    g_max_clusters.n[i] =
        cudaOccupancyMaxActiveClusters(&n, tc_kernel(RED_DSMEM, EK_SLICE), &cfg) == cudaSuccess && n > 0 ? n : 0;
  }
  cudaGetLastError();
  return cudaSuccess;
}

bool tc_gemm_supported(const GemmArgs& g) {
  // TMA: 16-byte aligned bases and row strides
  if (g.K % 8 || g.lda % 8 || g.ldw % 8) return false;
  if (((uintptr_t)g.A & 15) || ((uintptr_t)g.W & 15)) return false;
  if (g.epi == EPI_GEGLU && (g.N % 128)) return false;
  return g.M > 0 && g.N > 0 && g.K > 0;
}

cudaError_t launch_gemm_tc(const GemmArgs& g, const TcWorkspace& ws, int num_sms, cudaStream_t st) {
  if (!g_encode) return cudaErrorInitializationError;
  const bool out_bf = out_is_bf16(g), tma_out = out_aligned(g);
  const TcPlan plan = plan_gemm(g, tma_out, ws.ws_bytes, tma_out, num_sms, g_max_clusters);
  if (plan.pair) return launch_gemm_pair(g, ws, num_sms, st, plan.bn);
  const TcLayout l = one_layout(g, plan, num_sms);
  if (!l.smem) return cudaErrorInvalidConfiguration;
  const int bn = plan.bn, splits = plan.splits;
  const int tiles_n = (g.N + TC_BM - 1) / TC_BM;
  const int tiles_m = (g.M + bn - 1) / bn;
  const int num_kb = (g.K + TC_BK - 1) / TC_BK;
  const int tiles = tiles_n * tiles_m;
  const int kb_per_item = (num_kb + splits - 1) / splits;
  const int grid_ctas = splits > 1 ? tiles * splits : std::min(tiles, num_sms);
  const bool oneshot = l.oneshot, dsmem = splits > 1 && tma_out;
  CUtensorMap mw, mx, mo;
  memset(&mo, 0, sizeof(mo));
  cudaError_t e = oneshot ? encode_kt(&mw, g.W, g.N, g.K, g.ldw, TC_BM, kb_per_item)
                          : encode_2d(&mw, g.W, g.N, g.K, g.ldw, TC_BM);
  if (e == cudaSuccess)
    e = oneshot ? encode_kt(&mx, g.A, g.M, g.K, g.lda, bn, kb_per_item) : encode_2d(&mx, g.A, g.M, g.K, g.lda, bn);
  if (e == cudaSuccess && tma_out && !dsmem)
    e = encode_out(&mo, g.out, g.M, g.epi == EPI_GEGLU ? g.N / 2 : g.N, g.ldo, out_bf,
                   g.epi == EPI_GEGLU ? 64 : TC_BM, l.box_m);
  if (e != cudaSuccess) return e;
  TcParams p{g.M, g.N, bn, l.stages, splits, num_kb, l.ncols, l.acc_cols, l.accs, tiles_n,
             tiles_m, tiles, (int)g.epi, g.out_dt == DT_BF16 ? 1 : 0, g.out, g.ldo, g.bias, ws.ws, ws.err,
             oneshot ? 1 : 0, l.box_m, l.box_bytes, l.stg_off, l.xch_off, l.rcv_off, l.bar_off,
             kTcTimeoutNs, 0, g.skip};
  // fault injection (tests): a launch without a cluster may be told to wait
  // for an arrival that never comes, with a short limit
  if (l.reduce == RED_NONE && g_withhold.load() > 0 && g_withhold.fetch_sub(1) > 0) {
    p.withhold = 1;
    p.wait_ns = kWithholdWaitNs;
  }
  const dim3 grid = splits > 1 ? dim3(tiles_n, tiles_m, splits) : dim3(grid_ctas);
  const dim3 block(TC_THREADS);
  // persistent launches: one instantiation per epilogue kind; split-K
  // launches: one for all
  const int ek = !tma_out ? EK_GENERIC
                 : dsmem ? EK_SLICE
                 : g.epi == EPI_GEGLU ? EK_GEGLU : g.epi == EPI_ADD_F32 ? EK_ADD : out_bf ? EK_BF16 : EK_F32;
  const TcKernel k = tc_kernel(l.reduce, ek);
  if (!k) return cudaErrorInvalidConfiguration;
  return launch_kernel(k, grid, block, l.smem, st, (unsigned)splits, mw, mx, mo, p);
}

}  // namespace ravel

// What a tensor-core GEMM of these sizes is cut into, for tests: out = {1 on SM
// pairs, token-tile width, K splits, how they exchange (0 none, 1 fp32 through
// L2, 2 bf16 and 3 fp32 through shared memory), accumulators per item, TMEM
// columns, shared-memory bytes}.  clusters: how many clusters of 2, 4, 8, 16 fit.
extern "C" void ravel_debug_gemm_plan(int M, int N, int K, int epi, int out_bf16, int xbf16, int aligned,
                                      size_t ws_bytes, int num_sms, const int* clusters, int* out) {
  using namespace ravel;
  GemmArgs g{nullptr, K, nullptr, K, M, N, K, (Epi)epi, (void*)(uintptr_t)(aligned ? 16 : 4), (N + 7) / 8 * 8,
             out_bf16 ? DT_BF16 : DT_F32, nullptr};
  g.xbf16 = xbf16;
  const TcPlan plan = plan_gemm(g, aligned != 0, ws_bytes, aligned != 0, num_sms,
                                TcClusters{{clusters[0], clusters[1], clusters[2], clusters[3]}});
  const TcLayout l = plan.pair ? pair_layout(g, plan.bn) : one_layout(g, plan, num_sms);
  const int v[7] = {plan.pair, plan.bn, plan.splits, l.reduce, l.accs, (int)l.ncols, (int)l.smem};
  for (int i = 0; i < 7; ++i) out[i] = v[i];
}
