// Grouped-query attention of the action slots on the 5th-generation tensor
// cores (tcgen05 + TMEM + TMA), flash-attention style.
//
// One CTA owns a tile of up to 128 query rows of one (robot b, KV head g)
// pair -- row r = t*G + hh is slot j0+t of query head g*G+hh -- and walks the
// pair's keys in chunks of 128: first the active VLM context's prefix
// (context slot, valid length read on the device), then the FOP tokens and
// the H action slots of this step (the QKV buffer).  Per chunk:
//   S = Q K^T        tcgen05.mma, M = 128 query rows, N = 128 keys, into TMEM
//   P = exp(S - m)   softmax warps: TMEM -> registers -> bf16 P back into TMEM
//   O += P V         tcgen05.mma, M = 128, N = head dim, K = 16 keys at a time, O in TMEM
// What bounds it is the tensor pipe and the issue of its instructions (up to
// N = 128 an MMA takes its warp 71 cycles whatever its N): chunks of 64 keys
// spent 16 such MMAs on S for every 64 keys at head dim 256, 128-key chunks
// spend them on 128.  Shared memory holds no two such chunks beside Q, so K
// comes in units of 64 head dims (16 KB, freed as their four MMAs complete) and
// V in halves of 64 keys: 4 K units + 3 V halves at head dim 256, the next
// chunk's units streaming in behind the MMAs.  K is K-major, V the B operand of
// P V in its natural layout (MN-major).
// The online softmax rescales O in TMEM only when a row's running maximum
// grows by more than 2^8 (the kept maximum is exact for the final
// normalisation, so this is not an approximation).
// At batch 1 a (b, g) pair has only a few query tiles, so the key chunks are
// split over grid.z; the splits of a query tile form a thread-block cluster
// and rank q merges head-dim slice q of every split's partial.  Each split
// sends its rows' (m, l) and its output normalised by its own l, in bf16 (the
// precision of every activation between kernels of the bf16 path), by
// st.async straight into the owning rank's shared memory, overlaid on Q and
// the K ring, as soon as its own PV is done and every split's last S MMA has
// completed (a multicast tcgen05.commit on each split's "S done" barrier); an
// mbarrier at the owner counts the bytes.  Where that does not apply, the splits
// publish unnormalised fp32 partials through L2 and the cluster barrier.  The
// producer asks for the rest of its split's prefix in L2 as it starts.
//
// Warp roles (320 threads): warp 0 TMA producer, warp 1 TMEM allocator + MMA
// issuer, warps 2..9 softmax / epilogue (warp w owns TMEM lanes 32*(w%4)..).
// Every wait is bounded (ERR_TIMEOUT, then unwind).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "launch.h"
#include "tc_common.cuh"

namespace ravel {
namespace {

// warp 0: loads; warp 1: MMAs; warps 2-9: softmax and epilogue, two threads per
// query row (warps w and w + 4 share TMEM lanes): each takes 64 keys of a
// chunk, and half of O's columns; all ten merge the key splits
constexpr int AT_THREADS = 320;
constexpr int AT_BM = 128;
constexpr int AT_BKV = 128;          // keys of a chunk
constexpr int AT_SMEM_MAX = 227 * 1024;
constexpr uint32_t AT_QBLK = AT_BM * 128;     // bytes of one 64-wide head-dim block of Q
constexpr uint32_t AT_KUNIT = AT_BKV * 128;   // bytes of a K unit: 128 keys x 64 head dims
constexpr uint32_t AT_VBLK = 64 * 128;        // bytes of one 64-wide head-dim block of a V half (64 keys)

// Limit of the polling loops: a counter, because reading the global timer in
// each turn left the tensor pipe idle between S and P V.  A turn takes at
// least 30 cycles and at most some hundred: 0.5 to 5 s.
constexpr uint32_t kPollLimit = 1u << 25;

struct AtParams {
  int H, F, Hkv, G, hd, hdp;   // hdp: head dim rounded up to 16 (MMA N of P V)
  int TQ, q_tiles;
  int Pmax, n_kv, splits;
  int layer, Bmax, mask_mode;
  int nblk, k_slots, v_slots;         // head-dim blocks of 64; K units and V halves in their rings
  int xch;                            // splits > 1: partials through shared memory (1; the receive area lies in
                                      // Q and the K ring) or L2 (0)
  const int* ctx_state;
  const bf16 *ck[2], *cv[2];          // context slots [L][Bmax][Hkv][Pmax][hd]
  bf16* out;
  int ld_out;
  float* ws_o;
  float* ws_ml;
  int* err;
  float scale_log2;                   // log2(e) / sqrt(hd)
};

// boxes of [128 keys][64-wide head-dim block] (K) and [64 keys][64-wide block]
// (V), 128-byte swizzled.  V's maps end at the robot's last row, so that the rows
// of a 16-key group past it are zeros: their probability is 0, but 0 times
// another robot's Inf or NaN is not.  (K needs no such end: those scores are
// replaced.  The context's V rows up to the group's end are zeroed when it is
// installed.)
struct AtMaps {
  CUtensorMap q, k, v, pk0, pk1, pv0, pv1, o;   // o: (hd, heads, slots, robots), boxes as Q's
};

// Rows of the split-KV combine: out = sum_s wgt[s] * O_s * inv over float4
// columns [c4b, c4e) of this thread's row, the SP partials of a column batch
// loaded together (one L2 round trip per batch).  src0 points at split 0 of
// the row; splits are sstride floats apart, float4 columns 512.
template <int SP>
__device__ __forceinline__ void combine_slice(const float* src0, size_t sstride, int c4b, int c4e, const float* wgt,
                                              float inv, bf16* orow, int hd, bool row_ok) {
  constexpr int KC = 32 / SP;
  for (int c4 = c4b; c4 < c4e; c4 += KC) {
    float4 x[SP][KC];
#pragma unroll
    for (int s2 = 0; s2 < SP; ++s2)
#pragma unroll
      for (int k = 0; k < KC; ++k)
        x[s2][k] = (c4 + k < c4e) ? __ldcg((const float4*)(src0 + (size_t)s2 * sstride + (size_t)(c4 + k) * 512))
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < KC; ++k) {
      const int d = 4 * (c4 + k);
      if (c4 + k >= c4e || d >= hd) break;
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int s2 = 0; s2 < SP; ++s2) {
        acc.x += wgt[s2] * x[s2][k].x;
        acc.y += wgt[s2] * x[s2][k].y;
        acc.z += wgt[s2] * x[s2][k].z;
        acc.w += wgt[s2] * x[s2][k].w;
      }
      if (row_ok)   // hd % 8 == 0 and d % 4 == 0: all four columns exist; 8-byte aligned
        *(uint2*)(orow + d) = make_uint2(pack_bf16x2(acc.x * inv, acc.y * inv), pack_bf16x2(acc.z * inv, acc.w * inv));
    }
  }
}

__device__ __forceinline__ uint4 lds_u4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ float2 lds_f2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
  return v;
}

// Merge of row r, head-dim group gq, over the SP splits' shares received in
// shared memory (O groups [s][g][row] of 8 bf16 from `og`, (m, l) [s][row]
// from `ml`, both shared-memory addresses of row 0): columns d0 + 8 gq .. +7
// of slice q, stored as bf16 (a group past hd is skipped).
//   O = sum_s 2^(m_s - M) l_s Ohat_s / sum_s 2^(m_s - M) l_s
template <int SP>
__device__ __forceinline__ void xch_combine_group(uint32_t og, uint32_t ml, int r, int ngs, int gq, int d0, int hd,
                                                  bf16* orow) {
  const int d = d0 + 8 * gq;
  if (d >= hd) return;
  float2 v[SP];
#pragma unroll
  for (int s2 = 0; s2 < SP; ++s2) v[s2] = lds_f2(ml + (uint32_t)(s2 * AT_BM + r) * 8u);
  uint4 u[SP];
#pragma unroll
  for (int s2 = 0; s2 < SP; ++s2) u[s2] = lds_u4(og + ((uint32_t)(s2 * ngs + gq) * AT_BM + r) * 16u);
  float M = -INFINITY;
#pragma unroll
  for (int s2 = 0; s2 < SP; ++s2) M = fmaxf(M, v[s2].x);
  float w[SP];
  float L = 0.f;
#pragma unroll
  for (int s2 = 0; s2 < SP; ++s2) {
    w[s2] = (v[s2].x == -INFINITY) ? 0.f : exp2f(v[s2].x - M) * v[s2].y;
    L += w[s2];
  }
  const float inv = L > 0.f ? 1.f / L : 0.f;
  float acc[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = 0.f;
#pragma unroll
  for (int s2 = 0; s2 < SP; ++s2) {
    const float ws = w[s2] * inv;
    const uint32_t uu[4] = {u[s2].x, u[s2].y, u[s2].z, u[s2].w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      acc[2 * k] = fmaf(ws, __uint_as_float(uu[k] << 16), acc[2 * k]);
      acc[2 * k + 1] = fmaf(ws, __uint_as_float(uu[k] & 0xFFFF0000u), acc[2 * k + 1]);
    }
  }
  *(uint4*)(orow + d) = make_uint4(pack_bf16x2(acc[0], acc[1]), pack_bf16x2(acc[2], acc[3]),
                                   pack_bf16x2(acc[4], acc[5]), pack_bf16x2(acc[6], acc[7]));
}

__global__ void __launch_bounds__(AT_THREADS, 1) attn_tc_kernel(const __grid_constant__ AtMaps maps, AtParams p) {
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte aligned; derived from smem_raw by pointer arithmetic so that the
  // compiler keeps it (and everything indexed from it) in the shared window
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int SK = p.k_slots, SV = p.v_slots;   // K and V ring depths
  const uint32_t v_bytes = (uint32_t)p.nblk * AT_VBLK;   // one V half
  uint8_t* q_s = smem;
  uint8_t* kv_s = q_s + (size_t)p.nblk * AT_QBLK;   // K ring, then V ring
  uint8_t* v_ring = kv_s + (size_t)SK * AT_KUNIT;
  uint64_t* bars = (uint64_t*)(v_ring + (size_t)SV * v_bytes);
  // every K unit and V half has its own barriers: a K unit is released as its
  // MMAs of S = Q K^T complete, a V half as its MMAs of P V do
  uint64_t* q_full = bars;
  uint64_t* k_full = bars + 1;
  uint64_t* v_full = k_full + SK;
  uint64_t* k_empty = v_full + SV;
  uint64_t* v_empty = k_empty + SK;
  uint64_t* s_full = v_empty + SV;
  uint64_t* p_full = s_full + 2;
  uint64_t* pv_done = p_full + 2;   // [2]: PV of chunk i completes pv_done[i & 1]
  uint64_t* rcv_bar = pv_done + 2;  // xch: every split's share of this rank has arrived
  uint64_t* sdone = rcv_bar + 1;    // xch: every split's last S MMA has completed (one arrival each)
  uint32_t* tmem_slot = (uint32_t*)(sdone + 1);
  float* xm = (float*)((uint8_t*)bars + 512);   // [2][128] row maxima, then sums, of the two halves
  int* flags = (int*)(tmem_slot + 1);   // [0] abort, [1] K units issued, [2] consumed, [3] V halves issued, [4] consumed

  // (through a shuffle, so that the compiler knows it is uniform in the warp)
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int qt = blockIdx.x, bg = blockIdx.y, split = blockIdx.z;
  const int b = bg / p.Hkv, g = bg % p.Hkv;
  const int rows_per_robot = p.H + p.F;
  const int slot = p.ctx_state[2 * b];       // this robot's active context
  const int P = p.ctx_state[2 * b + 1];
  // this robot's chunks: npv of its prefix, then n_kv of the step's own keys; this
  // split's are c0 .. c1 - 1 (an even share of the keys that exist, whatever the
  // context's capacity)
  const int npv = (P + AT_BKV - 1) / AT_BKV;
  const int C = npv + p.n_kv;
  const int c0 = split * C / p.splits, c1 = (split + 1) * C / p.splits;
  constexpr uint32_t ncols = 512;   // two S tiles of 128 columns, O
  const int ctx_z = (p.layer * p.Bmax + b) * p.Hkv + g;
  // query rows of this tile that hold a slot (rows 0 .. vrows-1)
  const int vrows = p.G * max(0, min(p.TQ, p.H - qt * p.TQ));
  // xch: per rank, [split][cps / 8][128 rows] groups of 8 bf16, then [split][128 rows] (m, l)
  const int cps = p.hdp / p.splits;

  pdl_trigger();
  if (P < 1 || P > p.Pmax) {   // uniform across the CTA: nothing allocated yet
    pdl_wait();
    if (threadIdx.x == 0) raise_error(p.err, ERR_PREFIX_LEN);
    return;
  }
  const int n = c1 - c0;
  // keys of chunk c that exist (the prefix may end inside its last chunk, the
  // step's own keys inside theirs), from key `first` of the prefix / own keys on
  auto keys_of = [&](int c) {
    return min(AT_BKV, c < npv ? P - c * AT_BKV : rows_per_robot - (c - npv) * AT_BKV);
  };

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < SK; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);   // released by the S commit
    }
    for (int s = 0; s < SV; ++s) {
      mbar_init(&v_full[s], 1);
      mbar_init(&v_empty[s], 1);   // released by the PV commits
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s_full[i], 1);
      mbar_init(&p_full[i], 256);
    }
    mbar_init(&pv_done[0], 1);
    mbar_init(&pv_done[1], 1);
    mbar_init(rcv_bar, 1);
    mbar_init(sdone, p.splits);
    flags[0] = flags[1] = flags[2] = flags[3] = flags[4] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (p.xch) mbar_expect_tx(rcv_bar, (uint32_t)(p.splits * vrows * (2 * cps + 8)));
  }
  // (xch) every split's barriers must exist before a peer targets them
  if (p.xch) cluster_sync();
  const CUtensorMap* pk = slot ? &maps.pk1 : &maps.pk0;
  const CUtensorMap* pv = slot ? &maps.pv1 : &maps.pv0;
  uint32_t el = 0;   // the issuing lane of warps 0 (TMA) and 1 (MMA)
  const uint32_t q0 = smem_u32(q_s), k0 = smem_u32(kv_s), v0 = smem_u32(v_ring);
  // K unit (chunk c, head-dim block blk) and V half h of chunk c into their
  // slots (warp 0), each CTA loading its own copy (query tiles of one (b, g)
  // pair read the same chunk, which L2 serves to all)
  uint64_t pol_q = 0, pol_kv = 0;
  auto load_k = [&](int c, int blk, int s) {
    const bool pre = c < npv;
    mbar_expect_tx_el(&k_full[s], AT_KUNIT, el);
    tma_load_3d_el(pre ? pk : &maps.k, smem_u32(&k_full[s]), k0 + (uint32_t)s * AT_KUNIT, blk * 64,
                   pre ? c * AT_BKV : g, pre ? ctx_z : b * rows_per_robot + (c - npv) * AT_BKV, pre ? pol_kv : pol_q,
                   el);
  };
  auto load_v = [&](int c, int h, int s) {
    const bool pre = c < npv;
    const uint32_t vs = v0 + (uint32_t)s * v_bytes, bar = smem_u32(&v_full[s]);
    const CUtensorMap* vm = pre ? pv : &maps.v;
    const int key = (pre ? c : c - npv) * AT_BKV + 64 * h;
    mbar_expect_tx_el(&v_full[s], v_bytes, el);
    #pragma unroll 1
    for (int blk = 0; blk < p.nblk; ++blk)
      tma_load_4d_el(vm, bar, vs + (uint32_t)blk * AT_VBLK, blk * 64, pre ? 0 : g, key, pre ? ctx_z : b,
                     pre ? pol_kv : pol_q, el);
  };
  // next K unit (chunk kc, block kb, slot sk) and V half (chunk vc, half vh, slot
  // sv) to load, and the parities their `empty` waits take
  int kc = c0, kb = 0, nk = 0, sk = 0, vc = c0, vh = 0, nv = 0, sv = 0;
  uint32_t phk = 1, phv = 1;
  auto next_k = [&]() {
    load_k(kc, kb, sk);
    ++nk;
    if (++kb == p.nblk) {
      kb = 0;
      ++kc;
    }
    if (++sk == SK) {
      sk = 0;
      phk ^= 1u;
    }
  };
  auto next_v = [&]() {   // (a chunk of at most 64 keys has one half)
    load_v(vc, vh, sv);
    ++nv;
    if (vh == 1 || keys_of(vc) <= 64) {
      vh = 0;
      ++vc;
    } else {
      vh = 1;
    }
    if (++sv == SV) {
      sv = 0;
      phv ^= 1u;
    }
  };
  if (warp == 0) {
    __syncwarp();   // the barriers initialised above
    el = elect_one();
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_q));
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol_kv));
    // the active context (slot, length and its prefix K/V) is fixed for the
    // whole step, so the first prefix units are fetched before the wait on the
    // previous kernel (the QKV projection)
    const int pre_end = min(c1, npv);
    #pragma unroll 1
    while (nk < SK && kc < pre_end) next_k();
    #pragma unroll 1
    while (nv < SV && vc < pre_end) next_v();
    // the rest of the split's prefix goes to L2 now, K and V in one request
    // each (the query tiles of a pair share it): loads that the loop below
    // issues then find it there.  (Requests per chunk from the loop itself, a
    // box at a time, held up the next K unit: 3900 cycles per chunk at batch
    // 64, 2700 without them; the tensor pipe needs 2050.)
    if (qt == 0 && kc < pre_end && el) {
      const size_t row0 = (size_t)ctx_z * p.Pmax + (size_t)kc * AT_BKV;
      const uint32_t bytes = (uint32_t)(min(pre_end * AT_BKV, P) - kc * AT_BKV) * (uint32_t)p.hd * 2u;
      prefetch_l2_bulk(p.ck[slot ? 1 : 0] + row0 * p.hd, bytes);
      prefetch_l2_bulk(p.cv[slot ? 1 : 0] + row0 * p.hd, bytes);
    }
    __syncwarp();
  }
  // rows of the Q tile that no query fills are zeroed (their scores are unused)
  const int q_rows = p.TQ * p.G;
  if (q_rows < AT_BM) {
    for (int blk = 0; blk < p.nblk; ++blk) {
      uint4* z = (uint4*)(q_s + (size_t)blk * AT_QBLK + (size_t)q_rows * 128);
      for (int i = threadIdx.x; i < (AT_BM - q_rows) * 8; i += AT_THREADS) z[i] = make_uint4(0, 0, 0, 0);
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  pdl_wait();
  if (warp == 0) {   // Q, before the TMEM set-up, which it does not need
    mbar_expect_tx_el(q_full, (uint32_t)p.nblk * 128u * (uint32_t)q_rows, el);
    #pragma unroll 1
    for (int blk = 0; blk < p.nblk; ++blk)
      tma_load_3d_el(&maps.q, smem_u32(q_full), q0 + (uint32_t)blk * AT_QBLK, blk * 64, g * p.G,
                     b * rows_per_robot + qt * p.TQ, pol_q, el);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cta_sync();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t o_col = 256;

  if (warp == 0) {
    // K units and V halves, each as soon as its slot is free
    uint32_t spins = 0;   // polls without progress (kPollLimit of them take seconds)
    bool ok = true;
    while (ok && (kc < c1 || vc < c1)) {
      bool progress = false;
      if (kc < c1 && mbar_test_warp(&k_empty[sk], phk)) {
        next_k();
        progress = true;
      }
      if (vc < c1 && mbar_test_warp(&v_empty[sv], phv)) {
        next_v();
        progress = true;
      }
      spins = progress ? 0u : spins + 1u;
      if (spins > kPollLimit) ok = false;
    }
    if (lane == 0) {
      if (!ok) flags[0] = 1;
      flags[1] = nk;
      flags[3] = nv;
    }
    __syncwarp();
  } else if (warp == 1) {
    el = elect_one();
    const uint32_t idesc_s = idesc_bf16(AT_BM, AT_BKV);
    const uint32_t idesc_o = idesc_bf16_bmn(AT_BM, p.hdp);
    const uint64_t qd0 = sw128_desc(q0), kd0 = sw128_desc(k0), vd0 = sw128_mn_desc(v0, AT_VBLK);
    bool ok = mbar_wait_warp(q_full, 0);
    // Issue S of the next chunk and PV of the oldest chunk whose P is ready,
    // whichever can go: PV(i) never waits for chunk i+1's K/V (that would
    // chain every chunk's load behind the previous PV).  S runs at most one
    // chunk ahead of PV (two S buffers in TMEM).
    int ns = 0, i = 0;   // next S, next PV
    int uk = 0, uv = 0;  // K units and V halves consumed
    bool sdone_sent = false;
    // xch: every split learns when this split's last S has completed
    // (its Q and K ring may then receive the partials of the merge)
    const uint16_t smask = (uint16_t)((1u << p.splits) - 1u);
    phk = phv = 0;
    uint32_t spins = 0;   // polls without progress (kPollLimit of them take seconds)
    while (ok && i < n) {
      bool progress = false;
      if (ns < n && ns <= i + 1 && mbar_test_warp(&k_full[sk], phk)) {
        const uint32_t sd = tmem + (uint32_t)(ns & 1) * AT_BKV;
        uint64_t ad = qd0;
        #pragma unroll 1
        for (int blk = 0; blk < p.nblk; ++blk, ad += AT_QBLK >> 4) {
          if (blk) ok = mbar_wait_warp(&k_full[sk], phk);   // (the first is known to have arrived)
          if (!ok) break;
          tc_fence_after();
          const uint64_t bd = kd0 + (uint32_t)sk * (AT_KUNIT >> 4);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            umma_bf16(sd, ad + 2 * k, bd + 2 * k, idesc_s, (blk > 0 || k > 0) ? 1u : 0u, el);
          umma_commit(&k_empty[sk], el);
          ++uk;
          if (++sk == SK) {
            sk = 0;
            phk ^= 1u;
          }
        }
        if (!ok) break;
        umma_commit(&s_full[ns & 1], el);
        ++ns;
        if (p.xch && ns == n) {
          umma_commit_mc(sdone, smask, el);
          sdone_sent = true;
        }
        progress = true;
      }
      if (i < ns && mbar_test_warp(&p_full[i & 1], (uint32_t)(i >> 1) & 1u) && mbar_test_warp(&v_full[sv], phv)) {
        // A = P from TMEM (the S tile's first 64 columns, two bf16 per column),
        // B = V [64 keys][hd], MN-major: 16 keys (two 8-row groups) per MMA, only
        // the groups that hold keys
        const uint32_t pa = tmem + (uint32_t)(i & 1) * AT_BKV;
        const int groups = (keys_of(c0 + i) + 15) >> 4;
        #pragma unroll 1
        for (int h = 0; 4 * h < groups; ++h) {
          if (h) ok = mbar_wait_warp(&v_full[sv], phv);   // (as above)
          if (!ok) break;
          tc_fence_after();
          const uint64_t bd = vd0 + (uint32_t)sv * (v_bytes >> 4);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (4 * h + k < groups)
              umma_bf16_ts(tmem + o_col, pa + 8 * (4 * h + k), bd + 128 * k, idesc_o, (i + h + k > 0) ? 1u : 0u, el);
          umma_commit(&v_empty[sv], el);
          ++uv;
          if (++sv == SV) {
            sv = 0;
            phv ^= 1u;
          }
        }
        if (!ok) break;
        umma_commit(&pv_done[i & 1], el);
        ++i;
        progress = true;
      }
      spins = progress ? 0u : spins + 1u;
      if (spins > kPollLimit) ok = false;
    }
    // (no chunk, or an abort: arrive all the same, once earlier MMAs are done)
    if (p.xch && !sdone_sent) umma_commit_mc(sdone, smask, el);
    if (lane == 0) {
      if (!ok) flags[0] = 1;
      flags[2] = uk;   // K units whose arrival was consumed
      flags[4] = uv;   // V halves whose arrival was consumed
    }
    __syncwarp();
  } else {
    // softmax / epilogue: two threads per query row r (TMEM lane r), half hf = 0, 1
    const int q4 = warp & 3, hf = warp >= 6 ? 1 : 0;
    const int r = q4 * 32 + lane;
    auto pair_bar = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + q4) : "memory"); };   // warps w and w + 4
    const uint32_t lane_base = tmem + ((uint32_t)(q4 * 32) << 16);
    const int t = r / p.G;
    const int j = qt * p.TQ + t;
    float m_used = -INFINITY, l = 0.f;   // running max (log2 domain, scaled) of the row, sum of this half's P
    bool ok = true;
    int i = 0;
    const float sl2 = p.scale_log2;
    // (after a wait that ran out the loop goes on without waiting, so that the
    // two warps of a pair meet at every barrier)
    for (int c = c0; c < c1; ++c) {
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&s_full[i & 1], (uint32_t)(i >> 1) & 1u));
      tc_fence_after();
      float sc[64];   // this half's keys 64 hf .. 64 hf + 63 of the chunk
      {
        uint32_t raw[64];
        const uint32_t srow = lane_base + (uint32_t)(i & 1) * AT_BKV + 64 * hf;
#pragma unroll
        for (int q = 0; q < 4; ++q) tmem_ld16_async(srow + 16 * q, raw + 16 * q);
        tmem_wait_ld();
#pragma unroll
        for (int q = 0; q < 4; ++q) tmem_reg_fence16(raw + 16 * q);
#pragma unroll
        for (int k = 0; k < 64; ++k) sc[k] = __uint_as_float(raw[k]);
      }
      // keys of the chunk that do not exist and, in the slot-isolated test mode,
      // that are not visible count as -inf
      const int kleft = keys_of(c) - 64 * hf;
      if (kleft < 64) {
#pragma unroll
        for (int k = 0; k < 64; ++k) sc[k] = k < kleft ? sc[k] : -INFINITY;
      }
      const int own0 = (c - npv) * AT_BKV + 64 * hf;   // the step's own keys: index of this half's first
      if (p.mask_mode == 1 && c >= npv && own0 < p.H) {
#pragma unroll
        for (int k = 0; k < 64; ++k)
          if (own0 + k < p.H && own0 + k != j) sc[k] = -INFINITY;
      }
      float m8[8];
#pragma unroll
      for (int a = 0; a < 8; ++a)
        m8[a] = fmaxf(fmaxf(fmaxf(sc[8 * a], sc[8 * a + 1]), fmaxf(sc[8 * a + 2], sc[8 * a + 3])),
                      fmaxf(fmaxf(sc[8 * a + 4], sc[8 * a + 5]), fmaxf(sc[8 * a + 6], sc[8 * a + 7])));
      // the row's maximum over both halves; past the first barrier both have
      // read their scores (P may overwrite them), past the second the maxima
      xm[hf * 128 + r] =
          fmaxf(fmaxf(fmaxf(m8[0], m8[1]), fmaxf(m8[2], m8[3])), fmaxf(fmaxf(m8[4], m8[5]), fmaxf(m8[6], m8[7])));
      pair_bar();
      const float mx = fmaxf(xm[r], xm[128 + r]) * sl2;
      pair_bar();
      const float m_new = fmaxf(m_used, mx);
      const bool need = m_new > m_used + 8.f;
      if (i > 0 && __any_sync(0xffffffffu, need)) {
        // O must hold PV of every earlier chunk before it is rescaled
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&pv_done[(i - 1) & 1], (uint32_t)((i - 1) >> 1) & 1u));
        tc_fence_after();
        const float alpha = need ? exp2f(m_used - m_new) : 1.f;   // exp2(-inf) = 0
        for (int cb = 16 * hf; cb < p.hdp; cb += 32) {   // (the halves take alternate columns)
          float o[16];
          tmem_ld16(lane_base + o_col + cb, o);
#pragma unroll
          for (int q = 0; q < 16; ++q) o[q] *= alpha;
          tmem_st16(lane_base + o_col + cb, o);
        }
        tmem_wait_st();
        l *= alpha;
      }
      if (need) m_used = m_new;
      const float nb = (m_used == -INFINITY) ? 0.f : -m_used;
      // P (bf16) overwrites the first 64 columns of this chunk's S tile, 32 of
      // them this half's: S of chunk i + 2 reuses the tile only after PV of chunk
      // i has been issued, and the tensor pipe runs them in order
      const uint32_t prow = lane_base + (uint32_t)(i & 1) * AT_BKV + 32 * hf;
      float ls[8];
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2) {
        uint32_t w[16];
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          float e[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) e[q] = fast_exp2(fmaf(sc[32 * h2 + 8 * ch + q], sl2, nb));
          ls[4 * h2 + ch] = ((e[0] + e[1]) + (e[2] + e[3])) + ((e[4] + e[5]) + (e[6] + e[7]));
#pragma unroll
          for (int q = 0; q < 4; ++q) w[4 * ch + q] = pack_bf16x2(e[2 * q], e[2 * q + 1]);
        }
        tmem_st16u(prow + 16 * h2, w);
      }
      tmem_wait_st();
      l += ((ls[0] + ls[1]) + (ls[2] + ls[3])) + ((ls[4] + ls[5]) + (ls[6] + ls[7]));
      tc_fence_before();
      mbar_arrive(&p_full[i & 1]);
      ++i;
    }
    if (ok && n > 0) {
      ok = __all_sync(0xffffffffu, mbar_wait(&pv_done[(n - 1) & 1], (uint32_t)((n - 1) >> 1) & 1u));
      tc_fence_after();
    }
    if (!ok && lane == 0) flags[0] = 1;
    {   // the row's sum of P over both halves
      xm[hf * 128 + r] = l;
      pair_bar();
      l = xm[r] + xm[128 + r];
    }
    if (p.xch) {
      // every split's S MMAs are done: their Q and K rings, where the
      // partials land, are no longer read
      const bool okd = __all_sync(0xffffffffu, mbar_wait_cluster(sdone, 0));
      if (!okd && lane == 0) flags[0] = 1;
    }
    if (p.splits == 1) {
      // O / l as bf16 into Q's place and layout (every S has completed), from
      // where one TMA store per 64 head dims writes the tile's slots; the output
      // map clips the slots past H (a bulk copy per row took each warp 32 issues)
      const float inv = (l > 0.f && n > 0) ? 1.f / l : 0.f;
      for (int cb = 32 * hf; cb < p.hdp; cb += 64) {   // (the halves take alternate 32 columns)
        uint32_t raw[32];
        tmem_ld32_async(lane_base + o_col + cb, raw);
        tmem_wait_ld();
        tmem_reg_fence16(raw);
        tmem_reg_fence16(raw + 16);
        uint8_t* row = q_s + (size_t)(cb >> 6) * AT_QBLK + (size_t)r * 128;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint4 w;
          w.x = pack_bf16x2(__uint_as_float(raw[8 * q]) * inv, __uint_as_float(raw[8 * q + 1]) * inv);
          w.y = pack_bf16x2(__uint_as_float(raw[8 * q + 2]) * inv, __uint_as_float(raw[8 * q + 3]) * inv);
          w.z = pack_bf16x2(__uint_as_float(raw[8 * q + 4]) * inv, __uint_as_float(raw[8 * q + 5]) * inv);
          w.w = pack_bf16x2(__uint_as_float(raw[8 * q + 6]) * inv, __uint_as_float(raw[8 * q + 7]) * inv);
          *(uint4*)(row + ((((cb & 32) >> 3) + q) ^ (r & 7)) * 16) = w;   // 128-byte swizzle
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("bar.sync 5, 256;" ::: "memory");
      if (warp == 2 && vrows > 0) {
        el = elect_one();
        #pragma unroll 1
        for (int blk = 0; blk < p.nblk; ++blk)
          tma_store_4d_el(&maps.o, q0 + (uint32_t)blk * AT_QBLK, blk * 64, g * p.G, qt * p.TQ, b, el);
        bulk_commit();
        bulk_wait_read<0>();   // read out before the shared memory goes away
      }
    } else if (p.xch) {
      // rows holding a slot: (m, l) to every rank; O / l as bf16, head-dim
      // slice q to rank q, starting with this split's own slice so that the
      // splits send to different ranks at any moment.  The TMEM loads are
      // warp-collective: every lane runs them, only rows that hold a slot send.
      const bool snd = r < vrows;
      const bool has = n > 0 && !(l <= 0.f);   // (a sum that is not a number goes out as it is)
      const float inv = has ? 1.f / l : 0.f;
      const int ngs = cps / 8;
      const uint32_t base = smem_u32(smem);
      const uint32_t o0 = base + (uint32_t)(split * ngs * AT_BM + r) * 16u;
      const uint32_t bar0 = smem_u32(rcv_bar);
      if (snd && hf == 0) {
        const uint32_t ml0 = base + (uint32_t)(p.splits * ngs * AT_BM) * 16u + (uint32_t)(split * AT_BM + r) * 8u;
        const float m_s = has ? m_used : -INFINITY, l_s = has ? l : 0.f;
        for (int q = 0; q < p.splits; ++q) st_async_f2(mapa_shared(ml0, (uint32_t)q), m_s, l_s, mapa_shared(bar0, (uint32_t)q));
      }
      // 32 columns per TMEM load (16 where hdp is not a multiple of 32), the
      // next load in flight while this one goes out
      const int cw = (p.hdp % 32 == 0) ? 32 : 16;
      const int nch = p.hdp / cw, nown = (nch + 1 - hf) / 2;   // the halves take alternate chunks
      int ch = ((split * cps) / cw + hf) % nch;
      uint32_t cur[32];
      if (cw == 32 && nown) tmem_ld32_async(lane_base + o_col + 32 * ch, cur);
      else if (nown) tmem_ld16_async(lane_base + o_col + 16 * ch, cur);
      tmem_wait_ld();
      tmem_reg_fence16(cur);
      tmem_reg_fence16(cur + 16);
      for (int jj = 0; jj < nown; ++jj) {
        const int chn = ch + 2 >= nch ? ch + 2 - nch : ch + 2;
        uint32_t nxt[32];
        if (jj + 1 < nown) {
          if (cw == 32) tmem_ld32_async(lane_base + o_col + 32 * chn, nxt);
          else tmem_ld16_async(lane_base + o_col + 16 * chn, nxt);
        }
        if (snd) {
          // groups of 8 columns: group g of the row goes to rank g / ngs, slot
          // g % ngs there (one division per chunk, then a running count)
          const int gidx0 = (cw / 8) * ch;
          int dst = gidx0 / ngs, gl = gidx0 - dst * ngs;
          auto send8 = [&](int h) {
            uint4 w;
            w.x = pack_bf16x2(__uint_as_float(cur[8 * h]) * inv, __uint_as_float(cur[8 * h + 1]) * inv);
            w.y = pack_bf16x2(__uint_as_float(cur[8 * h + 2]) * inv, __uint_as_float(cur[8 * h + 3]) * inv);
            w.z = pack_bf16x2(__uint_as_float(cur[8 * h + 4]) * inv, __uint_as_float(cur[8 * h + 5]) * inv);
            w.w = pack_bf16x2(__uint_as_float(cur[8 * h + 6]) * inv, __uint_as_float(cur[8 * h + 7]) * inv);
            if (!has) w = make_uint4(0u, 0u, 0u, 0u);   // no key: the accumulator was never written
            st_async_u4(mapa_shared(o0 + (uint32_t)gl * (AT_BM * 16), (uint32_t)dst), w,
                        mapa_shared(bar0, (uint32_t)dst));
            const bool wrap = ++gl == ngs;
            gl = wrap ? 0 : gl;
            dst += wrap ? 1 : 0;
          };
          send8(0);
          send8(1);
          if (cw == 32) {
            send8(2);
            send8(3);
          }
        }
        if (jj + 1 < nown) {
          tmem_wait_ld();
          tmem_reg_fence16(nxt);
          tmem_reg_fence16(nxt + 16);
#pragma unroll
          for (int k = 0; k < 32; ++k) cur[k] = nxt[k];
        }
        ch = chn;
      }
    } else {
      // unnormalised partial O as [ti][d/4][row][4] (a warp stores one
      // contiguous 512-byte run per 4 columns), plus this split's (m, l)
      const size_t ti = ((size_t)bg * gridDim.x + qt) * p.splits + split;
      float* dst = p.ws_o + ti * (size_t)(p.hdp / 4) * 512 + (size_t)r * 4;
      for (int cb = 64 * hf; cb < p.hdp; cb += 128) {   // up to four TMEM loads in flight, one wait
        const int nq = min(4, (p.hdp - cb) / 16);
        uint32_t raw[64];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < nq) tmem_ld16_async(lane_base + o_col + cb + 16 * q, raw + 16 * q);
        tmem_wait_ld();
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (q < 4 * nq)
            __stcg((float4*)(dst + (size_t)(cb / 4 + q) * 512),
                   (n > 0) ? make_float4(__uint_as_float(raw[4 * q]), __uint_as_float(raw[4 * q + 1]),
                                         __uint_as_float(raw[4 * q + 2]), __uint_as_float(raw[4 * q + 3]))
                           : make_float4(0.f, 0.f, 0.f, 0.f));
      }
      if (hf == 0) {
        __stcg(p.ws_ml + (ti * 2) * AT_BM + r, (n > 0) ? m_used : -INFINITY);
        __stcg(p.ws_ml + (ti * 2 + 1) * AT_BM + r, (n > 0) ? l : 0.f);
      }
      __threadfence();
    }
  }
  tc_fence_before();
  cta_sync();
  if (flags[0]) {
    if (threadIdx.x == 0) {
      for (int i = flags[2]; i < flags[1]; ++i) mbar_wait(&k_full[i % SK], (uint32_t)(i / SK) & 1u);
      for (int i = flags[4]; i < flags[3]; ++i) mbar_wait(&v_full[i % SV], (uint32_t)(i / SV) & 1u);
      raise_error(p.err, ERR_TIMEOUT);
    }
    cta_sync();
  }
  if (p.xch) {
    // Rank q merges head-dim columns [q*cps, (q+1)*cps) of its rows once every
    // split's share has arrived (the wait also keeps this CTA alive until no
    // store into its shared memory is in flight):
    //   O = sum_s 2^(m_s - M) l_s Ohat_s / sum_s 2^(m_s - M) l_s,  Ohat_s = O_s / l_s.
    // Every warp takes part (the producer and MMA warps are idle by now):
    // work item (row r, 8-column group gq) of this rank's slice.
    {
      const bool ok = __all_sync(0xffffffffu, mbar_wait_cluster(rcv_bar, 0));
      if (!ok) {
        if (lane == 0) raise_error(p.err, ERR_TIMEOUT);
      } else {
        const int ngs = cps / 8, items = vrows * ngs;
        const uint32_t og = smem_u32(smem);
        const uint32_t ml = og + (uint32_t)(p.splits * ngs * AT_BM) * 16u;
        for (int it = threadIdx.x; it < items; it += AT_THREADS) {
          const int r = it % vrows, gq = it / vrows;
          const int t = r / p.G, hh = r % p.G;
          const int j = qt * p.TQ + t;
          bf16* orow = p.out + (size_t)(b * p.H + j) * p.ld_out + (size_t)(g * p.G + hh) * p.hd;
          switch (p.splits) {
            case 2: xch_combine_group<2>(og, ml, r, ngs, gq, split * cps, p.hd, orow); break;
            case 4: xch_combine_group<4>(og, ml, r, ngs, gq, split * cps, p.hd, orow); break;
            case 8: xch_combine_group<8>(og, ml, r, ngs, gq, split * cps, p.hd, orow); break;
            default: xch_combine_group<16>(og, ml, r, ngs, gq, split * cps, p.hd, orow); break;
          }
        }
      }
    }
  } else if (p.splits > 1) {
    // The key splits of this query tile form a cluster: once every split has
    // published its (O, m, l), rank q merges head-dim columns
    // [q*hdp/S, (q+1)*hdp/S):  O = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s.
    cluster_sync();
    if (warp >= 2 && warp < 6) {
      const int r = (warp & 3) * 32 + lane;
      const int Sp = p.splits;
      const int cps = p.hdp / Sp;   // a multiple of 4
      const int rank = (int)cluster_ctarank();
      const size_t t0 = ((size_t)bg * gridDim.x + qt) * Sp;
      float wgt[16];
      float M = -INFINITY, L = 0.f;
#pragma unroll
      for (int s2 = 0; s2 < 16; ++s2) {
        wgt[s2] = -INFINITY;
        if (s2 >= Sp) continue;
        wgt[s2] = __ldcg(p.ws_ml + ((t0 + s2) * 2) * AT_BM + r);
        M = fmaxf(M, wgt[s2]);
      }
#pragma unroll
      for (int s2 = 0; s2 < 16; ++s2) {
        if (s2 >= Sp) break;
        const float l_s = __ldcg(p.ws_ml + ((t0 + s2) * 2 + 1) * AT_BM + r);
        wgt[s2] = (wgt[s2] == -INFINITY) ? 0.f : exp2f(wgt[s2] - M);
        L += wgt[s2] * l_s;
      }
      const float inv = L > 0.f ? 1.f / L : 0.f;
      const int t = r / p.G, hh = r % p.G;
      const int j = qt * p.TQ + t;
      const bool row_ok = (r < p.TQ * p.G) && (j < p.H);
      bf16* orow = p.out + (size_t)(b * p.H + j) * p.ld_out + (size_t)(g * p.G + hh) * p.hd;
      const float* src0 = p.ws_o + t0 * (size_t)(p.hdp / 4) * 512 + (size_t)r * 4;
      const size_t sstride = (size_t)(p.hdp / 4) * 512;
      const int c4b = rank * cps / 4, c4e = (rank + 1) * cps / 4;
      switch (Sp) {
        case 2: combine_slice<2>(src0, sstride, c4b, c4e, wgt, inv, orow, p.hd, row_ok); break;
        case 4: combine_slice<4>(src0, sstride, c4b, c4e, wgt, inv, orow, p.hd, row_ok); break;
        case 8: combine_slice<8>(src0, sstride, c4b, c4e, wgt, inv, orow, p.hd, row_ok); break;
        default: combine_slice<16>(src0, sstride, c4b, c4e, wgt, inv, orow, p.hd, row_ok); break;
      }
    }
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
  }
}

PFN_cuTensorMapEncodeTiled_v12000 g_enc = nullptr;
struct AtClusters {
  int n[4];   // resident clusters of 2, 4, 8, 16 CTAs (0: not to be had)
};
AtClusters g_attn_clusters = {{0, 0, 0, 0}};

cudaError_t enc3(CUtensorMap* m, const void* base, uint64_t d0, uint64_t d1, uint64_t d2, uint64_t s1_bytes,
                 uint64_t s2_bytes, uint32_t b0, uint32_t b1, uint32_t b2) {
  cuuint64_t dims[3] = {d0, d1, d2};
  cuuint64_t strides[2] = {s1_bytes, s2_bytes};
  cuuint32_t box[3] = {b0, b1, b2};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = g_enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Rows as (hd, heads, rows of a group, groups), boxes of 64 x heads_box x rows_box
// x 1: rows past the group's own are clipped (stores) or zeros (loads).
cudaError_t enc4(CUtensorMap* m, const void* base, int hd, int heads, int rows, uint64_t groups, uint64_t row_bytes,
                 int heads_box, int rows_box, bool load) {
  cuuint64_t dims[4] = {(cuuint64_t)hd, (cuuint64_t)heads, (cuuint64_t)rows, (cuuint64_t)groups};
  cuuint64_t strides[3] = {(cuuint64_t)hd * 2, (cuuint64_t)row_bytes, (cuuint64_t)rows * row_bytes};
  cuuint32_t box[4] = {64, (cuuint32_t)heads_box, (cuuint32_t)rows_box, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = g_enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     load ? CU_TENSOR_MAP_L2_PROMOTION_L2_256B : CU_TENSOR_MAP_L2_PROMOTION_NONE,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// How a launch is cut: query tiles, key splits and how they merge, ring depths.
struct AtPlan {
  int q_tiles = 0, TQ = 0, splits = 1;
  bool smem_merge = false;   // partials normalised, in bf16, through shared memory; else fp32 through L2
  int k_slots = 0, v_slots = 0;
  size_t smem = 0;
};

// The most splits that 64-key pieces, two each, and SMs that half the grid leaves
// idle allow.  It is what the precision goes by, not the plan of least time: with
// one, keys are not split at all (a split rounds its share to bf16), and where its
// head-dim slices are not whole 8-column groups the partials stay in fp32
// through L2 however few the splits are (head dim 64 with 16 splits, 80, 96).
int most_splits(const AttnTcArgs& a, int hdp, bool clusters_of_16) {
  const int G = a.Hq / a.Hkv, pairs = a.B * a.Hkv;
  const int pieces = (a.Pmax + 63) / 64 + (a.H + a.F + 63) / 64;
  auto tiles = [&](int rows) { return (a.H + std::max(1, rows / G) - 1) / std::max(1, rows / G); };
  int qt = tiles(AT_BM);
  const int tq = (a.H + qt - 1) / qt, qt64 = tiles(64);
  if (qt * pairs * 2 <= a.num_sms && std::max(1, 64 / G) < tq && qt64 * pairs * 8 <= a.num_sms / 2 && pieces >= 3)
    qt = qt64;
  const int ctas = qt * pairs;
  if (ctas * 2 > a.num_sms) return 1;
  const int cap = std::min({(pieces + 1) / 2, a.num_sms / ctas, clusters_of_16 ? 16 : 8});
  int s = 1;
  while (s * 2 <= cap && (hdp / (s * 2)) % 4 == 0 && (size_t)(s * 2) * ctas * AT_BM * (hdp + 2) * 4 <= a.ws_bytes) s *= 2;
  return s;
}

AtPlan plan_attention(const AttnTcArgs& a, const AtClusters& clusters) {
  AtPlan p;
  const int G = a.Hq / a.Hkv, hdp = (a.hd + 15) / 16 * 16, nblk = (a.hd + 63) / 64;
  const int most = most_splits(a, hdp, clusters.n[3] > 0);
  // Query tiles of 128 rows, or of 64 where the keys are split (32: one robot's
  // 104 CTAs, 612 us per step against 601), and the number of key splits (one
  // cluster per query tile, a power of two whose head-dim slices are multiples
  // of 4 columns): the least estimated time, fitted to whole steps of 1 to 16
  // robots with every tile height and split count.  A CTA costs about 4 us and
  // each chunk 1.65 at head dim 256 (the tensor pipe's turns of S and P V), 0.95
  // at 64 (the softmax); the merge moves every split's rows x hd partial
  // between the SMs; CTAs past half the SMs delay the next kernel's; a grid that
  // does not fit at once (36 clusters of 4, 15 of 8, 7 of 16) takes another
  // round.  16 robots, 16 slots, 2048 keys: 4 splits of 64 rows, 964 us; of 128
  // rows 1005, 2 splits 1061, 8 (16 clusters in two rounds) 1118.
  const int C = (a.Pmax + AT_BKV - 1) / AT_BKV + (a.H + a.F + AT_BKV - 1) / AT_BKV;
  const float hd_rel = (float)hdp / 256.f;
  const float t_chunk = std::max(0.95f, 1.65f * hd_rel);
  float cost = 3.4e38f;
  auto consider = [&](int rows, int splits, int resident) {
    const int tq = std::max(1, rows / G);
    const int qt = (a.H + tq - 1) / tq, ctas = qt * a.B * a.Hkv;
    const int rounds = (ctas + resident - 1) / resident, half = a.num_sms / 2;
    float t = (float)rounds * (4.f + t_chunk * (float)((C + splits - 1) / splits));
    if (splits > 1) {
      const float tile_rows = (float)((a.H + qt - 1) / qt * G);
      t += (float)rounds * hd_rel * (2.4f + 1.5f * tile_rows / 128.f);
      t += 0.6f * (float)std::max(0, ctas * splits - half) / (float)half;
    }
    if (t < cost) {
      cost = t;
      p.q_tiles = qt;
      p.TQ = (a.H + qt - 1) / qt;
      p.splits = splits;
    }
  };
  consider(AT_BM, 1, a.num_sms);
  for (int i = 0; i < 4 && most > 1; ++i) {
    const int sp = 2 << i;
    if (sp >= 2 * C || (hdp / sp) % 4 != 0 || hdp % sp != 0 || !clusters.n[i]) break;
    for (int rows = AT_BM; rows >= 64; rows /= 2) {
      const int tq = std::max(1, rows / G);
      const size_t ctas = (size_t)((a.H + tq - 1) / tq) * a.B * a.Hkv;
      if ((size_t)sp * ctas * AT_BM * (hdp + 2) * 4 <= a.ws_bytes) consider(rows, sp, clusters.n[i]);
    }
  }
  p.smem_merge = p.splits > 1 && (hdp / most) % 8 == 0 && (hdp / p.splits) % 8 == 0;
  // K units and V halves beside Q: at head dim 256 one chunk's four units and
  // three halves; smaller heads have room for more.  (The receive area of a merge
  // -- 128 rows of bf16, as large as Q, and (m, l) of up to 16 splits, 16 KB --
  // always lies in Q and the K ring.)
  const size_t v_bytes = (size_t)nblk * AT_VBLK;
  const size_t fixed = 1024 + (size_t)nblk * AT_QBLK + 512 + 1024;   // alignment, Q, barriers, row maxima / sums
  p.k_slots = nblk == 4 ? 4 : nblk == 1 ? 8 : 6;
  p.v_slots = (int)std::min<size_t>(8, (AT_SMEM_MAX - fixed - p.k_slots * AT_KUNIT) / v_bytes);
  p.smem = fixed + (size_t)p.k_slots * AT_KUNIT + (size_t)p.v_slots * v_bytes;
  return p;
}

}  // namespace

cudaError_t init_attention_tc() {
  if (!g_enc) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess) return e;
    if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorSymbolNotFound;
    g_enc = (PFN_cuTensorMapEncodeTiled_v12000)fn;
  }
  cudaError_t e = cudaFuncSetAttribute(attn_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AT_SMEM_MAX);
  if (e != cudaSuccess) return e;
  const bool big = cudaFuncSetAttribute(attn_tc_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  for (int i = 0; i < (big ? 4 : 3); ++i) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 2u << i;
    cfg.gridDim = dim3(1, 1, 2u << i);
    cfg.blockDim = dim3(AT_THREADS);
    cfg.dynamicSmemBytes = AT_SMEM_MAX;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    g_attn_clusters.n[i] = cudaOccupancyMaxActiveClusters(&n, attn_tc_kernel, &cfg) == cudaSuccess && n > 0 ? n : 0;
  }
  cudaGetLastError();
  return cudaSuccess;
}

bool attention_tc_supported(int hd, int G) { return hd % 8 == 0 && hd <= 256 && G >= 1 && G <= 128; }

cudaError_t launch_attention_tc(const AttnTcArgs& a, cudaStream_t st) {
  if (!g_enc) return cudaErrorInitializationError;
  AtParams p{};
  p.H = a.H; p.F = a.F; p.Hkv = a.Hkv; p.G = a.Hq / a.Hkv; p.hd = a.hd;
  p.hdp = (a.hd + 15) / 16 * 16;
  p.Pmax = a.Pmax;
  p.n_kv = (a.H + a.F + AT_BKV - 1) / AT_BKV;
  p.layer = a.layer; p.Bmax = a.Bmax; p.mask_mode = a.mask_mode;
  p.nblk = (a.hd + 63) / 64;
  p.ctx_state = a.ctx_state;
  for (int s = 0; s < 2; ++s) {
    p.ck[s] = (const bf16*)a.ctx_k[s];
    p.cv[s] = (const bf16*)a.ctx_v[s];
  }
  p.out = (bf16*)a.out; p.ld_out = a.ld_out;
  p.err = a.err;
  p.scale_log2 = 1.4426950408889634f / sqrtf((float)a.hd);
  const AtPlan plan = plan_attention(a, g_attn_clusters);
  const int splits = plan.splits, nctas = plan.q_tiles * a.B * a.Hkv;
  p.q_tiles = plan.q_tiles;
  p.TQ = plan.TQ;
  p.splits = splits;
  p.xch = plan.smem_merge ? 1 : 0;
  p.ws_o = a.ws;
  p.ws_ml = a.ws + (size_t)splits * nctas * AT_BM * p.hdp;
  p.k_slots = plan.k_slots;
  p.v_slots = plan.v_slots;
  if (a.ld_out % 8 != 0 || ((uintptr_t)a.out & 15u) != 0) return cudaErrorMisalignedAddress;

  AtMaps m;
  const int hd = a.hd, rpr = a.H + a.F;
  const uint64_t rows = (uint64_t)a.B * rpr;
  cudaError_t e = enc3(&m.q, a.qkv, hd, a.Hq, rows, (uint64_t)hd * 2, (uint64_t)a.ld_qkv * 2, 64, p.G, p.TQ);
  if (e == cudaSuccess)
    e = enc3(&m.k, (const bf16*)a.qkv + (size_t)a.Hq * hd, hd, a.Hkv, rows, (uint64_t)hd * 2, (uint64_t)a.ld_qkv * 2,
             64, 1, AT_BKV);
  if (e == cudaSuccess)
    e = enc4(&m.v, (const bf16*)a.qkv + (size_t)(a.Hq + a.Hkv) * hd, hd, a.Hkv, rpr, a.B, (uint64_t)a.ld_qkv * 2, 1,
             64, true);
  if (e == cudaSuccess) e = enc4(&m.o, a.out, hd, a.Hq, a.H, a.B, (uint64_t)a.ld_out * 2, p.G, p.TQ, false);
  const uint64_t zc = (uint64_t)(a.layers * a.Bmax * a.Hkv);
  for (int s = 0; s < 2 && e == cudaSuccess; ++s) {
    e = enc3(s ? &m.pk1 : &m.pk0, a.ctx_k[s], hd, a.Pmax, zc, (uint64_t)hd * 2, (uint64_t)a.Pmax * hd * 2, 64,
             AT_BKV, 1);
    if (e == cudaSuccess)
      e = enc4(s ? &m.pv1 : &m.pv0, a.ctx_v[s], hd, 1, a.Pmax, zc, (uint64_t)hd * 2, 1, 64, true);
  }
  if (e != cudaSuccess) return e;
  dim3 grid(p.q_tiles, a.B * a.Hkv, splits);
  e = launch_kernel_cluster(attn_tc_kernel, grid, dim3(AT_THREADS), plan.smem, st, dim3(1, 1, splits), m, p);
  return e;
}

}  // namespace ravel

// What the tensor-core attention of these sizes is cut into, for tests: out =
// {query tiles, slots per tile, key splits, 1 if they merge in bf16 through
// shared memory, shared-memory bytes}.
extern "C" void ravel_debug_attention_plan(int B, int H, int F, int Hq, int Hkv, int hd, int Pmax, size_t ws_bytes,
                                           int num_sms, const int* clusters, int* out) {
  using namespace ravel;
  AttnTcArgs a{};
  a.B = B;
  a.H = H;
  a.F = F;
  a.Hq = Hq;
  a.Hkv = Hkv;
  a.hd = hd;
  a.Pmax = Pmax;
  a.ws_bytes = ws_bytes;
  a.num_sms = num_sms;
  const AtPlan p = plan_attention(a, AtClusters{{clusters[0], clusters[1], clusters[2], clusters[3]}});
  const int v[5] = {p.q_tiles, p.TQ, p.splits, p.smem_merge, (int)p.smem};
  for (int i = 0; i < 5; ++i) out[i] = v[i];
}
