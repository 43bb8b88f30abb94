// Prefill-regime group-sparse linear with zero-filled windows (1 x 256, 1 x 128
// and square groups, Eq. 1): the tensor work is that of the dense layer, and only
// kept weights move.
//
// A unit of work is a window of 256 output rows x a tile of N <= 256 tokens,
// owned by a cluster of two CTAs: CTA r holds window rows 128 r .. 128 r + 127
// and tokens r N / 2 .. of the tile.  The weights are the MMA's A operand and
// live in tensor memory, where lane = output row, so a kept row reaches its row
// position with one tcgen05.st by the lane that owns it and a pruned row is a
// register full of zeros:
//   packed tiles --TMA box--> shared (the half window's kept rows, compact)
//     --ld.shared by kept lanes--> registers --tcgen05.st--> TMEM A slot.
// x is the B operand (TMA, 128-byte swizzle).  Per K stage (128 deep, or 256 at N <= 128)
// the leader issues M = 256 x N x 16 cta_group::2 MMAs; D^T (rows x tokens, fp32)
// stays in TMEM for the whole unit.
//
// Why this split.  Shared memory receives x (N / 2 x 256 B a stage) and the kept
// rows only, and nothing is written there by threads, so no generic-to-async
// proxy fence lies between the weights and the tensor cores.  (With the rows
// placed in shared memory by cp.async, as zero-filled B operands, the copies'
// fences and the second operand's bytes held a 7B block at T = 2048 to 576 us,
// 1.44 PFLOP/s dense-equivalent; now 478 us, 1.73 PFLOP/s, a library GEMM's sustained
// rate at the chip's power limit.)
//
// What bounds it.  At N = 256 the tensor cores.  At small N the stream of kept weights
// (5.7 TB/s) and, where units are few, the chain of hand-offs of a stage (copy ->
// converters -> leader -> commit), about 0.35 us however deep the stage is: 13B block at
// T = 32 / 128 in 58 / 67 us with 256-deep stages, 71 / 76 us with 128.  The roles that
// issue MMAs and copies walk their stages with the whole warp and issue from one elected
// lane: inside a one-lane branch an MMA cost 70 cycles of issue and a copy 220 to 400
// (13B block at T = 128, 128-deep: 92 us).
//
// Roles (one CTA per SM, units persistent over the pairs): warp 0 x copies,
// warp 1 W copies, warp 2 TMEM allocator + MMA issuer (leader), warps 4..11
// converters (TMEM lane quarter warp & 3; two sets of four warps take the stages
// in turn), warps 12..19 epilogue (lane quarter warp & 3, half of the tokens
// each).  The epilogue packs its columns to bf16 in registers and hands D back
// before it stores, so a single D buffer costs the next unit only that read;
// tiles of up to 64 tokens have two.  Every wait is bounded.
#include "gs_common.cuh"
#include "gs_sm100.cuh"

#include <cuda.h>
#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

namespace gs {
namespace {
using namespace sm100;

constexpr int kDW = 256;                          // output rows per window (M of each MMA)
constexpr int kDHalf = kDW / 2;                   // window rows each CTA holds (TMEM lanes)
constexpr int kDN = 256;                          // most tokens per tile (N of each MMA)
constexpr int kDBoxK = 128;                       // k per copy: two 64-wide slabs
constexpr int kDMaxXSlots = 8;                    // x slots (shared), at most
constexpr int kDWSeq = 16;                        // W stages in flight, at most
constexpr int kDConvWarp0 = 4, kDConvSets = 2, kDConvWarps = 4 * kDConvSets;   // a set per stage, in turn
constexpr int kDEpiWarp0 = kDConvWarp0 + kDConvWarps, kDEpiWarps = 8;
constexpr int kDThreads = (kDEpiWarp0 + kDEpiWarps) * 32;
constexpr int kDMmaWarp = 2;
constexpr uint32_t kDTmemCols = 512;              // D first, then the A slots of SK / 2 columns each
constexpr int kDMaxLayers = 8;
constexpr int kDMaxChunks = 32767;                // wider inputs stay on the other kernels
constexpr int kDWMaps = 8;                        // W box heights: 16, 32, ..., 128 rows (square: g, 2g, ..., 128)
constexpr uint64_t kDWaitLimitNs = 2000000000ull;
constexpr uint64_t kDDrainLimitNs = 200000000ull;
// Shared memory: x slots of the tile's own size first, the rest is a byte ring
// for the kept rows, whose stages vary with the density: what is in flight is
// bytes that move, not slots sized for a full window.
constexpr int kDRing = 224 * 1024;
constexpr int kDSmem = kDRing + 1024;
static_assert(kDSmem <= 226 * 1024, "shared memory budget");
// A stage carries SK = 128 k, or 256 for tiles of up to 128 tokens (whose MMAs
// are short: a stage then costs its hand-offs, about 0.35 us, however deep it is).
// x slots of a tile of n tokens (both CTAs): eight where the tile is small and the
// stage short, so that the copies' round trip is hidden
__host__ __device__ constexpr int d_x_slots(int n, int sk) {
  return sk == 256 ? (n <= 96 ? 4 : 3) : n <= kDN / 2 ? kDMaxXSlots : kDMaxXSlots / 2;
}
__host__ __device__ constexpr int d_w_ring(int n, int sk) { return kDRing - d_x_slots(n, sk) * (n / 2) * sk * 2; }
// A W stage that would straddle the ring's end starts over at 0: with every
// earlier stage released that asks for at most twice the largest stage.
constexpr bool d_ring_holds_two(int sk, int n_max) {
  for (int n = 32; n <= n_max; n += 16)
    if (d_w_ring(n, sk) < 2 * kDHalf * sk * 2) return false;
  return true;
}
static_assert(d_ring_holds_two(128, kDN) && d_ring_holds_two(256, kDN / 2), "two largest W stages fit the ring");
// TMEM columns of D (n <= 64: two buffers), and the A slots the rest holds: six
// 128-deep slots at n <= 128 measured no faster than four
__host__ __device__ constexpr uint32_t d_d_cols(int n) { return n <= kDN / 2 ? kDN / 2 : kDN; }
__host__ __device__ constexpr uint32_t d_a_slots(int n, int sk) { return (512 - d_d_cols(n)) / (uint32_t)(sk / 2); }
static_assert(d_a_slots(kDN, 128) == 4 && d_a_slots(kDN / 2, 256) == 3, "A slots no more than x slots");

struct DLayer {
  CUtensorMap xmap;          // x as (64, T, in/64) slabs, box 64 x N/2 x 2
  CUtensorMap wmap[kDWMaps]; // kept rows: 1 x KW slabs (box 64 x 16(h+1) x 2), square g x g (box g x g(h+1))
  const uint16_t* tiles;     // packed weights (square groups of 16 and 32 copy from here)
  const int32_t* win_off;    // 1 x KW: [G][nw16 + 1]; square: gwoff [in / g][nwin + 1]
  const void* kmask;         // 1 x KW: uint16 [G][nw16]; square: uint8 [in / g][nwin]
  uint16_t* y;
  float* ws;                 // n_split > 1: [32-row blocks][n_split][32 rows][16 tokens] partial sums
  int32_t* cnt;              // ... and arrival counters [32-row blocks] (zero between launches)
  int32_t out, G, nw, n_m, n_split, tile_begin;   // G: chunks of KW columns (square: of 128); nw: 16-row (square: 128-row) windows
};
struct DParams {
  DLayer L[kDMaxLayers];
  int32_t n_layers, T, N, n_tiles;
  int* err;
  uint64_t inject_ns;   // test hook: CTA pair 0 first waits this long on a word nothing sets (0 = off)
  TileList tl;          // which pair takes which units
};
static_assert(sizeof(DParams) <= 32764, "kernel parameter limit");

// atomic add with acquire-release ordering at GPU scope; returns the old value
__device__ __forceinline__ int d_atom_add_acq_rel(int32_t* p, int v) {
  int old;
  asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ int d_layer_of(const DParams& P, int t) {
  int l = 0;
  while (l + 1 < P.n_layers && P.L[l + 1].tile_begin <= t) ++l;
  return l;
}

// D (M = 256: this CTA's 128 lanes and the peer's) (+)= A (TMEM, the same lanes
// and columns in both CTAs) * B^T (N rows, half in each CTA's shared memory)
__device__ __forceinline__ void mma_bf16_ts_pair(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                                 uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tmem_st_x32(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
      "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]),
      "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]),
      "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
      : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t saddr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(saddr) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t d_pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// An item is kCh chunks (of KW columns; square: of 128) that share a stage, or one
// chunk of one or more stages.
template <int kCh>
__device__ __forceinline__ int d_n_items(const DLayer& L) {
  return kCh == 1 ? L.G : (L.G + kCh - 1) / kCh;
}
// Whether item c of window w has MMAs: 1 x KW items with a kept row in the
// window (square groups: every item)
template <int SQ, int kCh>
__device__ __forceinline__ bool d_nonempty(const DLayer& L, int w, int c) {
  if (c >= d_n_items<kCh>(L)) return false;
  if constexpr (SQ > 0) return true;
  const int lo = w * (kDW / kWin16), hi = min(lo + kDW / kWin16, L.nw);
  bool ne = false;
#pragma unroll
  for (int h = 0; h < kCh; ++h) {
    const int32_t* wo = L.win_off + (int64_t)min(c * kCh + h, L.G - 1) * (L.nw + 1);
    ne |= wo[hi] > wo[lo];
  }
  return ne;
}
// A unit: window w, token tile m, and items i0 .. i1 - 1 (part sp of n_split)
struct DUnit {
  int w, m, sp, i0, i1;
};
template <int kCh, bool kSplit>
__device__ __forceinline__ DUnit d_unit(const DLayer& L, int u) {
  DUnit U;
  int lt = u - L.tile_begin;
  U.m = lt % L.n_m;
  U.w = lt / L.n_m;
  U.sp = 0;
  U.i0 = 0;
  U.i1 = d_n_items<kCh>(L);
  if constexpr (kSplit) {
    const int n = U.i1;
    U.sp = U.w % L.n_split;
    U.w /= L.n_split;
    U.i0 = U.sp * n / L.n_split;
    U.i1 = (U.sp + 1) * n / L.n_split;
  }
  return U;
}
// this lane's share of the number of items of a unit that have MMAs (summed over the warp later)
template <int SQ, int kCh>
__device__ __forceinline__ int d_count_part(const DLayer& L, const DUnit& U, int lane) {
  int n = 0;
  for (int c = U.i0 + lane; c < U.i1; c += 32) n += d_nonempty<SQ, kCh>(L, U.w, c) ? 1 : 0;
  return n;
}

__device__ __forceinline__ bool d_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err) {
  return mbar_wait_bounded(bar, parity, abort_flag, err, kDWaitLimitNs, kDevErrTimeout);
}
__device__ __forceinline__ bool d_wait_cluster(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err) {
  return mbar_wait_bounded_cluster(bar, parity, abort_flag, err, kDWaitLimitNs, kDevErrTimeout);
}
// the same for a whole warp
__device__ __forceinline__ bool d_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err) {
  return __all_sync(0xffffffffu, d_wait(bar, parity, abort_flag, err));
}

// Walks a pair's units in batches of 32 items.  Lane l of a warp looks after
// item c0 + l of the batch; what it loads for the next batch is in flight while
// the warp works through this one.
template <int SQ, int kCh, bool kSplit>
struct DWalk {
  const DParams* P;
  int pair, n_pairs, ku, u, c0, c1, w, m;   // c1: end of the unit's items
  const DLayer* L;
  __device__ __forceinline__ void unit() {
    u = owner_tile(P->tl, P->n_tiles, pair, n_pairs, ku);
    if (u < 0) return;
    L = &P->L[d_layer_of(*P, u)];
    const DUnit U = d_unit<kCh, kSplit>(*L, u);
    w = U.w;
    m = U.m;
    c0 = U.i0;
    c1 = U.i1;
  }
  // item c0 + lane is in the unit
  __device__ __forceinline__ bool has(int lane) const { return u >= 0 && c0 + lane < c1; }
  __device__ __forceinline__ DWalk(const DParams& p, int pr, int n) : P(&p), pair(pr), n_pairs(n), ku(0) { unit(); }
  __device__ __forceinline__ bool valid() const { return u >= 0; }
  __device__ __forceinline__ void next() {
    c0 += 32;
    if (c0 >= c1) {
      ++ku;
      unit();
    }
  }
};
// kept rows of a 1 x KW item's chunks: first packed row of the window's two halves and the end
template <int kCh>
struct DRows {
  int a[kCh], b[kCh], c[kCh];
};
template <int SQ, int kCh, bool kSplit>
__device__ __forceinline__ DRows<kCh> d_rows(const DWalk<SQ, kCh, kSplit>& W, int lane) {
  DRows<kCh> r;
#pragma unroll
  for (int h = 0; h < kCh; ++h) {
    r.a[h] = r.b[h] = r.c[h] = 0;
    const int c = (W.c0 + lane) * kCh + h;
    if (W.has(lane) && c < W.L->G) {
      const int nw = W.L->nw, lo = W.w * (kDW / kWin16);
      const int32_t* wo = W.L->win_off + (int64_t)c * (nw + 1);
      r.a[h] = wo[lo];
      r.b[h] = wo[min(lo + kDHalf / kWin16, nw)];
      r.c[h] = wo[min(lo + kDW / kWin16, nw)];
    }
  }
  return r;
}
// kept block rows of the column blocks of a square item's chunk h in 128-row window win, R bits each
template <int SQ, int kCh, bool kSplit>
__device__ __forceinline__ uint64_t d_blocks(const DWalk<SQ, kCh, kSplit>& W, int h, int win, int lane) {
  constexpr int kB = SQ > 0 ? kDBoxK / SQ : 1, kR = SQ > 0 ? kDHalf / SQ : 1;
  uint64_t v = 0;
  const int c = (W.c0 + lane) * kCh + h;
  if (W.has(lane) && c < W.L->G && win < W.L->nw) {
    const uint8_t* km = static_cast<const uint8_t*>(W.L->kmask) + (int64_t)c * kB * W.L->nw + win;
#pragma unroll
    for (int b = 0; b < kB; ++b) v |= (uint64_t)km[(int64_t)b * W.L->nw] << (b * kR);
  }
  return v;
}
// items of the batch that have MMAs (square groups: every item)
template <int SQ, int kCh, bool kSplit>
__device__ __forceinline__ uint32_t d_batch(const DWalk<SQ, kCh, kSplit>& W, const DRows<kCh>& r, int lane) {
  if constexpr (SQ > 0) return __ballot_sync(0xffffffffu, W.has(lane));
  bool ne = false;
#pragma unroll
  for (int h = 0; h < kCh; ++h) ne |= r.c[h] > r.a[h];
  return __ballot_sync(0xffffffffu, ne);
}

// The last part of a 32-row block to arrive adds them all, in split order, and
// writes y (part: this lane's row of split 0).
__device__ __forceinline__ void d_reduce_parts(const DLayer& L, const float4* part, int row0, int lane, int T) {
  if (lane == 0) L.cnt[row0 / 32] = 0;
  uint16_t* yp = L.y + row0 + lane;
  const bool in_row = row0 + lane < L.out;
#pragma unroll 1
  for (int c0 = 0; 4 * c0 < T; c0 += 2) {   // eight tokens, four splits' loads in flight
    float4 acc[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
#pragma unroll 1
    for (int s0 = 0; s0 < L.n_split; s0 += 4) {
      float4 f[4][2];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int c = 0; c < 2; ++c)
          if (s0 + j < L.n_split && 4 * (c0 + c) < T) f[j][c] = __ldcg(part + (s0 + j) * 128 + c0 + c);
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int c = 0; c < 2; ++c)
          if (s0 + j < L.n_split && 4 * (c0 + c) < T) {
            acc[c].x += f[j][c].x;
            acc[c].y += f[j][c].y;
            acc[c].z += f[j][c].z;
            acc[c].w += f[j][c].w;
          }
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float a[4] = {acc[c].x, acc[c].y, acc[c].z, acc[c].w};
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (in_row && 4 * (c0 + c) + t < T)
          yp[(int64_t)(4 * (c0 + c) + t) * L.out] = __bfloat16_as_ushort(__float2bfloat16_rn(a[t]));
    }
  }
}

// KW: chunk width (1 x KW groups; square groups: 128); SQ: 0, or g for square
// g x g groups; SK: k per stage; kSplit: layers may have several parts per window
template <int KW, int SQ, int SK, bool kSplit>
__global__ void __launch_bounds__(kDThreads, 1) k_prefill_dense(const __grid_constant__ DParams P) {
  constexpr int kCh = KW < SK ? SK / KW : 1;              // chunks per item
  constexpr int kItemK = KW * kCh;                        // columns per item
  constexpr int kStPer = kItemK / SK;                     // stages per item
  constexpr int kBoxes = SK / kDBoxK;                     // copies of x (1 x KW: of W) per stage
  constexpr int kRowK = SQ > 0 ? (SQ < 64 ? SQ : 64) : 64;   // columns of one kept-row piece in shared memory
  constexpr int kSub = 64 / kRowK;                        // row pieces per 64-wide slab
  constexpr int kPieces = kRowK / 8;                      // 16-byte pieces per row piece
  constexpr int kBlk = 2 * kSub;                          // row pieces (square: column blocks) per 128 k
  constexpr int kR = SQ > 0 ? kDHalf / SQ : 1;            // square: block rows per half window
  static_assert(SK % kDBoxK == 0 && kItemK % SK == 0 && (kCh == 1 || KW == kDBoxK), "whole stages, a box a chunk");
  extern __shared__ uint8_t d_smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kDMaxXSlots];  // leader: both CTAs' converters + both CTAs' x bytes
  __shared__ __align__(8) uint64_t done_bar[kDMaxXSlots];  // the stage's MMAs completed (both CTAs)
  __shared__ __align__(8) uint64_t wfull_bar[kDWSeq];      // local: W bytes landed
  __shared__ __align__(8) uint64_t wempty_bar[kDWSeq];     // local: the converters have read them
  __shared__ uint32_t w_end[kDWSeq];                       // virtual end of each W stage in the ring (W copy warp)
  constexpr int kStarts = SQ > 0 ? kBlk : 1;
  __shared__ int32_t w_start[32][kCh][kStarts];            // the batch's items: first packed row (square: tile) ...
  __shared__ __align__(8) uint64_t w_n[32][kCh];           // ... and kept rows (square: kept block rows, d_blocks)
  __shared__ __align__(8) uint64_t afull_bar[2];          // D complete (both CTAs)
  __shared__ __align__(8) uint64_t aempty_bar[2];         // leader: D read by both CTAs' epilogues
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(d_smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();   // 0: leader (issues the pair's MMAs)

  if (threadIdx.x == 0) {
    for (int s = 0; s < kDMaxXSlots; ++s) {
      mbar_init(&full_bar[s], 2 * 4 + 1);
      mbar_init(&done_bar[s], 1);
    }
    for (int s = 0; s < kDWSeq; ++s) {
      mbar_init(&wfull_bar[s], 1);
      mbar_init(&wempty_bar[s], 4);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&afull_bar[b], 1);
      mbar_init(&aempty_bar[b], 2 * kDEpiWarps);
    }
    mbar_init(&drain_bar, 1);
    abort_s = 0;
    fence_mbar_init();
  }
  if (warp == kDMmaWarp) {
    tmem_alloc_pair(&tmem_base_s, kDTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  // Programmatic dependent launch: a launch that follows may take over SMs as
  // they fall free; this one copies weights (which only packing writes) at once
  // and waits for the one before it where x is read and y written.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t tmem = tmem_base_s;
  volatile int* abort_flag = &abort_s;
  const int n_tiles = P.n_tiles;
  const int pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
  const int Nh = P.N / 2;                          // tokens of a tile each CTA loads
  const uint32_t xs_n = (uint32_t)d_x_slots(P.N, SK);  // x slots; full / done barriers in use
  const uint32_t xs_bytes = (uint32_t)Nh * (SK * 2);
  const uint32_t w_ring = (uint32_t)d_w_ring(P.N, SK);   // bytes of the W ring
  uint8_t* wsmem = smem + xs_n * xs_bytes;
  const uint32_t n_buf = P.N <= kDN / 4 ? 2u : 1u; // D buffers
  const uint32_t t_a = d_d_cols(P.N);              // first column of the A slots
  const uint32_t a_n = d_a_slots(P.N, SK);

  if (P.inject_ns != 0 && pair == 0) {
    // test hook: before any copy or MMA is issued, a bounded wait on a word
    // that nothing sets runs out in each CTA of pair 0; the pair then records
    // the timeout and skips its units (every role, both CTAs)
    if (threadIdx.x == 0) {
      const volatile int* never = P.err + 1;
      const uint64_t t0 = globaltimer_ns();
      while (*never == 0) {
        if (globaltimer_ns() - t0 > P.inject_ns) {
          atomicExch(P.err, kDevErrTimeout);
          abort_s = 1;
          break;
        }
        __nanosleep(1000);
      }
    }
    __syncthreads();
  }
  const bool injected_abort = pair == 0 && abort_s != 0;

  if (injected_abort) {
    // nothing was issued: go straight to the TMEM release
  } else if (warp == 0) {
    // ------------------------------------------------------------ x copies
    // Stage k's box goes to slot k % xs_n once stage k - xs_n is done, and
    // completes on the leader's full barrier.
    uint32_t s = 0, ph = 1u;
    bool ok = true;
    asm volatile("griddepcontrol.wait;" ::: "memory");   // x may be the previous launch's output
    DWalk<SQ, kCh, kSplit> W(P, pair, n_pairs);
    DRows<kCh> nx = {};
    if constexpr (SQ == 0) nx = d_rows(W, lane);
    while (ok && W.valid()) {
      const DLayer& L = *W.L;
      const int tok0 = W.m * P.N + (int)rank * Nh, c0 = W.c0;
      uint32_t items = d_batch(W, nx, lane);
      W.next();
      if constexpr (SQ == 0) nx = d_rows(W, lane);
      for (; items && ok; items &= items - 1) {
        const int c = c0 + __ffs(items) - 1;
        for (int st = 0; st < kStPer; ++st) {
          if (!d_wait_warp(&done_bar[s], ph, abort_flag, P.err)) {
            ok = false;
            break;
          }
          if (elect_one()) {
            if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], 2u * xs_bytes);
#pragma unroll
            for (int b = 0; b < kBoxes; ++b)
              tma_load_3d_pair(smem + s * xs_bytes + b * (xs_bytes / kBoxes), &L.xmap,
                               mapa_shared(smem_u32(&full_bar[s]), 0), 0, tok0, c * (kItemK / 64) + 2 * (st * kBoxes + b));
          }
          __syncwarp();
          if (++s == xs_n) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ W copies
    // 1 x KW: the half window's kept rows of a chunk are one contiguous slice of
    // the packed tiles; one box a stage (two slabs), rows rounded up to 16.
    // Square: the half window's kept tiles of a column block are one contiguous
    // run; lane b copies block b's, back to back.
    uint32_t k = 0, oldest = 0;                   // stages issued / known to be read
    uint32_t head = 0, tail = 0, hoff = 0;        // virtual bytes allocated / released, head's ring offset
    bool ok = true;
    // The whole warp walks the stages (the lookups of a batch reach every lane
    // through shared memory) and one elected lane issues, as in the MMA warp.
    auto slot = [&](uint32_t bytes, uint32_t& off) {   // room for a stage: its offset in the ring
      const uint32_t e = k % kDWSeq;
      off = hoff;
      uint32_t pad = 0u;
      if (off + bytes > w_ring) {
        pad = w_ring - hoff;
        off = 0u;
      }
      const uint32_t end = head + pad + bytes;
      while (end - tail > w_ring || k - oldest >= (uint32_t)kDWSeq) {
        const uint32_t j = oldest % kDWSeq;
        if (!d_wait_warp(&wempty_bar[j], (oldest / kDWSeq) & 1u, abort_flag, P.err)) return false;
        tail = w_end[j];
        ++oldest;
      }
      __syncwarp();
      if (elect_one()) {
        w_end[e] = end;
        mbar_arrive_expect_tx(&wfull_bar[e], bytes);
      }
      __syncwarp();
      head = end;
      hoff = off + bytes;
      ++k;
      return true;
    };
    DWalk<SQ, kCh, kSplit> W(P, pair, n_pairs);
    if constexpr (SQ > 0) {
      uint64_t mk_n[kCh];
      int st_n[kCh][kBlk];
      auto load = [&]() {
        const int win = 2 * W.w + (int)rank;
#pragma unroll
        for (int h = 0; h < kCh; ++h) {
          mk_n[h] = d_blocks(W, h, win, lane);
          const int c = (W.c0 + lane) * kCh + h;
          const bool in = W.has(lane) && c < W.L->G && win < W.L->nw;
#pragma unroll
          for (int b = 0; b < kBlk; ++b)
            st_n[h][b] = in ? W.L->win_off[(int64_t)(c * kBlk + b) * (W.L->nw + 1) + win] : 0;
        }
      };
      load();
      while (ok && W.valid()) {
        const DLayer& L = *W.L;
        const int n_it = min(32, W.c1 - W.c0);
#pragma unroll
        for (int h = 0; h < kCh; ++h) {
          w_n[lane][h] = mk_n[h];
#pragma unroll
          for (int b = 0; b < kBlk; ++b) w_start[lane][h][b] = st_n[h][b];
        }
        W.next();
        load();
        __syncwarp();
        const uint16_t* tiles = L.tiles;
        for (int i = 0; i < n_it && ok; ++i) {
          uint32_t off, n_all = 0;
#pragma unroll
          for (int h = 0; h < kCh; ++h) n_all += (uint32_t)__popcll(w_n[i][h]);
          ok = slot(n_all * (SQ * SQ * 2), off);
          if (ok && elect_one()) {
            uint8_t* dst = wsmem + off;
            uint64_t* bar = &wfull_bar[(k - 1) % kDWSeq];
#pragma unroll
            for (int h = 0; h < kCh; ++h) {
              const uint64_t v = w_n[i][h];
#pragma unroll
              for (int b = 0; b < kBlk; ++b) {
                const int n = __popc((uint32_t)(v >> (b * kR)) & ((1u << kR) - 1u));
                if (n > 0) {
                  const int start = w_start[i][h][b];
                  if constexpr (SQ < 64)
                    bulk_g2s(dst, tiles + (int64_t)start * (SQ * SQ), (uint32_t)n * (SQ * SQ * 2), bar);
                  else
                    tma_load_2d(dst, &L.wmap[n - 1], bar, 0, start * SQ);
                  dst += n * (SQ * SQ * 2);
                }
              }
            }
          }
          __syncwarp();
        }
        __syncwarp();   // every lane has read the batch
      }
    } else {
      DRows<kCh> nx = d_rows(W, lane);
      while (ok && W.valid()) {
        const DLayer& L = *W.L;
        uint32_t items = d_batch(W, nx, lane);
#pragma unroll
        for (int h = 0; h < kCh; ++h) {
          const int start_l = rank ? nx.b[h] : nx.a[h];
          w_start[lane][h][0] = start_l;
          w_n[lane][h] = (uint64_t)((rank ? nx.c[h] : nx.b[h]) - start_l);
        }
        W.next();
        nx = d_rows(W, lane);
        __syncwarp();
        for (; items && ok; items &= items - 1) {
          const int i = __ffs(items) - 1;
          uint32_t h16 = 0;   // 16-row steps of the item's chunks
#pragma unroll
          for (int h = 0; h < kCh; ++h) h16 += ((uint32_t)w_n[i][h] + 15) / 16;
          for (int st = 0; st < kStPer && ok; ++st) {
            uint32_t off;
            ok = slot(h16 * (16u * (SK / kCh) * 2), off);
            if (ok && elect_one()) {
              uint8_t* dst = wsmem + off;
              uint64_t* bar = &wfull_bar[(k - 1) % kDWSeq];
#pragma unroll
              for (int b = 0; b < kBoxes; ++b) {
                const int h = kCh > 1 ? b : 0;
                const int hb = ((int)w_n[i][h] + 15) / 16;
                if (hb > 0) {
                  tma_load_3d(dst, &L.wmap[hb - 1], bar, 0, w_start[i][h][0], kCh > 1 ? 0 : 2 * (st * kBoxes + b));
                  dst += hb * (16 * kDBoxK * 2);
                }
              }
            }
            __syncwarp();
          }
        }
        __syncwarp();   // every lane has read the batch
      }
    }
    if (!ok && lane == 0) {
      // let the W copies in flight land before the CTA winds down
      for (uint32_t b = 0; b < (uint32_t)kDWSeq && b < k; ++b) {
        const uint32_t kb = k - 1 - b;
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(&wfull_bar[kb % kDWSeq], (kb / kDWSeq) & 1u))
          if (globaltimer_ns() - t0 > kDDrainLimitNs) break;
      }
    }
    __syncwarp();
  } else if (warp == kDMmaWarp && rank == 0) {
    // ------------------------------------------------------------ MMA issuer (leader)
    uint32_t kb = 0, s = 0, ph = 0u, as = 0;
    bool ok = true;
    const uint32_t idesc = idesc_bf16_f32(kDW, 0) | ((uint32_t)(P.N >> 3) << 17);
    // x operand descriptors: 16-byte units from x slot 0, a slab, a K step
    const uint64_t xd = sdesc_sw128(smem_u32(smem));
    const uint32_t x_lo = (uint32_t)xd, x_hi = (uint32_t)(xd >> 32), slab = (uint32_t)Nh * 8u;
    int part = 0;   // items of the next unit, counted while this one runs
    auto count = [&](int u) {
      if (u < 0) return 0;
      const DLayer& L = P.L[d_layer_of(P, u)];
      return d_count_part<SQ, kCh>(L, d_unit<kCh, kSplit>(L, u), lane);
    };
    int u = owner_tile(P.tl, n_tiles, pair, n_pairs, 0);
    part = count(u);
    for (int ku = 0; ok && u >= 0; ++ku, ++kb) {
      const int n_st = (int)__reduce_add_sync(0xffffffffu, (uint32_t)part) * kStPer;
      u = owner_tile(P.tl, n_tiles, pair, n_pairs, ku + 1);
      part = count(u);
      // The whole warp walks the stages, so that every operand is warp-uniform, and
      // one elected lane issues: from inside a one-lane branch each MMA cost 70
      // cycles of issue, eight of them more than a stage's tensor work.
      const uint32_t buf = kb % n_buf;
      ok = __all_sync(0xffffffffu, d_wait_cluster(&aempty_bar[buf], ((kb / n_buf) & 1u) ^ 1u, abort_flag, P.err));
      tc_fence_after();
      const uint32_t d = tmem + buf * (kDN / 4);
      for (int i = 0; i < n_st && ok; ++i) {
        if (!__all_sync(0xffffffffu, d_wait_cluster(&full_bar[s], ph, abort_flag, P.err))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t a = tmem + t_a + as * (SK / 2);
        const uint32_t b = x_lo + s * (xs_bytes >> 4);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < SK / 16; ++kk)
            mma_bf16_ts_pair(d, a + 8 * kk, ((uint64_t)x_hi << 32) | (b + (uint32_t)(kk >> 2) * slab + 2 * (kk & 3)), idesc,
                             (i == 0 && kk == 0) ? 0u : 1u);
          mma_commit_pair_mc(&done_bar[s], 0x3);
        }
        __syncwarp();
        if (++as == a_n) as = 0;
        if (++s == xs_n) {
          s = 0;
          ph ^= 1u;
        }
      }
      if (ok && elect_one()) mma_commit_pair_mc(&afull_bar[buf], 0x3);
      __syncwarp();
    }
    if (elect_one()) {
      mma_commit_pair(&drain_bar);
      mbar_wait_bounded(&drain_bar, 0u, nullptr, P.err, kDWaitLimitNs, kDevErrTimeout);
    }
    __syncwarp();
  } else if (warp >= kDConvWarp0 && warp < kDEpiWarp0) {
    // ------------------------------------------------------------ converters
    // Lane l of quarter q owns window row 128 rank + 32 q + l; the sets of four
    // warps take the stages in turn.
    const int q = warp & 3;
    const uint32_t set = (uint32_t)(warp - kDConvWarp0) >> 2;
    const int r = 32 * q + lane;   // row within this CTA's half
    const uint32_t lane_addr = tmem + ((uint32_t)(32 * q) << 16) + t_a;
    const uint32_t leader_full = mapa_shared(smem_u32(full_bar), 0);
    uint32_t k = 0, hoff = 0;                  // stage, its ring offset
    uint32_t s = 0;                            // its full barrier
    uint32_t ds = xs_n - a_n, dph = 1u;        // done barrier of the stage a_n earlier (the A slot's last user)
    if (xs_n == a_n) ds = 0;
    uint32_t as = 0;                           // its A slot
    bool ok = true;
    // one stage of `bytes` in the ring; piece(h, b, row, off): this lane's row in the
    // compact block of row piece b of 128-wide part h (-1: pruned), and the block's
    // offset from the stage's start
    auto stage = [&](auto&& piece, uint32_t bytes) {
      if (hoff + bytes > w_ring) hoff = 0;
      if (k % kDConvSets == set) {
        const uint32_t e = k % kDWSeq;
        if (!d_wait_warp(&wfull_bar[e], (k / kDWSeq) & 1u, abort_flag, P.err)) return false;
        const uint32_t at = lane_addr + as * (SK / 2);
#pragma unroll
        for (int h = 0; h < kBoxes; ++h) {
          uint32_t v[2][32];
          const uint32_t base = smem_u32(wsmem) + hoff;
#pragma unroll
          for (int b = 0; b < kBlk; ++b) {
            int row;
            uint32_t off;
            piece(h, b, row, off);
            const uint32_t ro = (uint32_t)row * (kRowK * 2);
            // 16-byte piece j of a row is read from (64-wide rows, which TMA swizzled)
            // or at (plain rows) piece j ^ swz, which spreads eight rows over the banks
            const uint32_t swz = (ro >> 7) & (uint32_t)(kPieces - 1);
            const uint32_t a = base + off + ro;
            uint4 p[kPieces];
#pragma unroll
            for (int j = 0; j < kPieces; ++j) {
              p[j] = make_uint4(0u, 0u, 0u, 0u);
              if (row >= 0) p[j] = lds128(a + (((uint32_t)j ^ swz) << 4));
            }
            if constexpr (kRowK < 64) {
              // plain rows: piece j now lies in p[j ^ swz]
#pragma unroll
              for (int d = 1; d < kPieces; d *= 2)
#pragma unroll
                for (int j = 0; j < kPieces; ++j)
                  if ((j & d) == 0) {
                    const bool sw = (swz & (uint32_t)d) != 0;
                    const uint4 x = p[j], y = p[j + d];
                    p[j] = sw ? y : x;
                    p[j + d] = sw ? x : y;
                  }
            }
#pragma unroll
            for (int j = 0; j < kPieces; ++j) {
              uint32_t* o = &v[b / kSub][4 * (b % kSub * kPieces + j)];
              o[0] = p[j].x;
              o[1] = p[j].y;
              o[2] = p[j].z;
              o[3] = p[j].w;
            }
          }
          __syncwarp();
          if (h == kBoxes - 1 && lane == 0) mbar_arrive(&wempty_bar[e]);
          if (h == 0) {
            if (k >= a_n && !d_wait_warp(&done_bar[ds], dph, abort_flag, P.err)) return false;
            tc_fence_after();
          }
          tmem_st_x32(at + 64 * h, v[0]);
          tmem_st_x32(at + 64 * h + 32, v[1]);
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster_relaxed(leader_full + 8u * s);
      }
      hoff += bytes;
      if (++ds == xs_n) {
        ds = 0;
        dph ^= 1u;
      }
      if (++s == xs_n) s = 0;
      if (++as == a_n) as = 0;
      ++k;
      return true;
    };
    DWalk<SQ, kCh, kSplit> W(P, pair, n_pairs);
    if constexpr (SQ > 0) {
      const int br = r / SQ;
      uint64_t mk_n[kCh];
      auto load = [&]() {
#pragma unroll
        for (int h = 0; h < kCh; ++h) mk_n[h] = d_blocks(W, h, 2 * W.w + (int)rank, lane);
      };
      load();
      while (ok && W.valid()) {
        uint64_t mk[kCh];
#pragma unroll
        for (int h = 0; h < kCh; ++h) mk[h] = mk_n[h];
        const int n_it = min(32, W.c1 - W.c0);
        W.next();
        load();
        for (int i = 0; i < n_it && ok; ++i) {
          uint64_t v[kCh];
          uint32_t n_all = 0;
#pragma unroll
          for (int h = 0; h < kCh; ++h) {
            v[h] = __shfl_sync(0xffffffffu, mk[h], i);
            n_all += (uint32_t)__popcll(v[h]);
          }
          ok = stage([&](int h, int b, int& row, uint32_t& off) {
            const int at = b * kR;   // this block's bits
            const uint32_t mb = (uint32_t)(v[h] >> at) & ((1u << kR) - 1u);
            row = ((mb >> br) & 1u) ? (int)__popc(mb & ((1u << br) - 1u)) * SQ + r % SQ : -1;
            off = (uint32_t)__popcll(v[h] & ((1ull << at) - 1ull));
            for (int o = 0; o < h; ++o) off += (uint32_t)__popcll(v[o]);
            off *= SQ * SQ * 2;
          }, n_all * (SQ * SQ * 2));
        }
      }
    } else {
      // this warp's two 16-row windows in an item: kept masks, first packed row
      uint32_t mk_n[kCh];
      int wo_n[kCh];
      auto load = [&]() {
#pragma unroll
        for (int h = 0; h < kCh; ++h) {
          mk_n[h] = 0;
          wo_n[h] = 0;
          const int c = (W.c0 + lane) * kCh + h;
          if (!W.has(lane) || c >= W.L->G) continue;
          const int nw = W.L->nw, b16 = W.w * (kDW / kWin16) + (int)rank * (kDHalf / kWin16) + 2 * q;
          const uint16_t* km = static_cast<const uint16_t*>(W.L->kmask) + (int64_t)c * nw;
          if (b16 < nw) {
            mk_n[h] = km[b16];
            wo_n[h] = W.L->win_off[(int64_t)c * (nw + 1) + b16];
          }
          if (b16 + 1 < nw) mk_n[h] |= (uint32_t)km[b16 + 1] << 16;
        }
      };
      DRows<kCh> nx = d_rows(W, lane);
      load();
      while (ok && W.valid()) {
        uint32_t items = d_batch(W, nx, lane);
        uint32_t mk_l[kCh];
        int at_l[kCh];   // kept rows of the half window before this warp's rows | all of them << 16
#pragma unroll
        for (int h = 0; h < kCh; ++h) {
          const int start_l = rank ? nx.b[h] : nx.a[h];
          mk_l[h] = mk_n[h];
          at_l[h] = ((wo_n[h] - start_l) & 0xffff) | (((rank ? nx.c[h] : nx.b[h]) - start_l) << 16);
        }
        W.next();
        nx = d_rows(W, lane);
        load();
        for (; items && ok; items &= items - 1) {
          const int i = __ffs(items) - 1;
          // rows 32 q .. + 31 of the half window are consecutive bits, and consecutive in the slice
          int row_c[kCh];
          uint32_t slab[kCh], bytes = 0;
#pragma unroll
          for (int h = 0; h < kCh; ++h) {
            const uint32_t mk = __shfl_sync(0xffffffffu, mk_l[h], i);
            const int at = __shfl_sync(0xffffffffu, at_l[h], i);
            row_c[h] = ((mk >> lane) & 1u) ? (at & 0xffff) + (int)__popc(mk & ((1u << lane) - 1u)) : -1;
            slab[h] = (uint32_t)(((at >> 16) + 15) / 16) * (16 * 128);
            bytes += slab[h] * (SK / kCh / 64);
          }
#pragma unroll
          for (int st = 0; st < kStPer; ++st)
            if (ok)
              ok = stage([&](int h, int b, int& row, uint32_t& off) {
                const int ch = kCh > 1 ? h : 0;
                row = row_c[ch];
                off = (uint32_t)b * slab[ch];
                for (int o = 0; o < h; ++o) off += 2 * slab[kCh > 1 ? o : 0];
              }, bytes);
        }
      }
    }
  } else if (warp >= kDEpiWarp0) {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3, hh = (warp - kDEpiWarp0) >> 2;   // TMEM lane quarter, half of the tile's tokens
    const int nl = (Nh + 15) / 16;                           // 16-token loads per warp (the last may hold 8 of its own)
    asm volatile("griddepcontrol.wait;" ::: "memory");       // the previous launch may still use y
    uint32_t kb = 0;
    bool ok = true;
    const uint32_t leader_empty = mapa_shared(smem_u32(aempty_bar), 0);
    int part_n = 0;   // items of the next unit, counted while this one runs
    auto count = [&](int v) {
      if (v < 0) return 0;
      const DLayer& L = P.L[d_layer_of(P, v)];
      return d_count_part<SQ, kCh>(L, d_unit<kCh, kSplit>(L, v), lane);
    };
    int u_n = owner_tile(P.tl, n_tiles, pair, n_pairs, 0);
    part_n = count(u_n);
    for (int ku = 0; ok && u_n >= 0; ++ku, ++kb) {
      const int u = u_n;
      const DLayer& L = P.L[d_layer_of(P, u)];
      const DUnit U = d_unit<kCh, kSplit>(L, u);
      const int m = U.m, w = U.w;
      const bool any = __any_sync(0xffffffffu, part_n > 0);   // else no MMA wrote D: zeros
      u_n = owner_tile(P.tl, n_tiles, pair, n_pairs, ku + 1);
      part_n = count(u_n);
      const uint32_t buf = kb % n_buf;
      if (!d_wait_warp(&afull_bar[buf], (kb / n_buf) & 1u, abort_flag, P.err)) {
        ok = false;
        break;
      }
      tc_fence_after();
      if (kSplit && L.n_split > 1) {
        // T <= 16: the first half of the warps holds every token of the tile
        uint32_t v[16];
        if (hh == 0) {
          tmem_ld_x16(tmem + ((uint32_t)(32 * q) << 16) + buf * (kDN / 4), v);
          tmem_wait_ld();
          reg_fence(v);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster_relaxed(leader_empty + 8u * buf);   // D may be overwritten
        const int row0 = w * kDW + (int)rank * kDHalf + 32 * q;
        if (hh == 0 && row0 < L.out) {
          // a lane's row: 16 tokens, 64 bytes
          float4* part = reinterpret_cast<float4*>(L.ws + (int64_t)(row0 / 32) * L.n_split * 512) + 4 * lane;   // split 0
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (4 * c < P.T) {
              const float* f = reinterpret_cast<const float*>(v + 4 * c);
              part[U.sp * 128 + c] = any ? make_float4(f[0], f[1], f[2], f[3]) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
          __syncwarp();
          int old = 0;
          if (lane == 0) old = d_atom_add_acq_rel(&L.cnt[row0 / 32], 1);
          if (__shfl_sync(0xffffffffu, old, 0) == L.n_split - 1) {
            __syncwarp();
            d_reduce_parts(L, part, row0, lane, P.T);
          }
        }
        __syncwarp();
        continue;
      }
      constexpr int kNL = kSplit ? 1 : kDN / 32;   // most 16-token loads (T <= 16: one)
      uint32_t pk[8 * kNL];   // this lane's row: pairs of tokens
      const uint32_t dcol = tmem + ((uint32_t)(32 * q) << 16) + buf * (kDN / 4) + (uint32_t)(hh * Nh);
#pragma unroll
      for (int i = 0; i < kNL; ++i)
        if (i < nl) {
          uint32_t v[16];
          tmem_ld_x16(dcol + 16 * i, v);
          tmem_wait_ld();
          reg_fence(v);
#pragma unroll
          for (int e = 0; e < 8; ++e)
            pk[8 * i + e] = any ? d_pack_bf16x2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1])) : 0u;
        }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster_relaxed(leader_empty + 8u * buf);   // D may be overwritten
      const int row = w * kDW + (int)rank * kDHalf + 32 * q + lane;
      const int tok0 = m * P.N + hh * Nh;
      if ((L.out & 1) == 0) {
        // neighbouring lanes swap so that each holds one token of two rows: even
        // lanes the first token of every pair, odd lanes the second
        const uint32_t sel = (lane & 1) ? 0x3276u : 0x5410u;
        const bool in_row = (row & ~1) < L.out;
        uint16_t* yp = L.y + (int64_t)(tok0 + (lane & 1)) * L.out + (row & ~1);
#pragma unroll
        for (int i = 0; i < kNL; ++i)
          if (i < nl) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const int t = 16 * i + 2 * e;
              const uint32_t o = __shfl_xor_sync(0xffffffffu, pk[8 * i + e], 1);
              if (in_row && t < Nh && tok0 + t + (lane & 1) < P.T)
                *reinterpret_cast<uint32_t*>(yp + (int64_t)t * L.out) = __byte_perm(pk[8 * i + e], o, sel);
            }
          }
      } else if (row < L.out) {
        uint16_t* yp = L.y + (int64_t)tok0 * L.out + row;
#pragma unroll
        for (int i = 0; i < kNL; ++i)
          if (i < nl) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const int t = 16 * i + 2 * e;
              if (t < Nh && tok0 + t < P.T) yp[(int64_t)t * L.out] = (uint16_t)pk[8 * i + e];
              if (t < Nh && tok0 + t + 1 < P.T) yp[(int64_t)(t + 1) * L.out] = (uint16_t)(pk[8 * i + e] >> 16);
            }
          }
      }
      __syncwarp();
    }
  }

  tc_fence_before();
  __syncthreads();
  if (abort_s) {
    // a role gave up: give copies the peer may still have in flight time to land
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 2000000ull) {
    }
  }
  cluster_sync_all();
  if (warp == kDMmaWarp) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, kDTmemCols);
  }
  cluster_sync_all();
}

int d_sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 148;
  }
  return n;
}

template <int KW, int SQ, int SK, bool kSplit>
cudaError_t d_set_attr() {
  static std::once_flag once;
  static cudaError_t err = cudaSuccess;
  std::call_once(once, []() {
    err = cudaFuncSetAttribute(k_prefill_dense<KW, SQ, SK, kSplit>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDSmem);
  });
  return err;
}

template <int KW, int SQ, int SK, bool kSplit = false>
cudaError_t d_launch(const cudaLaunchConfig_t& cfg, const DParams& P) {
  const cudaError_t e = d_set_attr<KW, SQ, SK, kSplit>();
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, k_prefill_dense<KW, SQ, SK, kSplit>, P);
}

}  // namespace

// Parts per window of each layer of a launch of at most 16 tokens.  Whole windows
// alone can be too few or too long to fill 76 CTA pairs: a 5120 x 13824 layer (20
// windows of 54 items) took 35 us, 19 in three parts.  But a part costs what about
// six items do (partial sums out and in, an atomic): 13824 x 5120 took 17 us whole
// and 21 to 30 us in four parts, a 7B block 37 us whole and 43 us with its 43-item
// windows in parts of ten.
void d_plan_splits(const std::vector<int>& units, const std::vector<int>& items, const std::vector<int>& most,
                   int owners, std::vector<int>& split) {
  const int n = (int)units.size();
  int64_t total = 0;
  int longest = 0, n_units = 0;
  bool same = true;
  for (int i = 0; i < n; ++i) {
    total += (int64_t)units[i] * items[i];
    n_units += units[i];
    longest = std::max(longest, items[i]);
    same = same && items[i] == items[0];
  }
  split.assign(n, 1);
  const auto set = [&](int i, int s) { split[i] = std::max(1, std::min(s, std::min(most[i], items[i]))); };
  const int avg = (int)((total + owners - 1) / owners);
  if (same || n_units < owners) {
    // the parts per longest window that leave the least to the busiest pair
    int best = 1, best_cost = 1 << 30;
    for (int s = 1; s <= 16 && s <= longest; ++s) {
      int parts = 0, len = 0;
      for (int i = 0; i < n; ++i) {
        const int si = std::max(1, (s * items[i] + longest - 1) / longest);
        parts += units[i] * si;
        len = std::max(len, (items[i] + si - 1) / si);
      }
      const int cost = (parts + owners - 1) / owners * (len + (s > 1 ? 6 : 2));
      if (cost < best_cost) {
        best_cost = cost;
        best = s;
      }
    }
    for (int i = 0; i < n; ++i) set(i, (best * items[i] + longest - 1) / longest);
    return;
  }
  // several lengths: only where a long window by itself outlasts the mean pair
  // (Qwen2.5-7B block, 74 items against a mean of 47: 50 -> 44 us)
  if (10 * longest <= 13 * avg) return;
  const int len = std::max(8, avg / 2);
  for (int i = 0; i < n; ++i)
    if (2 * items[i] > avg) set(i, (items[i] + len - 1) / len);
}

// Tokens of each of n_m tiles of equal size: whole 16 tokens (swizzled 8-row groups of
// x in each CTA; T = 777 takes four of 208 where whole 32 would be 224), at least 32.
int64_t d_tile_tokens(int64_t T, int64_t n_m) { return std::max<int64_t>(32, ((T + n_m - 1) / n_m + 15) / 16 * 16); }

// Token tiles of a launch: as few as 256 tokens each allow, or more and narrower ones
// where those leave CTA pairs without a unit.  Estimated time: the busiest pair's
// 256-column items times what one takes at n tokens (measured, ns: about 540 + 1.6 n
// with 256-deep stages, up to 128 tokens; 4.4 n, at least 1000, above).  Narrower tiles
// change no result: a row's products are added in the same order.  From three units a
// pair on, or one with layers of several widths, the wide tiles stay (a Qwen2.5-7B block at
// T = 200 took 84 us in two tiles of 112 and 78 in one).  Layers alone, us as graph replays: 4096 x 4096 at T = 256
// 25 -> 16, 5120 x 13824 at T = 256 / 777 67 / 103 -> 42 / 80, 3000 x 12032 (1 x 128) at
// T = 512 59 -> 41, 4096 x 11008 (64x64) at T = 512 52 -> 38; 16x16 groups, whose stages
// are always 128 deep, 65 -> 66.
int64_t d_token_tiles(const std::vector<int64_t>& units, const std::vector<int64_t>& items, int64_t T, int64_t owners,
                      bool deep) {
  const int64_t least = (T + kDN - 1) / kDN;
  int64_t n_units = 0, total = 0, longest = 0;
  for (size_t i = 0; i < units.size(); ++i) {
    n_units += units[i];
    total += units[i] * items[i];
    longest = std::max(longest, items[i]);
  }
  const bool same = total == n_units * longest;
  if (!deep || T <= kDN / 2 || n_units * least >= (same ? 3 : 1) * owners) return least;
  int64_t best = least;
  double best_cost = 0.0;
  for (int64_t m = least; m <= 8 * least && (m == least || n_units * m <= 6 * owners); ++m) {
    const int64_t n = d_tile_tokens(T, m);
    const double item = n <= kDN / 2 ? 540.0 + 1.6 * (double)n : std::max(1000.0, 4.4 * (double)n);
    const int64_t rounds = (n_units * m + owners - 1) / owners;
    const int64_t busiest = same ? rounds * longest : std::max(longest * (rounds > 1 ? 2 : 1), (total * m + owners - 1) / owners);
    const double cost = (double)busiest * item;
    if (m == least || cost < 0.95 * best_cost) {
      best_cost = cost;
      best = m;
    }
  }
  return best;
}

// Which 1 x KW layers take this kernel: all that have kept groups, in the whole
// prefill regime.  Against the gathering kernel, d = 0.5, us per batched block:
// 13B 1 x 256 at T = 32 / 128 / 512 58 / 67 / 168 against 93 / 98 / 294.  One call per layer, over
// nine shapes from 1024 x 1024 to 20000 x 1024 and T = 17 to 640, it takes
// 0.4-0.97x the gathering kernel's time.
bool prefill_prefers_dense(const gs_packed* p) {
  return p->kept > 0 && p->g_out == 1 && (p->g_in == 128 || p->g_in == 256) && p->G <= kDMaxChunks;
}

// Whether a call of at most 16 tokens over layers of one chunk width takes this
// kernel (split) rather than the decode kernel.
bool decode_prefers_dense(const gs_packed* const* ps, int n, int64_t T) {
  if (T > 16) return false;
  std::vector<FewTokenLayer> layers;
  layers.reserve((size_t)n);
  for (int i = 0; i < n; ++i) {
    const gs_packed* p = ps[i];
    if (p->kept == 0) continue;
    if (!prefill_prefers_dense(p)) return false;
    layers.push_back({p->out, p->in, 2.0 * (double)p->kept * p->g_in, p->G, p->dec_cpu, p->dec_cpu_fine});
  }
  return !layers.empty() && zero_filled_first(layers, ps[0]->g_in, (int)T, d_sm_count());
}

gs_status launch_prefill_dense(const void* const* xs, const gs_packed* const* ps, int n, int64_t T, void* const* ys,
                               cudaStream_t s, const int* idx, bool split) {
  if (T <= 0 || n <= 0) return GS_OK;
  std::vector<int> order(n);
  for (int i = 0; i < n; ++i) order[i] = idx ? idx[i] : i;
  const int kw = ps[order[0]]->g_in, go = ps[order[0]]->g_out;
  for (int i : order)
    if (ps[i]->g_in != kw || ps[i]->g_out != go || ps[i]->kept == 0) return GS_ERR_UNSUPPORTED;
  const int sq = go > 1 ? go : 0;   // square g x g groups
  if (sq ? (sq != kw || (sq != 16 && sq != 32 && sq != 64)) : (kw != 256 && kw != 128)) return GS_ERR_UNSUPPORTED;
  for (int i : order)
    if (!sq && !ps[i]->wmaps_valid) return GS_ERR_UNSUPPORTED;
  int* err = device_error_flag();
  if (!err) return GS_ERR_CUDA;
  // most tensor work per unit (the widest input) first
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return ps[a]->in > ps[b]->in; });
  const int64_t max_pairs = d_sm_count() / 2;
  for (int b0 = 0; b0 < n; b0 += kDMaxLayers) {
    const int nb = std::min(kDMaxLayers, n - b0);
    DParams P;
    std::memset(&P, 0, sizeof(P));
    int64_t tiles = 0;
    int64_t n_m = (T + kDN - 1) / kDN;
    {
      std::vector<int64_t> units(nb), items(nb);
      for (int k = 0; k < nb; ++k) {
        units[k] = (ps[order[b0 + k]]->out + kDW - 1) / kDW;
        items[k] = (ps[order[b0 + k]]->in + 255) / 256;
      }
      n_m = d_token_tiles(units, items, T, max_pairs, sq != 16);
    }
    const int64_t tile_n = d_tile_tokens(T, n_m);
    const bool deep = tile_n <= kDN / 2 && sq != 16;   // 256-deep stages (16 x 16 groups: their lookups would not fit)
    const int item_k = sq == 0 && kw == 256 ? 256 : deep ? 256 : 128;
    std::vector<int> parts(nb, 1);
    if (split && T <= 16 && !sq) {
      std::vector<int> units(nb), items(nb), most(nb);
      for (int k = 0; k < nb; ++k) {
        const gs_packed* p = ps[order[b0 + k]];
        units[k] = (int)((p->out + kDW - 1) / kDW);
        items[k] = (int)((p->in + item_k - 1) / item_k);
        most[k] = p->dec_nsplit_max;
      }
      d_plan_splits(units, items, most, (int)max_pairs, parts);
    }
    for (int k = 0; k < nb; ++k) {
      const int i = order[b0 + k];
      const gs_packed* p = ps[i];
      DLayer& L = P.L[k];
      L.n_split = parts[k];
      if (L.n_split > 1) {
        // partial sums and counters in the decode path's per-stream scratch: 1024 floats per
        // 64-row block and split there too, and at least one counter per 32 rows
        const DecSlot* slot = nullptr;
        const gs_status st = decode_slot(p, s, &slot);
        if (st != GS_OK) return st;
        L.ws = slot->ws;
        L.cnt = slot->cnt;
      }
      if (!encode_tmap_slabs_bf16(&L.xmap, xs[i], (uint64_t)p->in, (uint64_t)T, (uint32_t)(tile_n / 2), 2))
        return GS_ERR_CUDA;
      L.tiles = p->tiles;
      L.y = static_cast<uint16_t*>(ys[i]);
      L.out = (int32_t)p->out;
      if (sq) {
        if (p->in % 128 != 0) return GS_ERR_UNSUPPORTED;
        for (int h = 0; h < kDHalf / sq; ++h) std::memcpy(&L.wmap[h], p->gmaps[h], sizeof(CUtensorMap));
        L.win_off = p->gwoff;
        L.kmask = p->gwmask;
        L.nw = p->nwin;
        L.G = (int32_t)(p->in / 128);   // 128-column items, one stage each
      } else {
        for (int h = 0; h < kDWMaps; ++h) std::memcpy(&L.wmap[h], p->wmaps_full[h], sizeof(CUtensorMap));
        L.win_off = p->win_off16;
        L.kmask = p->kmask16;
        L.nw = p->nw16;
        L.G = p->G;
      }
      if (L.G > kDMaxChunks) return GS_ERR_UNSUPPORTED;
      L.n_m = (int32_t)n_m;
      L.tile_begin = (int32_t)tiles;
      tiles += (int64_t)L.n_m * L.n_split * ((p->out + kDW - 1) / kDW);
    }
    if (tiles > INT32_MAX) return GS_ERR_UNSUPPORTED;
    P.n_layers = nb;
    P.T = (int32_t)T;
    P.N = (int32_t)tile_n;
    P.n_tiles = (int32_t)tiles;
    P.err = err;
    P.inject_ns = b0 == 0 ? take_injected_wait(split && T <= 16 ? GS_ALGO_DECODE : GS_ALGO_PREFILL_DENSE) : 0;
    const int owners = (int)std::min<int64_t>(tiles, max_pairs);
    if (tiles <= kTileListMax) {
      // A unit's time follows its item count (one launch holds one chunk width) and, at
      // 17 to 128 tokens, the kept rows each item brings (7B block at d = 0.3 / 0.5 / 0.7:
      // 40 / 49 / 66 us at T = 128): about 1/4 + density an item.  A 13B block of mixed
      // densities takes 73 -> 70 us so; at 16 tokens or fewer the same weights cost 2 to
      // 12 %, above 128 tokens (117 / 121 us at T = 512, d = 0.3 / 0.5) they change nothing.
      const bool by_kept = T > 16 && tile_n <= kDN / 2;
      std::vector<int32_t> cost((size_t)tiles);
      for (int k = 0; k < nb; ++k) {
        const int64_t nu = (int64_t)P.L[k].n_m * parts[k] * ((ps[order[b0 + k]]->out + kDW - 1) / kDW);
        const gs_packed* p = ps[order[b0 + k]];
        const double d = (double)p->kept * p->g_out * p->g_in / ((double)p->out * (double)p->in);
        const int32_t items = (P.L[k].G + parts[k] - 1) / parts[k];
        const int32_t c = by_kept ? (int32_t)(64.0 * items * (0.25 + d)) + 1 : items;
        for (int64_t t = 0; t < nu; ++t) cost[(size_t)(P.L[k].tile_begin + t)] = c;
      }
      plan_tiles(cost, owners, P.tl);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * owners));
    cfg.blockDim = dim3(kDThreads);
    cfg.dynamicSmemBytes = kDSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    bool overlap = true;
    for (int k = 0; k < nb; ++k) overlap &= may_overlap(ps[order[b0 + k]], s);
    cfg.numAttrs = overlap ? 2 : 1;
    bool any_split = false;
    for (int k = 0; k < nb; ++k) any_split |= parts[k] > 1;
    const cudaError_t e = any_split  ? (kw == 128 ? d_launch<128, 0, 256, true>(cfg, P) : d_launch<256, 0, 256, true>(cfg, P))
                          : sq == 16   ? d_launch<128, 16, 128>(cfg, P)
                          : sq == 32 ? (deep ? d_launch<128, 32, 256>(cfg, P) : d_launch<128, 32, 128>(cfg, P))
                          : sq == 64 ? (deep ? d_launch<128, 64, 256>(cfg, P) : d_launch<128, 64, 128>(cfg, P))
                          : kw == 128 ? (deep ? d_launch<128, 0, 256>(cfg, P) : d_launch<128, 0, 128>(cfg, P))
                                      : (deep ? d_launch<256, 0, 256>(cfg, P) : d_launch<256, 0, 128>(cfg, P));
    note_launch();
    if (e != cudaSuccess) return GS_ERR_CUDA;
    if (!overlap)
      for (int k = 0; k < nb; ++k) launch_queued(ps[order[b0 + k]], s);
  }
  return GS_OK;
}

}  // namespace gs
