// Logit gradient of the straight-through estimator for 1 x KW groups, in one
// pass: dL/dl[r, v] = ds/dl[r, v] * sum_k W[r, k] D[r, k] over the group's KW
// columns k, with D = dy^T x (fp32), for every group, pruned ones included.
//
// D is never written: a unit of work is 256 output rows x 256 input columns, owned
// by a cluster of two CTAs, whose D stays in TMEM (lane = output row), and a
// group is a stretch of one lane's columns.  The epilogue reads D and W side by
// side and keeps one number a group.
//
// Both operands are stored with the contracted dimension (tokens) outermost, so
// they go to the tensor cores MN-major: a TMA box is 64 tokens x 128 rows (or
// columns) as two 64-wide 128-byte-swizzled slabs.  cta_group::2 MMAs, M = N = 256;
// CTA r holds rows and columns 128 r .. of the tile.
//
// Bound by the tensor cores: 2 T out in FLOP, the dense product for every group.  An
// 11008 x 4096 layer at T = 2048: 103 us (1.80 PFLOP/s), where a library GEMM that wrote D
// (108 us) and a pass that read it back with W (52 us) took 160.  688 units over 76 pairs
// leave a tenth of the last round empty.
//
// Roles (one CTA per SM, units at a fixed stride over the pairs): warp 0 copies,
// warp 1 TMEM allocator + MMA issuer (leader), warps 4..11 epilogue (two sets of
// four warps, lane quarter warp & 3, take the units and D buffers in turn).
// Every wait is bounded.
#include "gs_common.cuh"
#include "gs_sm100.cuh"

#include <cuda.h>
#include <algorithm>
#include <mutex>

namespace gs {
namespace {
using namespace sm100;

constexpr int kGM = 256, kGN = 256;              // unit: output rows x input columns
constexpr int kGK = 64;                          // tokens per stage
constexpr int kGOpBytes = 128 * kGK * 2;         // one CTA's half of an operand: 16 KB
constexpr int kGStageBytes = 2 * kGOpBytes;
constexpr int kGStages = 7;
constexpr int kGEpiWarp0 = 4, kGEpiWarps = 8;
constexpr int kGThreads = (kGEpiWarp0 + kGEpiWarps) * 32;
constexpr uint32_t kGTmemCols = 512;             // two D buffers
constexpr int kGSmem = kGStages * kGStageBytes + 1024;
constexpr uint64_t kGWaitLimitNs = 2000000000ull;
static_assert(kGSmem <= 227 * 1024 - 1024, "shared memory budget");

struct GParams {
  CUtensorMap amap, bmap;   // dy (out) and x (in) as (64, T, width / 64) slabs, box 64 x 64 x 2
  const uint16_t* W;        // [out][in]
  const float* dsdl;        // [out][in / kw]
  float* dlogits;
  int32_t out, in, n_k, n_n, n_units;
  int* err;
};

// Shared-memory descriptor of an MN-major operand, 128-byte swizzle: 64-element
// blocks [kGK tokens][128 B]; 8-token groups 1024 bytes apart, blocks kGK * 128
__device__ __forceinline__ uint64_t sdesc_mn_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((kGK * 128) >> 4) << 16;   // leading: next 64 elements along M or N
  d |= (uint64_t)(1024 >> 4) << 32;          // stride: next 8 tokens
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

template <int KW>
__global__ void __launch_bounds__(kGThreads, 1) k_group_grad_mma(const __grid_constant__ GParams P) {
  extern __shared__ uint8_t g_smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kGStages];   // leader: both CTAs' bytes
  __shared__ __align__(8) uint64_t done_bar[kGStages];   // the stage's MMAs completed (both CTAs)
  __shared__ __align__(8) uint64_t afull_bar[2];
  __shared__ __align__(8) uint64_t aempty_bar[2];
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(g_smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  if (threadIdx.x == 0) {
    for (int s = 0; s < kGStages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&done_bar[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&afull_bar[b], 1);
      mbar_init(&aempty_bar[b], 2 * 4);
    }
    mbar_init(&drain_bar, 1);
    abort_s = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(&tmem_base_s, kGTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  volatile int* abort_flag = &abort_s;
  const int pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
  const auto wait_warp = [&](uint64_t* bar, uint32_t parity) {
    return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, abort_flag, P.err, kGWaitLimitNs, kDevErrTimeout)) != 0;
  };

  if (warp == 0) {
    // ------------------------------------------------------------ copies
    uint32_t s = 0, ph = 1u;
    bool ok = true;
    for (int u = pair; ok && u < P.n_units; u += n_pairs) {
      const int a_slab = (u / P.n_n) * (kGM / 64) + (int)rank * 2, b_slab = (u % P.n_n) * (kGN / 64) + (int)rank * 2;
      for (int k = 0; k < P.n_k; ++k) {
        if (!wait_warp(&done_bar[s], ph)) {
          ok = false;
          break;
        }
        if (elect_one()) {
          if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], 2u * kGStageBytes);
          const uint32_t fb = mapa_shared(smem_u32(&full_bar[s]), 0);
          tma_load_3d_pair(smem + s * kGStageBytes, &P.amap, fb, 0, k * kGK, a_slab);
          tma_load_3d_pair(smem + s * kGStageBytes + kGOpBytes, &P.bmap, fb, 0, k * kGK, b_slab);
        }
        __syncwarp();
        if (++s == kGStages) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
  } else if (warp == 1 && rank == 0) {
    // ------------------------------------------------------------ MMA issuer (leader)
    // bits 15 and 16: both operands MN-major
    const uint32_t idesc = idesc_bf16_f32(kGM, kGN) | (1u << 15) | (1u << 16);
    const uint64_t d0 = sdesc_mn_sw128(smem_u32(smem));
    uint32_t s = 0, ph = 0u, kb = 0;
    bool ok = true;
    for (int u = pair; ok && u < P.n_units; u += n_pairs, ++kb) {
      const uint32_t buf = kb & 1u;
      ok = __all_sync(0xffffffffu, mbar_wait_bounded_cluster(&aempty_bar[buf], ((kb >> 1) & 1u) ^ 1u, abort_flag, P.err,
                                                             kGWaitLimitNs, kDevErrTimeout));
      tc_fence_after();
      for (int k = 0; k < P.n_k && ok; ++k) {
        if (!__all_sync(0xffffffffu, mbar_wait_bounded_cluster(&full_bar[s], ph, abort_flag, P.err, kGWaitLimitNs,
                                                               kDevErrTimeout))) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (elect_one()) {
          const uint64_t a = d0 + (uint64_t)(s * (kGStageBytes >> 4)), b = a + (kGOpBytes >> 4);
#pragma unroll
          for (int kk = 0; kk < kGK / 16; ++kk)
            mma_bf16_ss_pair(tmem + buf * kGN, a + (uint64_t)(kk * (2048 >> 4)), b + (uint64_t)(kk * (2048 >> 4)), idesc,
                             (k == 0 && kk == 0) ? 0u : 1u);
          mma_commit_pair_mc(&done_bar[s], 0x3);
        }
        __syncwarp();
        if (++s == kGStages) {
          s = 0;
          ph ^= 1u;
        }
      }
      if (ok && elect_one()) mma_commit_pair_mc(&afull_bar[buf], 0x3);
      __syncwarp();
    }
    if (elect_one()) {
      mma_commit_pair(&drain_bar);
      mbar_wait_bounded(&drain_bar, 0u, nullptr, P.err, kGWaitLimitNs, kDevErrTimeout);
    }
    __syncwarp();
  } else if (warp >= kGEpiWarp0) {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3;
    const uint32_t set = (uint32_t)(warp - kGEpiWarp0) >> 2;   // units and D buffer this warp takes
    const uint32_t empty = mapa_shared(smem_u32(&aempty_bar[set]), 0);
    const int n_g = P.in / KW;
    uint32_t kb = 0;
    bool ok = true;
    for (int u = pair; ok && u < P.n_units; u += n_pairs, ++kb) {
      if ((kb & 1u) != set) continue;
      const int row = (u / P.n_n) * kGM + (int)rank * 128 + 32 * q + lane, col0 = (u % P.n_n) * kGN;
      const bool in_row = row < P.out;
      const uint4* w = reinterpret_cast<const uint4*>(P.W + (int64_t)(in_row ? row : 0) * P.in + col0);
      constexpr int kAhead = 4;   // 16-column pieces of W in flight
      uint4 wv[kAhead][2];
      auto load = [&](int j, uint4 (&v)[2]) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
          v[h] = in_row && col0 + 16 * j < P.in ? __ldg(w + 2 * j + h) : make_uint4(0u, 0u, 0u, 0u);
      };
#pragma unroll
      for (int j = 0; j < kAhead; ++j) load(j, wv[j]);
      if (!wait_warp(&afull_bar[set], (kb >> 1) & 1u)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t d = tmem + ((uint32_t)(32 * q) << 16) + set * kGN;
#pragma unroll
      for (int g = 0; g < kGN / KW; ++g) {
        float acc[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = 0.f;
#pragma unroll
        for (int jj = 0; jj < KW / 16; ++jj) {
          const int j = g * (KW / 16) + jj;
          uint32_t v[16];
          tmem_ld_x16(d + 16 * j, v);
          tmem_wait_ld();
          reg_fence(v);
          const uint4 c[2] = {wv[j % kAhead][0], wv[j % kAhead][1]};
          if (j + kAhead < kGN / 16) load(j + kAhead, wv[j % kAhead]);
          const uint32_t cw[8] = {c[0].x, c[0].y, c[0].z, c[0].w, c[1].x, c[1].y, c[1].z, c[1].w};
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            acc[2 * e] = fmaf(__uint_as_float(cw[e] << 16), __uint_as_float(v[2 * e]), acc[2 * e]);
            acc[2 * e + 1] = fmaf(__uint_as_float(cw[e] & 0xFFFF0000u), __uint_as_float(v[2 * e + 1]), acc[2 * e + 1]);
          }
        }
#pragma unroll
        for (int s = 8; s > 0; s >>= 1)
#pragma unroll
          for (int e = 0; e < s; ++e) acc[e] += acc[e + s];
        if (g == kGN / KW - 1) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster_relaxed(empty);   // D may be overwritten
        }
        if (in_row && col0 + g * KW < P.in) {
          const int64_t at = (int64_t)row * n_g + col0 / KW + g;
          P.dlogits[at] = acc[0] * P.dsdl[at];
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (abort_s) {
    // a role gave up: give copies in flight time to land
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 2000000ull) {
    }
  }
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, kGTmemCols);
  }
  cluster_sync_all();
}

template <int KW>
cudaError_t g_launch(const GParams& P, int pairs, cudaStream_t s) {
  static std::once_flag once;
  static cudaError_t attr_err = cudaSuccess;
  std::call_once(once, []() {
    attr_err = cudaFuncSetAttribute(k_group_grad_mma<KW>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGSmem);
  });
  if (attr_err != cudaSuccess) return attr_err;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * pairs));
  cfg.blockDim = dim3(kGThreads);
  cfg.dynamicSmemBytes = kGSmem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_group_grad_mma<KW>, P);
}

}  // namespace

// Where the one-pass kernel applies: row groups, rows in whole 64-wide TMA slabs, 16-byte
// aligned operands.  The rest (square groups, whose sums cross lanes and warps; other row
// counts) forms D with the library and reduces it in a second pass.
bool group_grad_fused(const void* x, const void* W, const gs_packed* p, const void* dy, int64_t T) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(dy);
  const int64_t units = ((p->out + kGM - 1) / kGM) * ((p->in + kGN - 1) / kGN);
  return p->g_out == 1 && (p->g_in == 128 || p->g_in == 256) && p->out % 64 == 0 && (a & 15u) == 0 && T > 0 &&
         T <= INT32_MAX - kGK && units <= INT32_MAX / 2;
}

gs_status launch_group_grad_fused(const void* x, const void* W, const gs_packed* p, const void* dy, int64_t T,
                                  const float* dsdl, float* dlogits, int sm_count, cudaStream_t s) {
  GParams P;
  int* err = device_error_flag();
  if (!err) return GS_ERR_CUDA;
  if (!encode_tmap_slabs_bf16(&P.amap, dy, (uint64_t)p->out, (uint64_t)T, kGK, 2) ||
      !encode_tmap_slabs_bf16(&P.bmap, x, (uint64_t)p->in, (uint64_t)T, kGK, 2))
    return GS_ERR_CUDA;
  P.W = static_cast<const uint16_t*>(W);
  P.dsdl = dsdl;
  P.dlogits = dlogits;
  P.out = (int32_t)p->out;
  P.in = (int32_t)p->in;
  P.n_k = (int32_t)((T + kGK - 1) / kGK);
  P.n_n = (int32_t)((p->in + kGN - 1) / kGN);
  P.n_units = P.n_n * (int32_t)((p->out + kGM - 1) / kGM);
  P.err = err;
  const int pairs = std::min(P.n_units, sm_count / 2);
  const cudaError_t e = p->g_in == 256 ? g_launch<256>(P, pairs, s) : g_launch<128>(P, pairs, s);
  note_launch();
  return e == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

}  // namespace gs
