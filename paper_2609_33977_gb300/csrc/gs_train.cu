// Training-side selectors (Sec. 2.2): a Gumbel-Sigmoid sample with a
// straight-through estimator (STE), and the backward pass of the masked linear
// y = x (W (.) (B (x) 1))^T with W frozen.
//
//   sample:   z = l + L (L: logistic noise, the difference of two standard
//             Gumbel draws, supplied by the caller), B = [z > 0] (the binary
//             selectors of the forward pass), and the derivative of the
//             relaxation s = sigmoid(z / tau) that the backward pass uses,
//             ds/dl = s (1 - s) / tau, written as t / (1 + t)^2 / tau with
//             t = exp(-|z| / tau) so that it keeps its precision where s is
//             near 0 or 1 (1 - s would cancel in float32).
//   backward: dL/dW_hat = dy^T x, dL/dB[u, v] = sum over the group of
//             W (.) dL/dW_hat, and the STE gives dL/dl = dL/dB ds/dl;
//             dL/dx = dy W_hat.
//
// dy^T x covers all groups, pruned ones included, since the STE passes gradients
// to every selector.  For row groups with whole 64-row slabs it stays on chip
// (gs_group_grad.cu); elsewhere cuBLAS forms it as a plain dense GEMM in the
// workspace and a kernel of this file reduces it with the STE factor.  dy W_hat
// on the masked weight is a cuBLAS GEMM.  The sampling is a kernel of this file;
// the forward pass is gs_pack with the sampled mask followed by gs_linear.
#include "gs_common.cuh"

#include <cublas_v2.h>
#include <algorithm>
#include <mutex>

namespace gs {
namespace {

constexpr int kGumbelThreads = 256;
constexpr int kGumbelWarps = kGumbelThreads / 32;
constexpr int64_t kGumbelPerWarp = 256;   // selectors per warp step: two 16-byte loads of each input per thread
constexpr int kGumbelSteps = 4;           // most warp steps per block and warp

// tau as the kernel uses it.  For tau in [2^-60, 2^60] 1 / tau is the sum of
// two floats, hi + lo: x / tau is then fma(x, hi, x lo), which rounds once
// (the product by lo is 2^-24 of the result), and d d / (1 / tau) needs one
// division instead of two.  Outside that range hi, lo or the products could
// overflow or lose bits to underflow, and the divisions are taken as written.
struct GumbelTau {
  float tau, hi, lo;
  int by_product;
};

__device__ __forceinline__ float over_tau(float x, const GumbelTau& t) { return fmaf(x, t.hi, x * t.lo); }

// {kept, ds/dl} of one selector
__device__ __forceinline__ bool gumbel_one(float l, float n, const GumbelTau& tau, float& ds) {
  const float z = __fadd_rn(l, n);
  const float az = fabsf(z);
  if (tau.by_product) {
    const float big = 0x1p67f;   // exp(-2^67 / tau) is 0 up to tau = 2^60; keeps inf out of the fma, lets NaN through
    const float t = expf(-over_tau(az > big ? big : az, tau));
    const float d = 1.f + t;
    ds = __fdiv_rn(over_tau(t, tau), d * d);
  } else {
    const float t = expf(-__fdiv_rn(az, tau.tau));
    const float d = 1.f + t;
    ds = __fdiv_rn(__fdiv_rn(t, d * d), tau.tau);
  }
  return z > 0.f;   // NaN prunes
}

// the block's kept count: one 64-bit atomic
__device__ __forceinline__ void add_kept(unsigned int cnt, unsigned long long* kept) {
  if (kept == nullptr) return;   // uniform over the grid
  __shared__ unsigned int warp_cnt[kGumbelWarps];
  const unsigned int w = __reduce_add_sync(0xffffffffu, cnt);
  if ((threadIdx.x & 31) == 0) warp_cnt[threadIdx.x >> 5] = w;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int total = 0;
#pragma unroll
    for (int i = 0; i < kGumbelWarps; ++i) total += warp_cnt[i];
    if (total) atomicAdd(kept, (unsigned long long)total);
  }
}

// HBM-bound: 13 bytes per selector.  A warp step covers 256 consecutive
// selectors, two 16-byte loads of each input and two 16-byte + two 4-byte
// stores per thread; a block takes kGumbelWarps * steps consecutive warp
// steps and adds its count with one atomic.  25.3 M selectors (329 MB): 55.6 us
// a call, 5.92 TB/s; one selector per thread with an atomic per warp took
// 135 us (65 K atomics to one address, byte stores, two divisions).
template <bool DS>
__global__ void __launch_bounds__(kGumbelThreads) k_gumbel4(const float4* __restrict__ logits,
                                                            const float4* __restrict__ noise, int64_t n, int steps,
                                                            GumbelTau tau, uint32_t* __restrict__ mask,
                                                            float4* __restrict__ dsdl,
                                                            unsigned long long* __restrict__ kept) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t nfull = n / kGumbelPerWarp;
  unsigned int cnt = 0;
  for (int k = 0; k < steps; ++k) {
    const int64_t u = ((int64_t)blockIdx.x * steps + k) * kGumbelWarps + warp;
    if (u >= nfull) break;
    const int64_t at = u * (kGumbelPerWarp / 4) + lane;
    float4 l[2], g[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      l[q] = __ldcs(logits + at + 32 * q);
      g[q] = __ldcs(noise + at + 32 * q);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float4 d;
      const uint32_t m = (gumbel_one(l[q].x, g[q].x, tau, d.x) ? 1u : 0u) |
                         (gumbel_one(l[q].y, g[q].y, tau, d.y) ? 0x100u : 0u) |
                         (gumbel_one(l[q].z, g[q].z, tau, d.z) ? 0x10000u : 0u) |
                         (gumbel_one(l[q].w, g[q].w, tau, d.w) ? 0x1000000u : 0u);
      mask[at + 32 * q] = m;
      if (DS) dsdl[at + 32 * q] = d;
      cnt += __popc(m);
    }
  }
  // the last n % 256 selectors, one per thread of block 0
  if (blockIdx.x == 0) {
    const int64_t i = nfull * kGumbelPerWarp + threadIdx.x;
    if (i < n) {
      float d;
      const bool keep = gumbel_one(reinterpret_cast<const float*>(logits)[i], reinterpret_cast<const float*>(noise)[i],
                                   tau, d);
      reinterpret_cast<uint8_t*>(mask)[i] = keep ? 1 : 0;
      if (DS) reinterpret_cast<float*>(dsdl)[i] = d;
      cnt += keep ? 1u : 0u;
    }
  }
  add_kept(cnt, kept);
}

// the same for pointers that 16-byte (inputs, ds/dl) or 4-byte (mask) accesses
// do not fit: one selector per thread and step
__global__ void __launch_bounds__(kGumbelThreads) k_gumbel(const float* __restrict__ logits,
                                                           const float* __restrict__ noise, int64_t n, GumbelTau tau,
                                                           uint8_t* __restrict__ mask, float* __restrict__ dsdl,
                                                           unsigned long long* __restrict__ kept) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  unsigned int cnt = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    float d;
    const bool keep = gumbel_one(logits[i], noise[i], tau, d);
    mask[i] = keep ? 1 : 0;
    if (dsdl) dsdl[i] = d;
    cnt += keep ? 1u : 0u;
  }
  add_kept(cnt, kept);
}

// dlogits[u, v] = ds/dl[u, v] * sum over group (u, v) of W (.) D, D = dy^T x
// (fp32 [out][in]); one warp per group, lanes over the group's cells four at a time
__global__ void k_group_grad(const uint16_t* __restrict__ W, const float* __restrict__ D, const float* __restrict__ dsdl,
                             int32_t out, int32_t in, int32_t g_out, int32_t g_in, float* __restrict__ dlogits) {
  const int lane = threadIdx.x & 31;
  const int64_t Gin = in / g_in, n = (int64_t)(out / g_out) * Gin;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int per_row = g_in / 4;
  for (int64_t e = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); e < n; e += warps) {
    const int64_t u = e / Gin, v = e % Gin;
    float acc = 0.f;
    for (int c = lane; c < g_out * per_row; c += 32) {
      const int64_t r = u * g_out + c / per_row;
      const int64_t k = v * g_in + 4 * (c % per_row);
      const float4 d = *reinterpret_cast<const float4*>(D + r * in + k);
      const uint2 wb = *reinterpret_cast<const uint2*>(W + r * in + k);
      acc = fmaf(__uint_as_float(wb.x << 16), d.x, acc);
      acc = fmaf(__uint_as_float(wb.x & 0xFFFF0000u), d.y, acc);
      acc = fmaf(__uint_as_float(wb.y << 16), d.z, acc);
      acc = fmaf(__uint_as_float(wb.y & 0xFFFF0000u), d.w, acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) dlogits[e] = acc * dsdl[e];
  }
}

std::mutex g_blas_mu;
cublasHandle_t g_blas[64] = {nullptr};

gs_status blas_handle(cublasHandle_t* h) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return GS_ERR_CUDA;
  if (!g_blas[dev] && cublasCreate(&g_blas[dev]) != CUBLAS_STATUS_SUCCESS) {
    g_blas[dev] = nullptr;
    return GS_ERR_CUDA;
  }
  *h = g_blas[dev];
  return GS_OK;
}

int sm_count_train() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 148;
  }
  return n;
}

size_t round256(size_t b) { return (b + 255) & ~size_t(255); }

}  // namespace

gs_status launch_gumbel(const float* logits, const float* noise, int64_t n, float tau, uint8_t* mask, float* dsdl,
                        int64_t* kept, cudaStream_t s) {
  if (kept && cudaMemsetAsync(kept, 0, sizeof(int64_t), s) != cudaSuccess) return GS_ERR_CUDA;
  if (n == 0) return GS_OK;
  GumbelTau t{tau, 0.f, 0.f, 0};
  if (tau >= 0x1p-60f && tau <= 0x1p60f) {
    const double inv = 1.0 / (double)tau;
    t.hi = (float)inv;
    t.lo = (float)(inv - (double)t.hi);
    t.by_product = 1;
  }
  unsigned long long* k64 = reinterpret_cast<unsigned long long*>(kept);
  const uintptr_t a16 = reinterpret_cast<uintptr_t>(logits) | reinterpret_cast<uintptr_t>(noise) |
                        reinterpret_cast<uintptr_t>(dsdl);   // a NULL ds/dl adds no bits
  if ((a16 & 15u) == 0 && (reinterpret_cast<uintptr_t>(mask) & 3u) == 0) {
    // blocks of up to four steps per warp; fewer while that leaves the SMs short of blocks
    const int64_t per_block = kGumbelPerWarp * kGumbelWarps;
    const int64_t units = (n + per_block - 1) / per_block;
    const int64_t steps = std::min<int64_t>(kGumbelSteps, std::max<int64_t>(1, units / (8 * sm_count_train())));
    // n < 2^36 keeps the grid below 2^23
    const unsigned grid = (unsigned)((units + steps - 1) / steps);
    auto kern = dsdl ? k_gumbel4<true> : k_gumbel4<false>;
    kern<<<grid, kGumbelThreads, 0, s>>>(reinterpret_cast<const float4*>(logits), reinterpret_cast<const float4*>(noise),
                                         n, (int)steps, t, reinterpret_cast<uint32_t*>(mask),
                                         reinterpret_cast<float4*>(dsdl), k64);
  } else {
    const int64_t blocks = std::min<int64_t>((n + kGumbelThreads - 1) / kGumbelThreads, 8 * sm_count_train());
    k_gumbel<<<(unsigned)blocks, kGumbelThreads, 0, s>>>(logits, noise, n, t, mask, dsdl, k64);
  }
  note_launch();
  return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

size_t backward_workspace_bytes(const gs_packed* p, bool want_dx) {
  const size_t cells = (size_t)p->out * (size_t)p->in;
  return round256(4 * cells) + (want_dx ? round256(2 * cells) : 0);
}

gs_status launch_backward(const void* x, const void* W, const gs_packed* p, const void* dy, int64_t T,
                          const float* dsdl, float* dlogits, void* dx, void* ws, cudaStream_t s) {
  const int64_t out = p->out, in = p->in;
  float* D = static_cast<float*>(ws);
  const bool fused = group_grad_fused(x, W, p, dy, T);
  if (fused) {
    const gs_status st = launch_group_grad_fused(x, W, p, dy, T, dsdl, dlogits, sm_count_train(), s);
    if (st != GS_OK || !dx) return st;
  }
  {
    std::lock_guard<std::mutex> lk(g_blas_mu);
    cublasHandle_t h = nullptr;
    gs_status st = blas_handle(&h);
    if (st != GS_OK) return st;
    if (cublasSetStream(h, s) != CUBLAS_STATUS_SUCCESS) return GS_ERR_CUDA;
    const float one = 1.f, zero = 0.f;
    // D [out][in] = dy^T x.  In cuBLAS's column-major terms D is (in x out) =
    // A (in x T) * B (T x out): x row-major [T][in] is A as stored; dy
    // row-major [T][out] is (out x T) as stored, so B is it transposed.
    if (!fused && cublasGemmEx(h, CUBLAS_OP_N, CUBLAS_OP_T, (int)in, (int)out, (int)T, &one, x, CUDA_R_16BF, (int)in, dy,
                     CUDA_R_16BF, (int)out, &zero, D, CUDA_R_32F, (int)in, CUBLAS_COMPUTE_32F,
                     CUBLAS_GEMM_DEFAULT) != CUBLAS_STATUS_SUCCESS)
      return GS_ERR_CUDA;
    if (dx) {
      // W_hat (dense, pruned groups +0.0) then dx [T][in] = dy W_hat:
      // column-major (in x T) = W_hat as (in x out) * dy as (out x T)
      uint16_t* What = reinterpret_cast<uint16_t*>(static_cast<uint8_t*>(ws) + round256(4 * (size_t)out * in));
      if (p->g_out > 1) st = sq_unpack(p, What, s);
      else st = launch_unpack(p, What, s);
      if (st != GS_OK) return st;
      if (cublasGemmEx(h, CUBLAS_OP_N, CUBLAS_OP_N, (int)in, (int)T, (int)out, &one, What, CUDA_R_16BF, (int)in, dy,
                       CUDA_R_16BF, (int)out, &zero, dx, CUDA_R_16BF, (int)in, CUBLAS_COMPUTE_32F,
                       CUBLAS_GEMM_DEFAULT) != CUBLAS_STATUS_SUCCESS)
        return GS_ERR_CUDA;
    }
  }
  if (fused) return GS_OK;
  const int64_t groups = (int64_t)(out / p->g_out) * (in / p->g_in);
  int64_t blocks = (groups + 7) / 8;
  if (blocks > (1 << 20)) blocks = 1 << 20;
  k_group_grad<<<(unsigned)blocks, 256, 0, s>>>(static_cast<const uint16_t*>(W), D, dsdl, (int32_t)out, (int32_t)in,
                                                p->g_out, p->g_in, dlogits);
  note_launch();
  return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

}  // namespace gs
