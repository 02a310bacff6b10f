// Cross-agent fusion of every backbone block's output, the first step of the
// shared post-join subgraph when the multi-scale maps are fused before the
// neck (the fusion/upsampling/concatenation placement of Sec. IV-A and the
// agent-indexed slots of Sec. IV-D): for each block b and each of its BEV
// cells, the present agents' C_b-channel vectors are fused -- per-channel max,
// or scaled dot-product attention with the ego agent 0 as the query -- and
// the fused vector is stored in the storage type.  The neck then runs once on
// the fused maps.
//
// Each thread owns 8 channels (16 bytes) of one cell, so the C_b / 8 threads
// of a cell read each agent's vector with one coalesced 16-byte load apiece
// and a warp covers 32 * 8 / C_b consecutive cells.  The kernel is bound by
// HBM bandwidth: every present agent's block outputs are read once and the
// fused maps written once.  One launch covers all blocks (warp tasks are
// numbered block after block).
//   max:        F = max_k X_k elementwise (exact in the 16-bit domain; the
//               block outputs are ReLU outputs, so a running max from +0
//               equals the max over the present agents)
//   attention:  s_k = <X_0, X_k> / sqrt(C_b), w = softmax over present k,
//               F = sum_k w_k X_k   (fp32; the dot product is each thread's
//               fused multiply-adds, then a butterfly over the cell's
//               threads, so every thread holds the same s_k; the softmax is
//               taken online in one pass over the agents)
// Every reduction has a fixed order: the result is bit-reproducible.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "kernels.h"

namespace rtcc {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kThreads = 256;

template <typename T>
__device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b);
template <>
__device__ __forceinline__ uint32_t max2<__half>(uint32_t a, uint32_t b) {
  __half2 r = __hmax2(*reinterpret_cast<__half2*>(&a), *reinterpret_cast<__half2*>(&b));
  return *reinterpret_cast<uint32_t*>(&r);
}
template <>
__device__ __forceinline__ uint32_t max2<__nv_bfloat16>(uint32_t a, uint32_t b) {
  __nv_bfloat162 r =
      __hmax2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
  return *reinterpret_cast<uint32_t*>(&r);
}

__device__ __forceinline__ uint4 ld16(const void* p) { return *reinterpret_cast<const uint4*>(p); }

// One thread's 8 * NV channels (NV 16-byte vectors) of one cell.  G threads
// share the cell (C = 8 * NV * G); they are lanes [g0, g0 + G) of the warp.
template <typename T, bool ATTN, int G, int NV>
__device__ __forceinline__ void fuse_vec(const T* src, long long astride, const unsigned pres, int K,
                                         size_t off, float inv_sqrt_c, uint4* out) {
  if (!ATTN) {
#pragma unroll
    for (int v = 0; v < NV; ++v) out[v] = make_uint4(0u, 0u, 0u, 0u);
    for (int k = 0; k < K; ++k) {
      if (!((pres >> k) & 1u)) continue;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const uint4 r = ld16(src + (size_t)k * astride + off + 8 * v);
        out[v].x = max2<T>(out[v].x, r.x);
        out[v].y = max2<T>(out[v].y, r.y);
        out[v].z = max2<T>(out[v].z, r.z);
        out[v].w = max2<T>(out[v].w, r.w);
      }
    }
  } else {
    // one pass over the present agents in index order, softmax online: a
    // running maximum m of the scores, the denominator and the weighted sum
    // rescaled by exp(m_old - m_new) when m grows (the ego agent 0, always
    // present, starts them).  The ego vector stays packed (16-bit pairs) for
    // the dot products, so each agent's vector is read once and few
    // registers stay live.
    constexpr int E = 8 * NV;
    uint32_t q[4 * NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const uint4 r = ld16(src + off + 8 * v);
      q[4 * v] = r.x;
      q[4 * v + 1] = r.y;
      q[4 * v + 2] = r.z;
      q[4 * v + 3] = r.w;
    }
    float F[E], m = 0.f, den = 0.f;
#pragma unroll
    for (int k = 0; k < RTCC_MAX_AGENTS; ++k) {
      if (k < K && ((pres >> k) & 1u)) {
        uint32_t x[4 * NV];
        if (k == 0) {
#pragma unroll
          for (int i = 0; i < 4 * NV; ++i) x[i] = q[i];
        } else {
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const uint4 r = ld16(src + (size_t)k * astride + off + 8 * v);
            x[4 * v] = r.x;
            x[4 * v + 1] = r.y;
            x[4 * v + 2] = r.z;
            x[4 * v + 3] = r.w;
          }
        }
        float d = 0.f;
#pragma unroll
        for (int i = 0; i < 4 * NV; ++i) {
          const float2 a = Store<T>::unpack2(q[i]), b = Store<T>::unpack2(x[i]);
          d = fmaf(a.x, b.x, d);
          d = fmaf(a.y, b.y, d);
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) d += __shfl_xor_sync(kFull, d, o);
        const float sk = d * inv_sqrt_c;
        if (k == 0) {
          m = sk;
          den = 1.f;
#pragma unroll
          for (int i = 0; i < 4 * NV; ++i) {
            const float2 b = Store<T>::unpack2(x[i]);
            F[2 * i] = b.x;
            F[2 * i + 1] = b.y;
          }
        } else {
          const float mn = fmaxf(m, sk);
          const float sc = expf(m - mn), wk = expf(sk - mn);
          m = mn;
          den = fmaf(den, sc, wk);
#pragma unroll
          for (int i = 0; i < 4 * NV; ++i) {
            const float2 b = Store<T>::unpack2(x[i]);
            F[2 * i] = fmaf(F[2 * i], sc, wk * b.x);
            F[2 * i + 1] = fmaf(F[2 * i + 1], sc, wk * b.y);
          }
        }
      }
    }
    const float inv = 1.f / den;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      out[v].x = Store<T>::pack2(F[8 * v + 0] * inv, F[8 * v + 1] * inv);
      out[v].y = Store<T>::pack2(F[8 * v + 2] * inv, F[8 * v + 3] * inv);
      out[v].z = Store<T>::pack2(F[8 * v + 4] * inv, F[8 * v + 5] * inv);
      out[v].w = Store<T>::pack2(F[8 * v + 6] * inv, F[8 * v + 7] * inv);
    }
  }
}

// Warp task w of block b: cells [w * 32 / G, (w + 1) * 32 / G) of that block.
template <typename T, bool ATTN, int G, int NV>
__device__ __forceinline__ void block_task(const FuseBlocksArgs& a, int b, int w, int lane, unsigned pres) {
  constexpr int CPW = 32 / G;                       // cells per warp task
  const int cell = w * CPW + lane / G;
  const bool valid = cell < a.cells[b];
  // lanes of a cell past the end still join the butterfly (their data is a
  // clamped copy of the last cell and is not stored)
  const int c = valid ? cell : a.cells[b] - 1;
  const size_t off = (size_t)c * (8 * NV * G) + (size_t)(lane % G) * (8 * NV);
  uint4 v[NV];
  fuse_vec<T, ATTN, G, NV>(static_cast<const T*>(a.src[b]), a.astride[b], pres, a.K, off, a.inv_sqrt_c[b], v);
  if (valid) {
#pragma unroll
    for (int i = 0; i < NV; ++i) reinterpret_cast<uint4*>(static_cast<T*>(a.dst[b]) + off)[i] = v[i];
  }
}

static_assert(RTCC_MAX_BLOCKS == 3, "the task numbering below covers three blocks");

// WIDE: one 384-channel map (the single-scale 384-channel slots; 16 threads of
// 24 channels per cell); otherwise block maps of 32 to 256 channels.  The max
// of the block maps runs 5 blocks per SM (more loads in flight: stress8's
// three maps 12.8 -> 10.7 us against 3 blocks); attention keeps 3 (80
// registers).
template <typename T, bool ATTN, bool WIDE>
__global__ void __launch_bounds__(kThreads, (ATTN || WIDE) ? 3 : 5) k_fuse_blocks(const __grid_constant__ FuseBlocksArgs a) {
  pdl_trigger();
  pdl_wait();
  span_begin(a.span);
  unsigned pres = 0;
  for (int k = 0; k < a.K; ++k) pres |= (a.present[k] ? 1u : 0u) << k;
  const int lane = threadIdx.x & 31;
  const int warps = (int)(gridDim.x * blockDim.x) >> 5;
  // warp tasks of the blocks, numbered block after block
  const int e0 = a.tasks[0];
  const int e1 = e0 + (a.n > 1 ? a.tasks[1] : 0);
  const int e2 = e1 + (a.n > 2 ? a.tasks[2] : 0);
  for (int t = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); t < e2; t += warps) {
    const int b = t < e0 ? 0 : (t < e1 ? 1 : 2);
    const int w = t - (b == 0 ? 0 : (b == 1 ? e0 : e1));
    if (WIDE) {
      block_task<T, ATTN, 16, 3>(a, b, w, lane, pres);
    } else {
      switch (a.ch[b]) {                             // warp-uniform
        case 32: block_task<T, ATTN, 4, 1>(a, b, w, lane, pres); break;
        case 64: block_task<T, ATTN, 8, 1>(a, b, w, lane, pres); break;
        case 128: block_task<T, ATTN, 16, 1>(a, b, w, lane, pres); break;
        default: block_task<T, ATTN, 32, 1>(a, b, w, lane, pres); break;
      }
    }
  }
  if (a.span) {
    __syncthreads();
    span_end(a.span);
  }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Attention over feature slots of C = 128 nb channels with every sum in the
// order of the kernel that fuses without stored slots (k_neck_head), so that
// both give the same bytes: the dot product as one chain over each 32
// channels, those of the same 32 columns added over the nb blocks, then over
// the four column groups; the softmax over all scores, the weights normalised
// before the sums.  Half a warp per cell, 4 nb of its lanes own 32 channels
// each.  The sums need every score first, so a warp brings its two cells'
// vectors of all agents into its part of shared memory (coalesced 16-byte
// copies, all agents in flight together) and reads them there twice: the maps
// are read once.  The chains' results meet in shared memory too, where one lane
// per agent adds them and takes the agent's weight: with every lane doing so for
// all agents the kernel was bound by instructions (2485 a warp and task; 60 us
// for 5 agents on the 352 x 100 map).  Now, with 2, 5 and 8 agents: 22, 36 and
// 53 us, 3.7 to 4.6 TB/s; reading the maps twice took 25, 57 and 89 us, the
// online softmax of k_fuse_blocks, whose sums differ, takes 16, 38 and 57.
constexpr int kDotStride = 33;                   // words per agent of a warp's 32 chain results (bank spread)
constexpr size_t slots_warp_bytes(int K, int C) {
  return (size_t)K * 2 * C * 2 + (size_t)(RTCC_MAX_AGENTS * kDotStride + 8) / 4 * 16;
}
template <typename T>
__global__ void __launch_bounds__(kThreads, 3) k_fuse_slots(const __grid_constant__ FuseBlocksArgs a) {
  extern __shared__ __align__(16) uint8_t slots_smem[];
  pdl_trigger();
  pdl_wait();
  span_begin(a.span);
  unsigned pres = 0;
  for (int k = 0; k < a.K; ++k) pres |= (a.present[k] ? 1u : 0u) << k;
  const int lane = threadIdx.x & 31, h0 = lane & 16, hl = lane & 15;
  const int C = a.ch[0], nb = C / 128, cpc = 16 * nb;        // 16-byte pieces per cell
  const bool mine = hl < 4 * nb;
  const int pair = 2 * cpc;                                  // and per two cells
  uint8_t* const wbase = slots_smem + (threadIdx.x >> 5) * slots_warp_bytes(a.K, C);
  uint4* const ws = reinterpret_cast<uint4*>(wbase);
  float* const dots = reinterpret_cast<float*>(ws + a.K * pair);
  // piece v of this lane's 64 bytes: the pieces of a lane rotate with it, so
  // that eight lanes' reads of piece v fall into different banks
  const uint4* const rd = ws + (lane >> 4) * cpc + (mine ? hl : 0) * 4;
  const int rot = (mine ? hl : 0) >> 1;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < a.tasks[0]; w += warps) {
    for (int i = 0; i < nb; ++i) {
      const int q = lane + 32 * i, c = q >= cpc ? 1 : 0, r = q - c * cpc;
      const int row = min((int)(2 * w) + c, a.cells[0] - 1);   // past the end: the last cell, not stored
      const T* src = static_cast<const T*>(a.src[0]) + (size_t)row * C + r * 8;
      uint4* dst = ws + c * cpc + (r & ~3) + ((r + (r >> 3)) & 3);
#pragma unroll
      for (int k = 0; k < RTCC_MAX_AGENTS; ++k)
        if ((pres >> k) & 1u) cp_async16(dst + k * pair, src + (size_t)k * a.astride[0]);
    }
    cp_async_wait_all();
    __syncwarp();
    float ego[32];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const uint4 x = rd[(v + rot) & 3];
      const uint32_t xk[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 y = Store<T>::unpack2(xk[i]);
        ego[8 * v + 2 * i] = y.x;
        ego[8 * v + 2 * i + 1] = y.y;
      }
    }
    for (unsigned left = pres; left; left &= left - 1u) {
      const int k = __ffs(left) - 1;
      float d = 0.f;
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const uint4 x = rd[k * pair + ((v + rot) & 3)];
        const uint32_t xk[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 y = Store<T>::unpack2(xk[i]);
          d = fmaf(ego[8 * v + 2 * i], y.x, d);
          d = fmaf(ego[8 * v + 2 * i + 1], y.y, d);
        }
      }
      dots[k * kDotStride + lane] = d;
    }
    __syncwarp();
    // lane hl of a cell: agent hl's score, softmax term and weight
    const bool has = hl < RTCC_MAX_AGENTS && ((pres >> hl) & 1u);
    float sc = -INFINITY;
    if (has) {
      const float* d = dots + hl * kDotStride + h0;
      float part[4];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        part[g] = d[g];
        for (int b = 1; b < nb; ++b) part[g] += d[4 * b + g];
      }
      sc = __fmul_rn(part[0] + part[1] + part[2] + part[3], a.inv_sqrt_c[0]);
    }
    float m = sc;
#pragma unroll
    for (int o = RTCC_MAX_AGENTS / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    const float ex = has ? expf(sc - m) : 0.f;
    float den = 0.f;
#pragma unroll
    for (int k = 0; k < RTCC_MAX_AGENTS; ++k) den += __shfl_sync(kFull, ex, h0 + k);
    const float wgt = __fmul_rn(ex, 1.f / den);
    float f[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) f[i] = 0.f;
    for (unsigned left = pres; left; left &= left - 1u) {
      const int k = __ffs(left) - 1;
      const float wk = __shfl_sync(kFull, wgt, h0 + k);
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const uint4 x = rd[k * pair + ((v + rot) & 3)];
        const uint32_t xk[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 y = Store<T>::unpack2(xk[i]);
          f[8 * v + 2 * i] = fmaf(wk, y.x, f[8 * v + 2 * i]);
          f[8 * v + 2 * i + 1] = fmaf(wk, y.y, f[8 * v + 2 * i + 1]);
        }
      }
    }
    const int cell = (int)(2 * w) + (lane >> 4);
    if (mine && cell < a.cells[0]) {
      uint4* out = reinterpret_cast<uint4*>(static_cast<T*>(a.dst[0]) + (size_t)cell * C + hl * 32);
#pragma unroll
      for (int v = 0; v < 4; ++v)
        out[v] = make_uint4(Store<T>::pack2(f[8 * v], f[8 * v + 1]), Store<T>::pack2(f[8 * v + 2], f[8 * v + 3]),
                            Store<T>::pack2(f[8 * v + 4], f[8 * v + 5]), Store<T>::pack2(f[8 * v + 6], f[8 * v + 7]));
    }
    __syncwarp();                                // the next cells overwrite these
  }
  if (a.span) {
    __syncthreads();
    span_end(a.span);
  }
}

template <typename T>
cudaError_t launch_fuse_slots(const FuseBlocksArgs& a, int sms, cudaStream_t st) {
  constexpr int warps = kThreads / 32;
  static_assert(slots_warp_bytes(RTCC_MAX_AGENTS, 384) * warps <= 227 * 1024, "shared memory of a block");
  const size_t smem = slots_warp_bytes(a.K, a.ch[0]) * warps;   // 109 KB for 8 agents of 384 channels
  const cudaError_t e = cudaFuncSetAttribute(k_fuse_slots<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(slots_warp_bytes(RTCC_MAX_AGENTS, 384) * warps));
  if (e != cudaSuccess) return e;
  int per = 0;                                     // one wave: a block more than fits would start at the end
  const cudaError_t eo = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_fuse_slots<T>, kThreads, smem);
  if (eo != cudaSuccess) return eo;
  const long long blocks = std::min<long long>((a.tasks[0] + warps - 1) / warps, (long long)per * sms);
  if (blocks < 1) return cudaErrorInvalidValue;
  return launch_pdl(k_fuse_slots<T>, dim3((unsigned)blocks), dim3(kThreads), smem, st, a);
}

}  // namespace

cudaError_t launch_fuse_blocks(FuseBlocksArgs a, bool bf16, cudaStream_t st) {
  if (a.K < 1 || a.K > RTCC_MAX_AGENTS || a.n < 1 || a.n > RTCC_MAX_BLOCKS) return cudaErrorInvalidValue;
  long long work = 0;
  const bool wide = a.ch[0] == 384;
  if (wide && a.n != 1) return cudaErrorInvalidValue;
  if (a.slot_order && (a.n != 1 || !a.attention || a.ch[0] < 128 || a.ch[0] > 384 || a.ch[0] % 128))
    return cudaErrorInvalidValue;
  for (int b = 0; b < a.n; ++b) {
    if (!wide && a.ch[b] != 32 && a.ch[b] != 64 && a.ch[b] != 128 && a.ch[b] != 256)
      return cudaErrorInvalidValue;
    if (a.cells[b] < 1 || !a.src[b] || !a.dst[b] || a.astride[b] < (long long)a.cells[b] * a.ch[b])
      return cudaErrorInvalidValue;
    // 16-byte loads and stores: every base and the agent stride 16-byte aligned
    if ((reinterpret_cast<uintptr_t>(a.src[b]) | reinterpret_cast<uintptr_t>(a.dst[b])) & 15u ||
        (a.astride[b] * 2) % 16)
      return cudaErrorInvalidValue;
    const int cpw = wide || a.slot_order ? 2 : 32 / (a.ch[b] / 8);   // cells per warp task
    a.tasks[b] = (a.cells[b] + cpw - 1) / cpw;
    a.inv_sqrt_c[b] = 1.0f / sqrtf((float)a.ch[b]);
    work += a.tasks[b];
  }
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long per_block = kThreads / 32;
  long long blocks = (work + per_block - 1) / per_block;
  if (blocks > 8LL * sms) blocks = 8LL * sms;       // grid-stride beyond 8 blocks per SM
  if (blocks < 1) blocks = 1;
  const dim3 g((unsigned)blocks), t(kThreads);
  if (a.slot_order) return bf16 ? launch_fuse_slots<__nv_bfloat16>(a, sms, st) : launch_fuse_slots<__half>(a, sms, st);
  if (bf16) {
    if (wide)
      return a.attention ? launch_pdl(k_fuse_blocks<__nv_bfloat16, true, true>, g, t, 0, st, a)
                         : launch_pdl(k_fuse_blocks<__nv_bfloat16, false, true>, g, t, 0, st, a);
    return a.attention ? launch_pdl(k_fuse_blocks<__nv_bfloat16, true, false>, g, t, 0, st, a)
                       : launch_pdl(k_fuse_blocks<__nv_bfloat16, false, false>, g, t, 0, st, a);
  }
  if (wide)
    return a.attention ? launch_pdl(k_fuse_blocks<__half, true, true>, g, t, 0, st, a)
                       : launch_pdl(k_fuse_blocks<__half, false, true>, g, t, 0, st, a);
  return a.attention ? launch_pdl(k_fuse_blocks<__half, true, false>, g, t, 0, st, a)
                     : launch_pdl(k_fuse_blocks<__half, false, false>, g, t, 0, st, a);
}

}  // namespace rtcc
