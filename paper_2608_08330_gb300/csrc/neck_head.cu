// The deconv neck, the cross-agent fusion and the 1x1 detection head in one
// kernel (the shared post-join subgraph, Sec. III-B / Sec. IV-D), on the
// 5th-generation tensor cores.
//
//   X_k[cell][128 b + c] = relu(bias_b[c] + sum_i W_b[sub][c][i] Y_kb[pixel][i])
//   F[cell][.]           = max over present agents k of X_k[cell][.], or
//                          sum_k w_k X_k[cell][.], w = softmax over present k of
//                          <X_0[cell], X_k[cell]> / sqrt(128 blocks)  (attention)
//   out[cell][o]         = head_b[o] + sum_c W_head[o][c] F[cell][c],  o < 16
//
// with Y_kb agent k's output of backbone block b, pixel the input pixel under
// the cell and sub the cell's position within it (kernel = stride = s_b).
//
// Why one kernel.  Run by the branches, the neck writes 384 channels per cell
// and agent that the fusion then reads back: on the 352 x 100 map with 8
// agents 2 x 216 MB through HBM, 125 us of deconvs behind the last conv (their
// strided 128-channel stores bound them) and 48 us of fusion (0.67 of the
// measured copy rate).  The blocks' outputs are 63 MB, mostly still in the
// 129 MB L2, and the deconvs' 32 GFLOP are a fraction of the tensor cores'
// time, so here the neck's output never leaves the SM.
//
// The maximum is taken on the fp32 accumulators, before bias, ReLU and the
// rounding to 16 bits: all three are monotone, so rounding the maximum gives
// the very bits of the maximum of the rounded values.
//
// Attention needs the scores over all 384 channels before the first sum, so an
// item makes two passes over blocks and agents: the first computes every X_k
// (rounded to 16 bits, as stored maps are) and its dot product with the ego's,
// the second computes it again and adds w_k X_k in fp32.  Computing twice costs
// the MMAs of 21 GFLOP and the L2 reads of the blocks' outputs once more: 66 us
// for 5 agents on the 352 x 100 map, near the 50 us of its 315 MB of L2 reads.
// Storing the maps cost 68 us of deconvs in the branches' launch, 38 us of
// fusion and 14 us of head.  Where the maps are stored all the same,
// k_fuse_slots (fuse_blocks.cu) takes the sums in this kernel's order.
// The fused map itself is written out: it stands for read-backs until the next
// frame's fusion, whatever the branches have overwritten by then.  The chunks
// the head reads go out as TMA boxes beside its MMAs, 27 MB on the 352 x 100
// map: the kernel takes 64.4 us without the store and 65.7 with it, the frame of
// 5 agents 481 to 484 and 482.
//
// Work item: 128 cells that share their position (sy, sx) modulo the largest
// stride S, i.e. cells (S qy + sy, S qx + sx) of a tw x th rectangle of
// (qx, qy).  They have one weight matrix per block -- 128 x C_b, all of them
// resident in shared memory (112 KB for 64 + 128 + 256 channels) while the CTA
// stays at that position -- and their pixels of block b form a dense
// rectangle of a strided view of its map: one TMA box of 64 channels per
// chunk (5-D view (r C, W / r, r, H / r, agent), r = S / s_b).  Items are
// numbered position-major and each CTA takes a contiguous range.
// The rectangle is the one that covers the map with the fewest tiles (88 x 25:
// 5 x 25, 18 tiles against 22 of 8 x 16).
//
// Per item and block: for each present agent the block's chunks accumulate
// into one of three 128-column accumulators; the epilogue keeps the running
// maximum in registers (32 columns per thread); after the last agent it adds
// the bias, applies ReLU, rounds and writes the 128 x 128 fused chunk as the A
// operand of the head's N = 16 MMAs, which accumulate over the blocks in
// channel order.
//
// Roles (800 threads; attention 768): warps 0..15 fusion epilogue
// (tensor-memory lane quarter warp % 4, columns 32 (warp / 4)), warps 16..19
// head epilogue, then four warps (attention three) with one TMA producer thread
// each (a thread's boxes complete one after another, so the stages are dealt
// over them), the last warp tensor-memory owner and MMA issuer.  Attention's
// first head epilogue warp also stores the fused map.  Every wait is bounded (an
// error bit, no hang); the summation order is fixed, so the output is
// bit-reproducible.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "common.cuh"
#include "kernels.h"

namespace rtcc {

namespace {

constexpr int kEpiWarps = 16;
constexpr int kHeadWarp0 = kEpiWarps;          // 4 head epilogue warps
constexpr int kProdWarp0 = kHeadWarp0 + 4;
// Producer warps: attention has one less, which makes 24 warps and 80 registers
// a thread instead of 72.  Its epilogue keeps its biases packed in shared memory
// and loads 8 columns at a time for the same reason: with 50 words spilled the
// kernel took 119 us instead of 64.
constexpr int producers(bool attn) { return attn ? 3 : 4; }
constexpr int threads(bool attn) { return (kProdWarp0 + producers(attn) + 1) * 32; }
constexpr int kStages = 4;
constexpr int kTile = 128;                     // cells per item (MMA M)
constexpr int kUp = 128;                       // channels per deconv
constexpr int kChunk = kTile * 64 * 2;         // 64 channels of 128 rows, 128-byte swizzle
constexpr int kMaxChunks = 7;                  // weight chunks resident per position
constexpr int kHeadChunk = kFuseHeadOut * 64 * 2;
constexpr int kAccs = 3;
constexpr uint32_t kHeadCol = kAccs * kUp;     // two 16-column head accumulators follow
constexpr uint32_t kTmemCols = 512;
// shared memory: A stages, resident weights, fused chunk pair, head weights
constexpr int kWOff = kStages * kChunk;
constexpr int kFOff = kWOff + kMaxChunks * kChunk;
constexpr int kHOff = kFOff + 2 * kChunk;
constexpr int kBarOff = kHOff + RTCC_MAX_BLOCKS * 2 * kHeadChunk;
constexpr int kSmem = kBarOff + 256 + 1024;    // barriers; alignment to 1024
// the static arrays: biases, agent list and count, attention's weights
constexpr int static_smem(bool attn) {
  return RTCC_MAX_BLOCKS * kUp * 4 + RTCC_MAX_AGENTS * 4 + 16 + (attn ? RTCC_MAX_AGENTS * kTile : 1) * 4;
}
static_assert(kSmem + static_smem(true) <= 227 * 1024 && kSmem + static_smem(false) <= 227 * 1024,
              "shared memory of a block");
// the producers take turns on the stages: a thread's wait for a stage rules out
// the phase before the one its next wait is for
static_assert(producers(false) <= kStages, "phase parity");

// tile t of a CTA's range: position (sy, sx), origin in the quotient grid
struct NhItem {
  int sub, sy, sx, x0, y0;
};
__device__ __forceinline__ NhItem item_at(const NeckHeadParams& P, int t) {
  NhItem I;
  I.sub = t / P.tiles;
  const int tau = t - I.sub * P.tiles;
  I.sy = I.sub / P.S;
  I.sx = I.sub - I.sy * P.S;
  const int ty = tau / P.tiles_x;
  I.x0 = (tau - ty * P.tiles_x) * P.tw;
  I.y0 = ty * P.th;
  return I;
}

// barrier among the 16 epilogue warps (named barrier 1)
__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory"); }

// ATTN: attention fusion instead of the maximum (see the top of the file).
template <typename T, bool ATTN>
__global__ void __launch_bounds__(threads(ATTN), 1) k_neck_head(const __grid_constant__ NeckHeadParams P) {
  constexpr int kProducers = producers(ATTN), kMmaWarp = kProdWarp0 + kProducers, kThreads = threads(ATTN);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* wsm = smem + kWOff;
  uint8_t* fsm = smem + kFOff;
  uint8_t* hsm = smem + kHOff;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kBarOff);   // [kStages]
  uint64_t* empty = full + kStages;            // [kStages]
  uint64_t* accfull = empty + kStages;         // [kAccs]
  uint64_t* accempty = accfull + kAccs;        // [kAccs]
  uint64_t* hfull = accempty + kAccs;          // [2] head accumulator complete
  uint64_t* hempty = hfull + 2;                // [2]
  uint64_t* wfull = hempty + 2;                // a position's weights landed
  uint64_t* wempty = wfull + 1;                // the MMAs that read them are done
  uint64_t* hwfull = wempty + 1;               // head weights landed
  uint64_t* fready = hwfull + 1;               // fused chunk pair written
  uint64_t* fempty = fready + 1;               // head MMAs (and the fused map's store) have read it
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fempty + 1);
  __shared__ __align__(16) float s_bias[RTCC_MAX_BLOCKS][kUp];
  __shared__ int s_list[RTCC_MAX_AGENTS];
  __shared__ int s_kp;
  __shared__ float s_w[ATTN ? RTCC_MAX_AGENTS : 1][ATTN ? kTile : 1];   // an item's weights, agents in list order
  static_assert(sizeof(s_bias) + sizeof(s_list) + sizeof(s_kp) + sizeof(s_w) <= static_smem(ATTN), "see static_smem");

  const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0);   // warp-uniform
  const int lane = threadIdx.x & 31;
  const int nb = P.n_blocks;
  const int n_items = P.S * P.S * P.tiles;
  const int lo = (int)((long long)blockIdx.x * n_items / gridDim.x);
  const int hi = (int)((long long)(blockIdx.x + 1) * n_items / gridDim.x);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < kAccs; ++a) {
      mbar_init(&accfull[a], 1);
      mbar_init(&accempty[a], kEpiWarps);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(&hfull[h], 1);
      mbar_init(&hempty[h], 4);
    }
    mbar_init(wfull, kProducers);
    mbar_init(wempty, 1);
    mbar_init(hwfull, 1);
    mbar_init(fready, kEpiWarps);
    mbar_init(fempty, ATTN ? 2 : 1);           // the head MMAs' commit; the fused map's store
    fence_barrier_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  // the biases; for attention two a word in the storage type, which holds them
  uint32_t* const bias2 = reinterpret_cast<uint32_t*>(&s_bias[0][0]);
  if (ATTN) {
    for (int i = threadIdx.x; i < nb * kUp / 2; i += kThreads) {
      const float* b = P.bias[i / (kUp / 2)] + i % (kUp / 2) * 2;
      bias2[i] = Store<T>::pack2(b[0], b[1]);
    }
  } else {
    for (int i = threadIdx.x; i < nb * kUp; i += kThreads) s_bias[i / kUp][i % kUp] = P.bias[i / kUp][i % kUp];
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();

  // Weights of position `sub`: producer thread pid issues every kProducers-th
  // of the 64-channel chunks (blocks in order, chunk index running on).
  auto load_weights = [&](const NhItem& I, int pid) {
    uint32_t mine = 0;
    int idx = 0;
    for (int b = 0; b < nb; ++b)
      for (int c = 0; c < P.cin[b] / 64; ++c, ++idx)
        if (idx % kProducers == pid) mine += kChunk;
    mbar_arrive_expect_tx(wfull, mine);
    idx = 0;
    for (int b = 0; b < nb; ++b) {
      const int s = P.s[b];
      const int row = ((I.sy % s) * s + I.sx % s) * kUp;
      for (int c = 0; c < P.cin[b] / 64; ++c, ++idx)
        if (idx % kProducers == pid) tma_load_2d(wsm + idx * kChunk, &P.w[b], wfull, c * 64, row);
    }
  };
  // the weights are constant: the first position's loads overlap the previous kernel
  const int pid = warp - kProdWarp0;
  const bool producer = pid >= 0 && pid < kProducers && lane == 0;
  if (producer && lo < hi) {
    if (pid == 0) {
      mbar_arrive_expect_tx(hwfull, (uint32_t)(nb * 2 * kHeadChunk));
      for (int j = 0; j < nb * 2; ++j) tma_load_2d(hsm + j * kHeadChunk, &P.wh, hwfull, j * 64, 0);
    }
    load_weights(item_at(P, lo), pid);
  }
  pdl_wait();                                  // the maps are the branches' output
  span_begin(P.span);
  if (threadIdx.x == 0) {
    int n = 0;
    for (int k = 0; k < P.K; ++k)
      if (P.present[k]) s_list[n++] = k;
    s_kp = n;
  }
  __syncthreads();
  const int Kp = s_kp;

  constexpr int kPasses = ATTN ? 2 : 1;        // passes over the agents per item
  if (warp < kEpiWarps && ATTN) {
    // ---------------- attention: scores, softmax, weighted sums ----------------
    const int qd = warp & 3, cg = warp >> 2;
    const int row = qd * 32 + lane;
    const uint32_t tcol = tmem + (static_cast<uint32_t>(qd * 32) << 16) + (uint32_t)(cg * 32);
    uint8_t* frow = fsm + (cg >> 1) * kChunk + row * 128;
    float* part = reinterpret_cast<float*>(fsm);   // [agent][column group][row] score parts
    uint32_t st = 0, ph = 0;
    bool alive = true;
    // 8 columns from column 8 h on of the step in hand, rounded after bias and
    // ReLU, two a word (8 at a time, to stay within a thread's registers)
    auto rounded8 = [&](int h, const uint32_t* bias, uint32_t (&x)[4]) {
      uint32_t r[8];
      tmem_ld8_issue(tcol + (st % kAccs) * kUp + 8 * h, r);
      const uint4 pb = *reinterpret_cast<const uint4*>(bias + 4 * h);
      const uint32_t bb[4] = {pb.x, pb.y, pb.z, pb.w};
      tmem_ld_wait();
      tmem_reg_fence(r);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 b = Store<T>::unpack2(bb[i]);
        x[i] = Store<T>::relu2(Store<T>::pack2(__uint_as_float(r[2 * i]) + b.x, __uint_as_float(r[2 * i + 1]) + b.y));
      }
    };
    auto wait_full = [&]() {
      if (alive && !mbar_wait(&accfull[st % kAccs], (st / kAccs) & 1, P.wait_budget)) {
        if (lane == 0) atomicOr(P.err, ERR_WAIT_FUSE);
        alive = false;
      }
      tc_fence_after();
    };
    auto release = [&]() {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&accempty[st % kAccs]);
    };
    auto wait_fempty = [&]() {                 // the head MMAs of the block before have read the fused chunk
      if (alive && !mbar_wait(fempty, (ph & 1) ^ 1, P.wait_budget)) {
        if (lane == 0) atomicOr(P.err, ERR_WAIT_FUSE);
        alive = false;
      }
    };
    for (int t = lo; t < hi; ++t) {
      // First pass: <X_ego, X_k> over this thread's channels of every block, in
      // the fused chunk's memory, which is idle until the second pass.
      wait_fempty();
      float* mine = part + cg * kTile + row;   // agent k's part: + 4 k kTile
      for (int b = 0; b < nb; ++b) {
        const uint32_t* bias = bias2 + b * (kUp / 2) + cg * 16;   // of this thread's 32 channels
        uint32_t ego[16];
        for (int k = 0; k < Kp; ++k, ++st) {
          wait_full();
          float d = 0.f;
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            uint32_t x[4];
            rounded8(h, bias, x);
            if (h == 3) release();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (k == 0) ego[4 * h + i] = x[i];
              const float2 a = Store<T>::unpack2(ego[4 * h + i]), c = Store<T>::unpack2(x[i]);
              d = fmaf(a.x, c.x, d);
              d = fmaf(a.y, c.y, d);
            }
          }
          mine[4 * k * kTile] = b == 0 ? d : mine[4 * k * kTile] + d;
        }
      }
      epilogue_sync();
      // the column groups' parts meet: group 0 takes the softmax, a row a thread
      if (cg == 0) {
        float w[RTCC_MAX_AGENTS], m = -INFINITY, den = 0.f;
#pragma unroll
        for (int j = 0; j < RTCC_MAX_AGENTS; ++j) {
          if (j < Kp) {
            const float* q = part + j * 4 * kTile + row;
            w[j] = __fmul_rn(q[0] + q[kTile] + q[2 * kTile] + q[3 * kTile], P.inv_sqrt_c);
            m = fmaxf(m, w[j]);
          }
        }
#pragma unroll
        for (int j = 0; j < RTCC_MAX_AGENTS; ++j) {
          w[j] = j < Kp ? expf(w[j] - m) : 0.f;
          den += w[j];
        }
        const float inv = 1.f / den;
#pragma unroll
        for (int j = 0; j < RTCC_MAX_AGENTS; ++j) s_w[j][row] = __fmul_rn(w[j], inv);
      }
      epilogue_sync();                         // the parts have been read, the weights written
      // second pass: the weighted sums
      for (int b = 0; b < nb; ++b, ++ph) {
        const uint32_t* bias = bias2 + b * (kUp / 2) + cg * 16;
        float f[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) f[i] = 0.f;
        for (int k = 0; k < Kp; ++k, ++st) {
          const float wk = s_w[k][row];
          wait_full();
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            uint32_t x[4];
            rounded8(h, bias, x);
            if (h == 3) release();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float2 c = Store<T>::unpack2(x[i]);
              f[8 * h + 2 * i] = fmaf(wk, c.x, f[8 * h + 2 * i]);
              f[8 * h + 2 * i + 1] = fmaf(wk, c.y, f[8 * h + 2 * i + 1]);
            }
          }
        }
        wait_fempty();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float* v = f + 8 * j;
          *reinterpret_cast<uint4*>(frow + ((((cg & 1) * 4 + j) ^ (row & 7)) << 4)) =
              make_uint4(Store<T>::pack2(v[0], v[1]), Store<T>::pack2(v[2], v[3]), Store<T>::pack2(v[4], v[5]),
                         Store<T>::pack2(v[6], v[7]));
        }
        fence_async_smem();                    // generic writes -> the MMA
        __syncwarp();
        if (lane == 0) mbar_arrive(fready);
      }
    }
  } else if (warp < kEpiWarps) {
    // ---------------- running max, bias + ReLU + rounding ----------------
    const int qd = warp & 3, cg = warp >> 2;
    const int row = qd * 32 + lane;
    const uint32_t tcol = tmem + (static_cast<uint32_t>(qd * 32) << 16) + (uint32_t)(cg * 32);
    // this thread's 32 channels of row `row` in the fused chunk pair: 16-byte
    // pieces 4 (cg & 1) .. + 3 of the row in chunk cg / 2, 128-byte swizzle
    uint8_t* frow = fsm + (cg >> 1) * kChunk + row * 128;
    uint32_t st = 0, ph = 0;
    bool alive = true;
    for (int t = lo; t < hi; ++t) {
      for (int b = 0; b < nb; ++b, ++ph) {
        float mx[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) mx[i] = -INFINITY;
        for (int k = 0; k < Kp; ++k, ++st) {
          const uint32_t buf = st % kAccs;
          if (alive && !mbar_wait(&accfull[buf], (st / kAccs) & 1, P.wait_budget)) {
            if (lane == 0) atomicOr(P.err, ERR_WAIT_FUSE);
            alive = false;
          }
          tc_fence_after();
          uint32_t r0[16], r1[16];
          tmem_ld16_issue(tcol + buf * kUp, r0);
          tmem_ld16_issue(tcol + buf * kUp + 16, r1);
          tmem_ld_wait();
          tmem_reg_fence(r0);
          tmem_reg_fence(r1);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&accempty[buf]);
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            mx[i] = fmaxf(mx[i], __uint_as_float(r0[i]));
            mx[16 + i] = fmaxf(mx[16 + i], __uint_as_float(r1[i]));
          }
        }
        // the head MMAs of the previous block have read the fused chunk pair
        if (alive && !mbar_wait(fempty, (ph & 1) ^ 1, P.wait_budget)) {
          if (lane == 0) atomicOr(P.err, ERR_WAIT_FUSE);
          alive = false;
        }
        const float4* bias = reinterpret_cast<const float4*>(&s_bias[b][cg * 32]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 ba = bias[2 * j], bb = bias[2 * j + 1];
          const float* v = mx + 8 * j;
          uint4 o;
          o.x = Store<T>::pack2(relu_f(v[0] + ba.x), relu_f(v[1] + ba.y));
          o.y = Store<T>::pack2(relu_f(v[2] + ba.z), relu_f(v[3] + ba.w));
          o.z = Store<T>::pack2(relu_f(v[4] + bb.x), relu_f(v[5] + bb.y));
          o.w = Store<T>::pack2(relu_f(v[6] + bb.z), relu_f(v[7] + bb.w));
          *reinterpret_cast<uint4*>(frow + ((((cg & 1) * 4 + j) ^ (row & 7)) << 4)) = o;
        }
        fence_async_smem();                    // generic writes -> the MMA
        __syncwarp();
        if (lane == 0) mbar_arrive(fready);
      }
    }
  } else if (warp < kProdWarp0) {
    // ---------------- head epilogue ----------------
    const int qd = warp & 3;
    const int row = qd * 32 + lane;
    const int ry = row / P.tw, rx = row - ry * P.tw;
    float hb[kFuseHeadOut];
#pragma unroll
    for (int o = 0; o < kFuseHeadOut; ++o) hb[o] = P.head_b[o];
    bool alive = true;
    uint32_t ph = 0;
    for (int t = lo; t < hi; ++t) {
      const int n = t - lo, acc = n & 1;
      const NhItem I = item_at(P, t);
      if (ATTN && warp == kHeadWarp0) {
        // store the item's fused chunk pairs (its boxes start inside the map;
        // what lies beyond the map is not written)
        for (int b = 0; b < nb; ++b, ++ph) {
          if (alive && !mbar_wait_warp(fready, ph & 1, P.wait_budget)) {
            if (lane == 0) atomicOr(P.err, ERR_WAIT_FUSE);
            alive = false;
          }
          if (lane == 0) {
            if (alive) {
#pragma unroll
              for (int q = 0; q < 2; ++q)
                tma_store_5d(&P.fused, fsm + q * kChunk, b * kUp + q * 64, I.sx, I.x0, I.sy, I.y0);
              bulk_commit();
              bulk_wait_read_all();
            }
            mbar_arrive(fempty);
          }
          __syncwarp();
        }
      }
      if (alive && !mbar_wait(&hfull[acc], (n >> 1) & 1, P.wait_budget)) {
        if (lane == 0) atomicOr(P.err, ERR_WAIT_FUSE);
        alive = false;
      }
      tc_fence_after();
      float v[16];
      tmem_ld16(tmem + kHeadCol + acc * kFuseHeadOut + (static_cast<uint32_t>(qd * 32) << 16), v);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&hempty[acc]);
      const int qx = I.x0 + rx, qy = I.y0 + ry;
      const bool cv = ry < P.th && qx < P.Wq && qy < P.Hq;
      const int cell = (qy * P.S + I.sy) * P.Wf + qx * P.S + I.sx;
#pragma unroll
      for (int o = 0; o < kFuseHeadOut; ++o) v[o] += hb[o];
      if (cv) {
        float4* ho = reinterpret_cast<float4*>(P.head_out + (size_t)cell * kFuseHeadOut);
#pragma unroll
        for (int q = 0; q < 4; ++q) ho[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      }
#pragma unroll
      for (int o = 0; o < kFuseHeadOut; ++o) {
        if (o < P.anchors) {
          const bool keep = cv && v[o] >= P.cls_thresh;
          const uint32_t key = keep ? ord_desc(v[o]) : 0xFFFFFFFFu;
          if (cv) P.keys[(size_t)cell * P.anchors + o] = key;
          hist_add(P.hist0, keep, key, lane);
        }
      }
    }
    if (ATTN && warp == kHeadWarp0 && lane == 0) bulk_wait_all();
  } else if (warp < kMmaWarp) {
    // ---------------- TMA producers (one thread in each of kProducers warps) ----------------
    if (lane == 0 && lo < hi) {
      const uint32_t bytes = (uint32_t)(P.tw * P.th * 128);
      uint32_t it = 0, loads = 1, mine = 0;    // weight loads so far; this thread's last stage + 1
      int cur = item_at(P, lo).sub;
      bool alive = true;
      for (int t = lo; t < hi && alive; ++t) {
        const NhItem I = item_at(P, t);
        if (I.sub != cur) {
          // the MMAs that read the previous position's weights are done
          if (!mbar_wait(wempty, (loads - 1) & 1, P.wait_budget)) {
            alive = false;
            break;
          }
          load_weights(I, pid);
          ++loads;
          cur = I.sub;
        }
        for (int pb = 0; pb < kPasses * nb && alive; ++pb) {
          const int b = pb < nb ? pb : pb - nb;
          const int ox = I.sx / P.s[b], oy = I.sy / P.s[b];
          const int nc = P.cin[b] / 64;
          for (int k = 0; k < Kp && alive; ++k) {
            const int agent = s_list[k];
            for (int c = 0; c < nc; ++c, ++it) {
              if ((int)(it % kProducers) != pid) continue;
              const uint32_t s = it % kStages;
              if (!mbar_wait(&empty[s], ((it / kStages) & 1) ^ 1, P.wait_budget)) {
                alive = false;
                break;
              }
              mbar_arrive_expect_tx(&full[s], bytes);
              tma_load_5d(smem + s * kChunk, &P.in[b], &full[s], ox * P.cin[b] + c * 64, I.x0, oy, I.y0, agent);
              mine = it + 1;
            }
          }
        }
      }
      if (!alive) {
        atomicOr(P.err, ERR_WAIT_FUSE);
        // this thread's last box may still be in flight into the CTA's memory
        if (mine > 0)
          (void)mbar_wait(&full[(mine - 1) % kStages], ((mine - 1) / kStages) & 1, P.wait_budget);
        (void)mbar_wait(wfull, (loads - 1) & 1, P.wait_budget);
      }
    }
  } else if (lo < hi) {
    // ---------------- MMA issuer (the whole warp, one elected lane issuing) ----------------
    // The MMA's descriptors have to be in uniform registers: issued from a
    // branch that one lane takes, each of a chunk's 4 MMAs cost about 150
    // clocks (64 in the pipe).  So the warp stays converged -- waits end with
    // a vote -- and only the issue itself is predicated: 8 agents on the
    // 352 x 100 map 53.6 -> 40.9 us.
    const uint32_t idesc = idesc_f16(kTile, kUp, std::is_same<T, __nv_bfloat16>::value);
    const uint32_t hdesc = idesc_f16(kTile, kFuseHeadOut, std::is_same<T, __nv_bfloat16>::value);
    const uint64_t d0 = smem_desc(smem_u32(smem), 1024, 2);
    const uint32_t lo0 = (uint32_t)d0, hi0 = (uint32_t)(d0 >> 32);   // operands differ in the address only
    const long long budget = P.wait_budget;
    const bool leader = elect_one();
    uint32_t it = 0, st = 0, loads = 0, ph = 0;
    int cur = -1;
    bool alive = mbar_wait_warp(hwfull, 0, budget);
    // Head MMAs of a finished block (phase pph): issued after the next step's
    // MMAs, which keep the pipe busy while the epilogue writes the fused chunk.
    bool pend = false;
    int pb = 0, pn = 0;
    uint32_t pph = 0;
    auto flush = [&]() {
      pend = false;
      if (!mbar_wait_warp(fready, pph & 1, budget) ||
          (pb == 0 && !mbar_wait_warp(&hempty[pn & 1], ((pn >> 1) & 1) ^ 1, budget))) {
        alive = false;
        return;
      }
      tc_fence_after();
      const uint32_t d = tmem + kHeadCol + (pn & 1) * kFuseHeadOut;
      if (leader) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
          mma_kblock(d, lo0 + ((kFOff + q * kChunk) >> 4), hi0,
                     lo0 + ((kHOff + (pb * 2 + q) * kHeadChunk) >> 4), hi0, hdesc, (pb > 0 || q > 0) ? 1u : 0u,
                     true);
        umma_commit(fempty);
        if (pb == nb - 1) umma_commit(&hfull[pn & 1]);
      }
      __syncwarp();
    };
    for (int t = lo; t < hi && alive; ++t) {
      const int sub = t / P.tiles;
      if (sub != cur) {
        if (cur >= 0 && leader) umma_commit(wempty);
        alive = mbar_wait_warp(wfull, loads & 1, budget);
        ++loads;
        cur = sub;
      }
      uint32_t w_lo = 0;                       // block b's first weight chunk
      for (int ps = 0; ps < kPasses * nb && alive; ++ps) {
        const int b = ps < nb ? ps : ps - nb;
        const bool head = ps >= (kPasses - 1) * nb;   // the pass whose sums the head reads
        if (b == 0) w_lo = lo0 + (kWOff >> 4);
        const int nc = P.cin[b] / 64;
        for (int k = 0; k < Kp && alive; ++k, ++st) {
          const uint32_t buf = st % kAccs;
          alive = mbar_wait_warp(&accempty[buf], ((st / kAccs) & 1) ^ 1, budget);
          const uint32_t d = tmem + buf * kUp;
          for (int c = 0; c < nc && alive; ++c, ++it) {
            const uint32_t s = it % kStages;
            alive = mbar_wait_warp(&full[s], (it / kStages) & 1, budget);
            if (!alive) break;
            tc_fence_after();
            if (leader) {
              mma_kblock(d, lo0 + s * (kChunk >> 4), hi0, w_lo + c * (kChunk >> 4), hi0, idesc, c > 0 ? 1u : 0u,
                         true);
              umma_commit(&empty[s]);
              if (c == nc - 1) umma_commit(&accfull[buf]);
            }
            __syncwarp();
          }
          if (pend && alive) flush();
        }
        if (pend && alive) flush();            // no agent present
        if (head) {
          pend = true;
          pb = b;
          pn = t - lo;
          pph = ph++;
        }
        w_lo += nc * (kChunk >> 4);
      }
    }
    if (pend && alive) flush();
    if (!alive && lane == 0) atomicOr(P.err, ERR_WAIT_FUSE);
  }

  tc_fence_before();
  __syncthreads();
  span_end(P.span);
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace

bool neck_head_ok(int n_blocks, const int* cin, const int* stride, int up_ch) {
  if (n_blocks < 1 || n_blocks > RTCC_MAX_BLOCKS || up_ch != kUp) return false;
  int chunks = 0, S = 1;
  for (int b = 0; b < n_blocks; ++b) {
    if (cin[b] < 64 || cin[b] % 64) return false;
    if (stride[b] != 1 && stride[b] != 2 && stride[b] != 4) return false;
    chunks += cin[b] / 64;
    S = std::max(S, stride[b]);
  }
  return chunks <= kMaxChunks;
}

// The tw x th rectangle of at most 128 pixels that covers W x H with the
// fewest tiles (the widest of those).
void neck_head_tile(int W, int H, int* tw, int* th) {
  long long best = -1;
  for (int w = 1; w <= kTile && w <= W; ++w) {
    const int h = std::min(kTile / w, H);
    const long long n = (long long)((W + w - 1) / w) * ((H + h - 1) / h);
    if (best < 0 || n <= best) {
      best = n;
      *tw = w;
      *th = h;
    }
  }
}

cudaError_t neck_head_fill(const NeckHeadArgs& a, bool bf16, NeckHeadParams* P) {
  if (!neck_head_ok(a.n_blocks, a.cin, a.stride, kUp) || a.K < 1 || a.K > RTCC_MAX_AGENTS ||
      a.anchors < 1 || a.anchors > kFuseHeadOut || a.wait_budget < 1 || (a.attention && !a.fused))
    return cudaErrorInvalidValue;
  std::memset(P, 0, sizeof(*P));
  int S = 1;
  for (int b = 0; b < a.n_blocks; ++b) S = std::max(S, a.stride[b]);
  if (a.feat_w < S || a.feat_h < S || a.feat_w % S || a.feat_h % S) return cudaErrorInvalidValue;
  P->n_blocks = a.n_blocks;
  P->S = S;
  P->Wf = a.feat_w;
  P->Wq = a.feat_w / S;
  P->Hq = a.feat_h / S;
  neck_head_tile(P->Wq, P->Hq, &P->tw, &P->th);
  P->tiles_x = (P->Wq + P->tw - 1) / P->tw;
  P->tiles = P->tiles_x * ((P->Hq + P->th - 1) / P->th);
  for (int b = 0; b < a.n_blocks; ++b) {
    const int s = a.stride[b], r = S / s;
    const uint64_t C = (uint64_t)a.cin[b], W = (uint64_t)(a.feat_w / s), H = (uint64_t)(a.feat_h / s);
    if (a.astride[b] < (long long)(C * W * H) || (a.astride[b] * 2) % 16) return cudaErrorInvalidValue;
    P->cin[b] = a.cin[b];
    P->s[b] = s;
    P->bias[b] = a.bias[b];
    const uint64_t dims[5] = {(uint64_t)r * C, W / r, (uint64_t)r, H / r, (uint64_t)a.K};
    const uint64_t strides[4] = {(uint64_t)r * C * 2, W * C * 2, (uint64_t)r * W * C * 2,
                                 (uint64_t)a.astride[b] * 2};
    const uint32_t box[5] = {64, (uint32_t)P->tw, 1, (uint32_t)P->th, 1};
    cudaError_t e = tmap_nd(&P->in[b], a.in[b], bf16, 5, dims, strides, box, 128);
    if (e != cudaSuccess) return e;
    e = tmap_2d(&P->w[b], a.w[b], bf16, C, (uint64_t)(s * s * kUp), 64, kUp, 128);
    if (e != cudaSuccess) return e;
  }
  const uint64_t Cf = (uint64_t)(a.n_blocks * kUp), W = (uint64_t)a.feat_w, s64 = (uint64_t)S;
  cudaError_t e = tmap_2d(&P->wh, a.head_w, bf16, Cf, kFuseHeadOut, 64, kFuseHeadOut, 128);
  if (e != cudaSuccess) return e;
  if (a.attention) {
    const uint64_t dims[5] = {Cf, s64, W / s64, s64, (uint64_t)a.feat_h / s64};
    const uint64_t strides[4] = {Cf * 2, s64 * Cf * 2, W * Cf * 2, s64 * W * Cf * 2};
    const uint32_t box[5] = {64, 1, (uint32_t)P->tw, 1, (uint32_t)P->th};
    e = tmap_nd(&P->fused, a.fused, bf16, 5, dims, strides, box, 128);
    if (e != cudaSuccess) return e;
  }
  P->K = a.K;
  P->attention = a.attention;
  P->inv_sqrt_c = 1.0f / sqrtf((float)(a.n_blocks * kUp));
  P->present = a.present;
  P->head_b = a.head_b;
  P->head_out = a.head_out;
  P->keys = a.keys;
  P->hist0 = a.hist0;
  P->cls_thresh = a.cls_thresh;
  P->anchors = a.anchors;
  P->err = a.err;
  P->span = a.span;
  P->wait_budget = a.wait_budget;
  return cudaSuccess;
}

cudaError_t launch_neck_head(const NeckHeadParams& p, bool bf16, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // equal ranges: as many CTAs as keep the longest range at its minimum
  const int items = p.S * p.S * p.tiles;
  if (items < 1 || sms < 1) return cudaErrorInvalidValue;
  const int rounds = (items + sms - 1) / sms;
  const int grid = (items + rounds - 1) / rounds;
  auto kern = p.attention ? (bf16 ? k_neck_head<__nv_bfloat16, true> : k_neck_head<__half, true>)
                          : (bf16 ? k_neck_head<__nv_bfloat16, false> : k_neck_head<__half, false>);
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(grid), dim3(threads(p.attention != 0)), kSmem, st, p);
}

}  // namespace rtcc
