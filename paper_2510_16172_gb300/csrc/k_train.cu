// k_train.cu -- forward pass, loss and back-propagation of a training batch in one launch (tcgen05, CTA pairs).
//
// Run layer by layer, a batch of 8192 rows took 19 dependent launches a step, 64 CTAs each on 152 SMs, and
// every hidden layer wrote its activations, their transpose and the FP32 GELU derivative to HBM and read
// them back (15 KB per sample): 165 us a step for 7 GFLOP.  Here a cluster of two CTAs takes a tile of 128
// rows through all layers and back.  Each CTA computes half of every hidden layer's outputs (M = 128, N = 128
// MMAs), so the epilogues, which cost more than the MMAs, are spread over twice the SMs; it stores its
// half of the BF16 activations into both CTAs' shared memory, where the next layer reads all of them.  The
// derivatives stay in TMEM, in FP32, in place of the accumulators they came from: three 128-column regions
// for the hidden layers, one for the output layer and the first back-propagated accumulator; each further
// one takes the region whose derivative was used last.  What leaves the chip is what the weight gradients
// read: the transposed activations and layer gradients (3 KB per sample), and the bias gradients' column
// sums, kept per CTA until its last tile.
//
// Shared memory (220 KB, one CTA per SM): the CTA's halves of W1, W4 and W4^T for the whole launch; two 64 KB
// buffers for W2 then W3^T, and W3 then W2^T, refilled while other layers run; 64 KB of activations.
// The chain per tile is serial: seven MMA groups, each followed by its epilogue.  Waits are bounded as in
// k_infer.cu.
#include <cuda_bf16.h>

#include "fpt_kernels.h"
#include "mlp.h"
#include "mlp_device.cuh"
#include "tc.cuh"

namespace fpt {

constexpr int kTrainEpiWarps = 16;   // four per 32-lane quarter of TMEM, 32 of the CTA's 128 columns each
constexpr int kTrainLoadWarps = 4;   // one thread per row
constexpr int kTrainThreads = 32 * (kTrainEpiWarps + kTrainLoadWarps + 1);
constexpr uint32_t kW4tBytes = 128 * kMlpOut * 2;

struct TrainSmem {
  unsigned char buf[2][4 * kMlpChunk];  // W2 / W3^T, W3 / W2^T (this CTA's 128 rows of B, 64-column chunks)
  unsigned char act[4 * kMlpChunk];     // the tile's activations (A); chunk 0 also its features and its dY
  unsigned char w1[kMlpChunk];
  unsigned char w4[4 * kMlpW4Chunk];
  unsigned char w4t[kW4tBytes];
  float bias[3 * 128 + kMlpOut];        // this CTA's outputs
  float col[3 * 128 + kMlpOut];         // column sums of the layer gradients
  uint64_t src[128];                    // the rows' samples
  uint64_t fixed, full[2];              // weight copies
  uint64_t rows;                        // the tile's features are in act
  uint64_t act_full;                    // both CTAs' halves of the activations are written
  uint64_t dy;                          // dY is written
  uint64_t tile;                        // the epilogues have read the tile's last accumulator
  uint64_t layer;                       // an MMA group of both CTAs is done
  uint64_t act_free;                    // the tile's last MMA group of this CTA has read act
  uint64_t drain;
  uint32_t tmem;
  int fail;
};
static_assert(sizeof(TrainSmem) <= 227 * 1024, "one CTA per SM");

// Rows of A^T (bf16, [columns][ld]) from a thread's 16 consecutive columns of its row.
__device__ __forceinline__ void store_transposed(__nv_bfloat16* dst, uint64_t ld, const uint32_t (&w)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const __nv_bfloat162 p = *reinterpret_cast<const __nv_bfloat162*>(&w[i]);
    dst[(uint64_t)(2 * i) * ld] = p.x;
    dst[(uint64_t)(2 * i + 1) * ld] = p.y;
  }
}

// The 64 features of sample src as 16-byte words.
__device__ __forceinline__ void load_features(const TrainArgs& a, uint64_t src, uint4 (&f)[kMlpIn / 8]) {
  const __nv_bfloat16* x = a.X + src * kMlpIn;
  if (a.vec_x) {
#pragma unroll
    for (int k = 0; k < kMlpIn / 8; ++k) f[k] = __ldg(reinterpret_cast<const uint4*>(x) + k);
  } else {
    const unsigned short* u = reinterpret_cast<const unsigned short*>(x);
#pragma unroll
    for (int k = 0; k < kMlpIn / 8; ++k) {
      uint32_t w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i] = (uint32_t)u[8 * k + 2 * i] | ((uint32_t)u[8 * k + 2 * i + 1] << 16);
      f[k] = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// Targets t[0..7] and Gram entries t[8..19] of sample src.
__device__ __forceinline__ void load_targets(const TrainArgs& a, uint64_t src, float (&t)[20]) {
  const float *T = a.T + src * 8, *G = a.G + src * 12;
  if (a.vec_tg) {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const float4 v = k < 2 ? __ldg(reinterpret_cast<const float4*>(T) + k) : __ldg(reinterpret_cast<const float4*>(G) + (k - 2));
      t[4 * k] = v.x;
      t[4 * k + 1] = v.y;
      t[4 * k + 2] = v.z;
      t[4 * k + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 20; ++k) t[k] = k < 8 ? T[k] : G[k - 8];
  }
}

// Gram-weighted loss sum_s d_s^T G_s d_s of a sample, d = y[:8] - t, and its gradient g = w G d (the padded
// outputs keep theirs); G_s = A_s^T A_s / S^2 per slot, zero for unused slots.
__device__ __forceinline__ float row_loss(const float* t, const float* gm, const float (&y)[16], float w,
                                          float (&g)[16]) {
  float acc = 0.f;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const float g11 = gm[3 * s], g12 = gm[3 * s + 1], g22 = gm[3 * s + 2];
    const float d0 = y[2 * s] - t[2 * s];
    const float d1 = y[2 * s + 1] - t[2 * s + 1];
    const float m0 = g11 * d0 + g12 * d1, m1 = g12 * d0 + g22 * d1;
    acc += d0 * m0 + d1 * m1;
    g[2 * s] = w * m0;
    g[2 * s + 1] = w * m1;
  }
  return acc;
}

__device__ __forceinline__ void pack_bf16(const float (&x)[16], uint32_t (&w)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(x[2 * i], x[2 * i + 1]);
    w[i] = *reinterpret_cast<const uint32_t*>(&p);
  }
}

__device__ __forceinline__ bool train_warp_wait(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, tc::mbar_wait_cluster(bar, parity, kWaitNs));
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTrainThreads, 1) mlp_train_kernel(TrainArgs a) {
  extern __shared__ __align__(1024) unsigned char train_smem[];
  TrainSmem& sm = *reinterpret_cast<TrainSmem*>(train_smem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = tc::cluster_rank();
  const uint64_t n_clusters = gridDim.x >> 1, cluster = blockIdx.x >> 1;
  const uint64_t n_tiles = (a.B + 127) / 128;
  const uint64_t my_tiles = cluster < n_tiles ? (n_tiles - cluster + n_clusters - 1) / n_clusters : 0;
  const unsigned char* wf = reinterpret_cast<const unsigned char*>(a.wt) + rank * kMlpHalfBytes;
  const unsigned char* wb = reinterpret_cast<const unsigned char*>(a.wtT) + rank * kMlpHalfTBytes;
  // buffer b's contents by turns: W2 / W3^T in buffer 0, W3 / W2^T in buffer 1
  auto fill = [&](int b, bool back) {
    const unsigned char* s = back ? wb + (b == 0 ? kMlpTileW3t : kMlpTileW2t) : wf + (b == 0 ? kMlpTileW2 : kMlpTileW3);
    tc::mbar_expect_tx(&sm.full[b], 4 * kMlpChunk);
    for (uint32_t o = 0; o < 4 * kMlpChunk; o += kMlpChunk) tc::bulk_g2s(sm.buf[b] + o, s + o, kMlpChunk, &sm.full[b]);
  };
  if (tid == 0) {
    tc::mbar_init(&sm.fixed, 1);
    tc::mbar_init(&sm.full[0], 1);
    tc::mbar_init(&sm.full[1], 1);
    tc::mbar_init(&sm.rows, kTrainLoadWarps);
    tc::mbar_init(&sm.act_full, 2 * kTrainEpiWarps);
    tc::mbar_init(&sm.dy, kTrainEpiWarps);
    tc::mbar_init(&sm.tile, kTrainEpiWarps);
    tc::mbar_init(&sm.layer, 2);
    tc::mbar_init(&sm.act_free, 1);
    tc::mbar_init(&sm.drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sm.fail = 0;
    tc::mbar_expect_tx(&sm.fixed, kMlpChunk + 4 * kMlpW4Chunk + kW4tBytes);
    tc::bulk_g2s(sm.w1, wf, kMlpChunk, &sm.fixed);
    tc::bulk_g2s(sm.w4, wf + kMlpTileW4, 4 * kMlpW4Chunk, &sm.fixed);
    tc::bulk_g2s(sm.w4t, wb + kMlpTileW4t, kW4tBytes, &sm.fixed);
    fill(0, false);
    fill(1, false);
  }
  for (int i = tid; i < 3 * 128; i += blockDim.x) {
    const int off = i < 128 ? kOffB1 : (i < 256 ? kOffB2 : kOffB3);
    sm.bias[i] = a.params[off + (int)rank * 128 + (i & 127)];
  }
  if (tid < kMlpOut) sm.bias[384 + tid] = a.params[kOffB4 + tid];
  for (int i = tid; i < 3 * 128 + kMlpOut; i += blockDim.x) sm.col[i] = 0.f;
  __syncwarp();
  if (warp == 0) {
    tc::tmem_alloc(&sm.tmem, 512);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::cluster_sync();  // the peer's barriers are initialised before anything arrives on them
  tc::fence_after_sync();
  const uint32_t tmem = sm.tmem;

  if (warp < kTrainEpiWarps) {
    // ---- epilogues ----
    const int q = warp & 3, jc = warp >> 2;  // TMEM lane quarter; which 32 of the CTA's 128 columns
    const int row = q * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    // this warp's 32 columns of the activations: chunk and the column within it
    const uint32_t act_off = (2u * rank + (uint32_t)(jc >> 1)) * kMlpChunk;
    unsigned char* act_own = sm.act + act_off;
    const uint32_t act_peer = tc::map_rank(sm.act, rank ^ 1u) + act_off;
    uint32_t ph_layer = 0u;
    float loss = 0.f;
    bool ok = true;
    auto layer_wait = [&]() {
      ok = train_warp_wait(&sm.layer, ph_layer);
      ph_layer ^= 1u;
      tc::fence_after_sync();
      return ok;
    };
    // 16 columns (step s) of the half-layer into both CTAs' activations
    auto put_act = [&](int s, const uint32_t (&w)[8]) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint4 v = make_uint4(w[4 * h], w[4 * h + 1], w[4 * h + 2], w[4 * h + 3]);
        const uint32_t o = tc::sw128_offset(row, (jc & 1) * 32 + 16 * s + 8 * h);
        *reinterpret_cast<uint4*>(act_own + o) = v;
        tc::st_cluster(act_peer + o, v);
      }
    };
    auto act_done = [&]() {
      tc::fence_async_all();
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) {
        tc::mbar_arrive(&sm.act_full);
        tc::mbar_arrive_rank(&sm.act_full, rank ^ 1u);
      }
    };
    for (uint64_t ti = 0; ti < my_tiles && ok; ++ti) {
      const uint64_t b = (cluster + ti * n_clusters) * 128 + row;
      const bool live = b < a.B;
      const int c0 = (int)rank * 128 + jc * 32;  // this warp's first output
#pragma unroll 1
      for (int l = 0; l < 3 && ok; ++l) {  // hidden layers: activation, its transpose, the derivative
        if (!layer_wait()) break;
        const uint32_t acc = lane_addr + (uint32_t)(l * 128 + jc * 32);
        __nv_bfloat16* ht = a.Ht + ((uint64_t)l * kMlpHidden + c0) * a.B + b;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          float z[16], d[16];
          tc::tmem_ld16(acc + 16u * s, z);
          const float* bias = sm.bias + l * 128 + jc * 32 + s * 16;
#pragma unroll
          for (int i = 0; i < 16; ++i) z[i] = gelu_with_grad(z[i] + bias[i], d[i]);
          tc::tmem_st16(acc + 16u * s, d);
          uint32_t w[8];
          pack_bf16(z, w);
          put_act(s, w);
          if (live) store_transposed(ht + (uint64_t)(16 * s) * a.B, a.B, w);
        }
        act_done();
      }
      if (!ok) break;
      // output layer: loss and dY, a thread per row (both CTAs compute them, the first keeps the sums)
      float tg[20];
      if (jc == 0) {
        ok = train_warp_wait(&sm.rows, (uint32_t)(ti & 1));
        if (live && ok) load_targets(a, sm.src[row], tg);
      }
      ok = __all_sync(0xffffffffu, ok) && layer_wait();
      if (!ok) break;
      if (jc == 0) {
        float y[16], g[16];
        tc::tmem_ld16(lane_addr + 384u, y);
#pragma unroll
        for (int i = 0; i < 16; ++i) g[i] = 0.f;
        if (live) {
#pragma unroll
          for (int i = 0; i < 8; ++i) y[i] += sm.bias[384 + i];
          loss += row_loss(tg, tg + 8, y, 2.f / (float)a.B, g);
        }
        uint32_t w[8];
        pack_bf16(g, w);
        *reinterpret_cast<uint4*>(sm.act + tc::kmajor_offset(row, 0, 16)) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(sm.act + tc::kmajor_offset(row, 8, 16)) = make_uint4(w[4], w[5], w[6], w[7]);
        if (rank == 0) {
          if (live) store_transposed(a.dYt + b, a.B, w);
          const float v = warp_colsum16(g, lane);
          if (!(lane & 1)) atomicAdd(&sm.col[384 + warp_colsum16_column(lane)], v);
        }
        tc::fence_async_smem();
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sm.dy);
#pragma unroll 1
      for (int l = 2; l >= 0 && ok; --l) {  // layer gradients: the accumulator times the derivative in TMEM
        if (!layer_wait()) break;
        const uint32_t acc = lane_addr + (uint32_t)((l + 1) * 128 + jc * 32);
        __nv_bfloat16* zt = a.dZt + ((uint64_t)l * kMlpHidden + c0) * a.B + b;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          float x[16], d[16];
          tc::tmem_ld16(acc + 16u * s, x);
          tc::tmem_ld16(acc - 128u + 16u * s, d);
#pragma unroll
          for (int i = 0; i < 16; ++i) x[i] *= d[i];
          uint32_t w[8];
          pack_bf16(x, w);
          if (l > 0) put_act(s, w);
          if (live) store_transposed(zt + (uint64_t)(16 * s) * a.B, a.B, w);
          const float v = warp_colsum16(x, lane);
          if (!(lane & 1)) atomicAdd(&sm.col[l * 128 + jc * 32 + s * 16 + warp_colsum16_column(lane)], v);
        }
        if (l > 0) {
          act_done();
        } else {
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&sm.tile);
        }
      }
    }
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (jc == 0 && rank == 0 && lane == 0) atomicAdd(a.loss, loss / (float)a.B);
    if (!ok) sm.fail = 1;
  } else if (warp < kTrainEpiWarps + kTrainLoadWarps) {
    // ---- the tile's rows: sample numbers, features, their transpose ----
    const int row = tid - 32 * kTrainEpiWarps;
    bool ok = true;
    for (uint64_t ti = 0; ti < my_tiles; ++ti) {
      const uint64_t b = (cluster + ti * n_clusters) * 128 + row;
      uint4 f[kMlpIn / 8];
      uint64_t src = 0;
#pragma unroll
      for (int k = 0; k < kMlpIn / 8; ++k) f[k] = make_uint4(0u, 0u, 0u, 0u);
      if (b < a.B) {
        src = a.n ? perm_index(a.first + b, a.n, a.h, a.key) : b;
        load_features(a, src, f);
      }
      if (ti > 0 && !train_warp_wait(&sm.act_free, (uint32_t)(ti - 1) & 1u)) {
        ok = false;
        break;
      }
#pragma unroll
      for (int k = 0; k < kMlpIn / 8; ++k)
        *reinterpret_cast<uint4*>(sm.act + tc::sw128_offset(row, k * 8)) = f[k];
      sm.src[row] = src;
      tc::fence_async_smem();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sm.rows);
      if (b < a.B) {  // each CTA writes half of the features' transpose
        const __nv_bfloat16* e = reinterpret_cast<const __nv_bfloat16*>(f);
        if (rank == 0) {
#pragma unroll
          for (int k = 0; k < kMlpIn / 2; ++k) a.Xt[(uint64_t)k * a.B + b] = e[k];
        } else {
#pragma unroll
          for (int k = kMlpIn / 2; k < kMlpIn; ++k) a.Xt[(uint64_t)k * a.B + b] = e[k];
        }
      }
    }
    // the last tile's arrival too, so that none is on its way to a CTA that has left
    if (ok && my_tiles > 0) ok = train_warp_wait(&sm.act_free, (uint32_t)(my_tiles - 1) & 1u);
    if (!ok) sm.fail = 1;
  } else {
    if (lane == 0) {
      // ---- copies and MMAs ----
      bool ok = tc::mbar_wait(&sm.fixed, 0u, kWaitNs);
      const uint32_t act = tc::smem_u32(sm.act);
      constexpr uint32_t id128 = tc::idesc_bf16(128, 128), id16 = tc::idesc_bf16(128, kMlpOut);
      uint32_t ph_act = 0u, n_fill[2] = {1u, 1u}, n_full[2] = {0u, 0u};
      // one 64-column chunk: four K = 16 steps
      auto chunk = [&](uint32_t d, uint32_t x, uint32_t w, uint32_t idesc, bool fresh) {
        const uint64_t ad = tc::smem_desc_sw128(x), bd = tc::smem_desc_sw128(w);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) tc::mma_bf16(d, ad + 2u * kk, bd + 2u * kk, idesc, fresh && kk == 0 ? 0u : 1u);
      };
      auto act_wait = [&]() {
        ok = ok && tc::mbar_wait_cluster(&sm.act_full, ph_act, kWaitNs);
        ph_act ^= 1u;
        tc::fence_async_all();
        tc::fence_after_sync();
        return ok;
      };
      // a layer from the activations and weight buffer b
      auto buffered = [&](int b, uint32_t d) {
        ok = ok && tc::mbar_wait(&sm.full[b], n_full[b] & 1u, kWaitNs);
        ++n_full[b];
        if (!ok) return;
        const uint32_t w = tc::smem_u32(sm.buf[b]);
        for (int c = 0; c < 4; ++c) chunk(d, act + c * kMlpChunk, w + c * kMlpChunk, id128, c == 0);
        tc::mma_commit_both(&sm.layer);
      };
      auto refill = [&](int b, bool back) {
        fill(b, back);
        ++n_fill[b];
      };
      for (uint64_t ti = 0; ti < my_tiles && ok; ++ti) {
        const bool more = ti + 1 < my_tiles;
        if (!(ok = tc::mbar_wait(&sm.rows, (uint32_t)(ti & 1), kWaitNs))) break;
        if (ti > 0) {
          if (!(ok = tc::mbar_wait(&sm.tile, (uint32_t)(ti - 1) & 1u, kWaitNs))) break;
          refill(1, false);  // the last tile's W2^T has been read (its epilogue is done)
        }
        tc::fence_after_sync();
        chunk(tmem, act, tc::smem_u32(sm.w1), id128, true);
        tc::mma_commit_both(&sm.layer);
        if (!act_wait()) break;
        buffered(0, tmem + 128u);
        if (!act_wait()) break;
        refill(0, true);  // the epilogue behind this wait waited for layer 2's MMAs: W2 has been read
        buffered(1, tmem + 256u);
        if (!act_wait()) break;
        refill(1, true);
        for (int c = 0; c < 4; ++c)
          chunk(tmem + 384u, act + c * kMlpChunk, tc::smem_u32(sm.w4) + c * kMlpW4Chunk, id16, c == 0);
        tc::mma_commit_both(&sm.layer);
        if (!(ok = tc::mbar_wait(&sm.dy, (uint32_t)(ti & 1), kWaitNs))) break;
        tc::fence_after_sync();
        tc::mma_bf16(tmem + 384u, tc::smem_desc(act, 128u, 256u), tc::smem_desc(tc::smem_u32(sm.w4t), 128u, 256u), id128,
                     0u);
        tc::mma_commit_both(&sm.layer);
        if (!act_wait()) break;
        buffered(0, tmem + 256u);
        if (!act_wait()) break;
        if (more) refill(0, false);
        buffered(1, tmem + 128u);
        if (ok) tc::mma_commit(&sm.act_free);
      }
      if (!ok) {  // let the copies and MMAs in flight finish before the memory goes
        tc::mma_commit(&sm.drain);
        tc::mbar_wait(&sm.drain, 0u, kWaitNs);
        for (int b = 0; b < 2; ++b)
          if (n_full[b] < n_fill[b]) tc::mbar_wait(&sm.full[b], (n_fill[b] - 1u) & 1u, kWaitNs);
        sm.fail = 1;
      }
    }
    __syncwarp();
  }
  tc::fence_before_sync();
  __syncthreads();
  if (tid < 3 * 128) {
    const int off = tid < 128 ? kOffB1 : (tid < 256 ? kOffB2 : kOffB3);
    atomicAdd(a.grad + off + (int)rank * 128 + (tid & 127), sm.col[tid]);
  } else if (rank == 0 && tid < 3 * 128 + kMlpOut) {
    atomicAdd(a.grad + kOffB4 + tid - 3 * 128, sm.col[tid]);
  }
  if (sm.fail && tid == 0 && a.err) atomicCAS(a.err, 0, ERR_MMA_TIMEOUT);
  __syncwarp();
  tc::cluster_sync();  // no store or arrival of the peer reaches a CTA that has left
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

cudaError_t launch_mlp_train(const TrainArgs& args, cudaStream_t stream, int n_sm) {
  TrainArgs a = args;
  if (!a.B) return cudaSuccess;
  auto a16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  a.vec_x = a16(a.X);
  a.vec_tg = a16(a.T) && a16(a.G);
  a.h = 1;
  while ((1ULL << (2 * a.h)) < a.n) ++a.h;
  const int smem = (int)sizeof(TrainSmem);
  cudaError_t e = cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const uint64_t tiles = (a.B + 127) / 128, cap = (uint64_t)(n_sm > 1 ? n_sm / 2 : 1);
  mlp_train_kernel<<<2u * (unsigned)(tiles < cap ? tiles : cap), kTrainThreads, smem, stream>>>(a);
  count_launch();
  return cudaGetLastError();
}

}  // namespace fpt
