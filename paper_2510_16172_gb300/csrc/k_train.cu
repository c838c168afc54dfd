// k_train.cu -- a training step's batch in two launches (tcgen05): forward pass, loss and back-propagation on CTA
// pairs, then the weight gradients.
//
// Run layer by layer, a batch of 8192 rows took 19 dependent launches a step, 64 CTAs each on 152 SMs, and every
// hidden layer wrote its activations, their transpose and the FP32 GELU derivative to HBM and read them back (15 KB
// per sample): 165 us a step for 7 GFLOP.
//
// mlp_train_kernel: a cluster of two CTAs takes a tile of 128 rows through all layers and back.  Each CTA computes half
// of every hidden layer's outputs (M = 128, N = 128 MMAs), so the epilogues, which cost more than the MMAs, are spread
// over twice the SMs.  An epilogue writes its half of the BF16 activations into its own shared memory; from there the
// TMA engine copies it into the peer's, where the next layer reads all of it, and stores it to HBM for the weight
// gradients, while the next layer's MMAs already run on the halves that are there.  (Threads storing to the peer and, two
// bytes at a time, to transposed arrays in HBM took 39 us a batch of 8192; this takes 25.4.)  The derivatives stay in TMEM, in FP32, in place of
// the accumulators they came from: three 128-column regions for the hidden layers, one for the output layer and the
// first back-propagated accumulator; each further one takes the region whose derivative was used last.  Bias gradients
// are column sums kept per CTA until its last tile.
// Shared memory (220 KB, one CTA per SM): the CTA's halves of W1, W4 and W4^T for the whole launch; two 64 KB buffers
// for W2 then W3^T, and W3 then W2^T, refilled while other layers run; 64 KB of activations.  The chain per tile is
// serial: seven MMA groups, each followed by its epilogue; that latency bounds it (one tile per pair at 8192 rows).
//
// mlp_wgrad_kernel: all four weight gradients dW = dZ^T act at once, one CTA per item (128 rows of a dW, a slice of the
// batch).  Both operands are read as they were stored, [row][column], as MN-major operands of the MMAs, so nothing is
// transposed; partial products are added by TMA reductions.  10.8 us at 8192 rows (four GEMMs side by side 20): about
// half of it is the start of a CTA and the reductions, the rest 48 KB of loads per 64 rows.
//
// Waits are bounded as in k_infer.cu.
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include "fpt_kernels.h"
#include "mlp.h"
#include "mlp_device.cuh"
#include "tc.cuh"

namespace fpt {

constexpr int kTrainEpiWarps = 16;   // four per 32-lane quarter of TMEM, 16 columns of each of the CTA's two chunks each
constexpr int kTrainLoadWarps = 4;   // one thread per row
constexpr int kTrainThreads = 32 * (kTrainEpiWarps + kTrainLoadWarps + 2);  // + MMAs, + activation copies
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
  uint64_t half[2];                     // the CTA's own chunks of the activations are written,
  uint64_t peer[2];                     // the peer's have arrived,
  uint64_t stored;                      // and its own have been read by their copies to HBM
  uint64_t dy;                          // dY is written
  uint64_t tile;                        // the epilogues have read the tile's last accumulator
  uint64_t layer;                       // an MMA group of both CTAs is done
  uint64_t act_free;                    // the tile's last layer gradient has been read
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

// BF16 GELU of two accumulator values plus bias (returned) and its derivative gelu'(z) = (1 + th) / 2 + (z / 2)
// (1 - th^2) K0 (1 + 3 K1 z^2) in FP32 (d0, d1), from one tanh each, in packed FP32 instructions.
__device__ __forceinline__ uint32_t gelu_grad_pair(float v0, float v1, uint64_t bias, float& d0, float& d1) {
  const uint64_t half = tc::splat2(0.5f), k0 = tc::splat2(kGeluK0);
  const uint64_t z = tc::add2(tc::pack2(__float_as_uint(v0), __float_as_uint(v1)), bias);
  const uint64_t z2 = tc::mul2(z, z), h = tc::mul2(half, z);
  float u0, u1;
  tc::unpack2(tc::mul2(z, tc::fma2(tc::splat2(kGeluK01), z2, k0)), u0, u1);
  const uint64_t th = tc::pack2(__float_as_uint(tanh_approx(u0)), __float_as_uint(tanh_approx(u1)));
  const uint64_t s = tc::fma2(tc::mul2(th, tc::splat2(-1.f)), th, tc::splat2(1.f));  // 1 - th^2
  const uint64_t q = tc::fma2(tc::splat2(3.f * kGeluK1), z2, tc::splat2(1.f));
  tc::unpack2(tc::fma2(tc::mul2(tc::mul2(h, s), k0), q, tc::fma2(half, th, half)), d0, d1);
  float y0, y1;
  tc::unpack2(tc::fma2(h, th, h), y0, y1);
  const __nv_bfloat162 p = __floats2bfloat162_rn(y0, y1);
  return *reinterpret_cast<const uint32_t*>(&p);
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

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTrainThreads, 1)
    mlp_train_kernel(TrainArgs a, const __grid_constant__ CUtensorMap tmH, const __grid_constant__ CUtensorMap tmZ) {
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
    tc::mbar_init(&sm.half[0], kTrainEpiWarps);
    tc::mbar_init(&sm.half[1], kTrainEpiWarps);
    tc::mbar_init(&sm.peer[0], 1);
    tc::mbar_init(&sm.peer[1], 1);
    tc::mbar_init(&sm.stored, 1);
    tc::mbar_init(&sm.dy, kTrainEpiWarps);
    tc::mbar_init(&sm.tile, kTrainEpiWarps);
    tc::mbar_init(&sm.layer, 2);
    tc::mbar_init(&sm.act_free, 1);
    tc::mbar_init(&sm.drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sm.fail = 0;
  }
  for (int i = tid; i < 3 * 128 + kMlpOut; i += blockDim.x) sm.col[i] = 0.f;
  __syncwarp();
  if (warp == 0) {
    tc::tmem_alloc(&sm.tmem, 512);
    tc::tmem_relinquish();
  }
  // loader warps: a row's sample and features; the first tile's on the way while the CTA sets up
  const int load_row = tid - 32 * kTrainEpiWarps;
  uint4 f[kMlpIn / 8];
  uint64_t src = 0;
  auto load_rows = [&](uint64_t ti) {
    const uint64_t b = (cluster + ti * n_clusters) * 128 + load_row;
    src = 0;
#pragma unroll
    for (int k = 0; k < kMlpIn / 8; ++k) f[k] = make_uint4(0u, 0u, 0u, 0u);
    if (b < a.B) {
      src = a.n ? perm_index(a.first + b, a.n, a.h, a.key) : b;
      load_features(a, src, f);
    }
  };
  if (warp >= kTrainEpiWarps && warp < kTrainEpiWarps + kTrainLoadWarps && my_tiles > 0) load_rows(0);
  wait_previous();  // what the last step's Adam wrote, and what its weight gradients read
  // The weight gradients' CTAs set up on SMs this launch leaves idle or has left.  Only after the wait, so that no
  // later link of the chain starts before the last step is complete.
  launch_dependents();
  if (tid == 0) {
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
  tc::fence_before_sync();
  __syncthreads();
  tc::cluster_sync();  // the peer's barriers are initialised before anything arrives on them
  tc::fence_after_sync();
  const uint32_t tmem = sm.tmem;

  if (warp < kTrainEpiWarps) {
    // ---- epilogues ----
    const int q = warp & 3, jc = warp >> 2;  // TMEM lane quarter; which 16 columns of a chunk
    const int row = q * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    unsigned char* const act_own = sm.act + 2u * rank * kMlpChunk;  // the CTA's two chunks of the activations
    uint32_t ph_layer = 0u, ph_stored = 0u;
    bool first_store = true;
    float loss = 0.f;
    bool ok = true;
    auto layer_wait = [&]() {
      ok = train_warp_wait(&sm.layer, ph_layer);
      ph_layer ^= 1u;
      tc::fence_after_sync();
      return ok;
    };
    // the copies of the last activations have read them
    auto stored_wait = [&]() {
      if (!first_store) {
        ok = train_warp_wait(&sm.stored, ph_stored);
        ph_stored ^= 1u;
      }
      first_store = false;
      return ok;
    };
    // 16 columns of chunk s into the CTA's activations, and the chunk handed over: its copies start while the
    // next one is worked on
    auto put_act = [&](int s, const uint32_t (&w)[8]) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
        *reinterpret_cast<uint4*>(act_own + s * kMlpChunk + tc::sw128_offset(row, jc * 16 + 8 * h)) =
            make_uint4(w[4 * h], w[4 * h + 1], w[4 * h + 2], w[4 * h + 3]);
      tc::fence_async_smem();
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sm.half[s]);
    };
    for (uint64_t ti = 0; ti < my_tiles && ok; ++ti) {
      const uint64_t b = (cluster + ti * n_clusters) * 128 + row;
      const bool live = b < a.B;
#pragma unroll 1
      for (int l = 0; l < 3 && ok; ++l) {  // hidden layers: activation and derivative
        if (!layer_wait() || !stored_wait()) break;
        const uint32_t acc = lane_addr + (uint32_t)(l * 128 + jc * 16);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          float z[16], d[16];
          tc::tmem_ld16(acc + 64u * s, z);
          const float* bias = sm.bias + l * 128 + s * 64 + jc * 16;
          uint32_t w[8];
#pragma unroll
          for (int i = 0; i < 8; ++i)
            w[i] = gelu_grad_pair(z[2 * i], z[2 * i + 1], *reinterpret_cast<const uint64_t*>(bias + 2 * i), d[2 * i],
                                  d[2 * i + 1]);
          tc::tmem_st16(acc + 64u * s, d);
          put_act(s, w);
        }
      }
      if (!ok) break;
      // output layer: loss and dY, a thread per row (both CTAs compute them, the first keeps the sums)
      float tg[20];
      if (jc == 0) {
        ok = train_warp_wait(&sm.rows, (uint32_t)(ti & 1));
        if (live && ok) load_targets(a, sm.src[row], tg);
      }
      // (dY goes where the last activations were)
      if (!__all_sync(0xffffffffu, ok) || !layer_wait() || !stored_wait()) {
        ok = false;
        break;
      }
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
          if (live) store_transposed(a.dYt + b, a.ldY, w);
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
        if (!layer_wait() || (l < 2 && !stored_wait())) break;
        const uint32_t acc = lane_addr + (uint32_t)((l + 1) * 128 + jc * 16);
        // both chunks' values leave TMEM before the first chunk is handed over: the next MMAs, which wait for it in either
        // CTA, write the region that held this layer's derivative
        float x[2][16];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          float d[16];
          tc::tmem_ld16(acc + 64u * s, x[s]);
          tc::tmem_ld16(acc - 128u + 64u * s, d);
#pragma unroll
          for (int i = 0; i < 16; ++i) x[s][i] *= d[i];
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          uint32_t w[8];
          pack_bf16(x[s], w);
          put_act(s, w);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const float v = warp_colsum16(x[s], lane);
          if (!(lane & 1)) atomicAdd(&sm.col[l * 128 + s * 64 + jc * 16 + warp_colsum16_column(lane)], v);
        }
        if (l == 0 && lane == 0) tc::mbar_arrive(&sm.tile);
      }
    }
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (jc == 0 && rank == 0 && lane == 0) atomicAdd(a.loss, loss / (float)a.B);
    if (!ok) sm.fail = 1;
  } else if (warp < kTrainEpiWarps + kTrainLoadWarps) {
    // ---- the tile's rows: sample numbers, features ----
    const int row = load_row;
    bool ok = true;
    for (uint64_t ti = 0; ti < my_tiles; ++ti) {
      const uint64_t b = (cluster + ti * n_clusters) * 128 + row;
      if (ti > 0) load_rows(ti);
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
      if (b < a.B) {  // each CTA writes half of the row for the weight gradient
        uint4* xb = reinterpret_cast<uint4*>(a.Xb + b * kMlpIn);
#pragma unroll
        for (int k = 0; k < kMlpIn / 16; ++k) xb[rank * (kMlpIn / 16) + k] = rank == 0 ? f[k] : f[kMlpIn / 16 + k];
      }
    }
    // the last tile's arrival too, so that none is on its way to a CTA that has left
    if (ok && my_tiles > 0) ok = train_warp_wait(&sm.act_free, (uint32_t)(my_tiles - 1) & 1u);
    if (!ok) sm.fail = 1;
  } else if (warp == kTrainEpiWarps + kTrainLoadWarps + 1) {
    if (lane == 0) {
      // ---- copies of the CTA's half of the activations: to the peer for the next layer, to HBM ----
      const uint32_t peer_act = tc::map_rank(sm.act, rank ^ 1u), peer_bar = tc::map_rank(sm.peer, rank ^ 1u);
      uint32_t ph = 0u;
      bool ok = true;
      for (uint64_t ti = 0; ti < my_tiles && ok; ++ti) {
        const int row0 = (int)((cluster + ti * n_clusters) * 128);
        for (int e = 0; e < 6 && ok; ++e) {  // activations of layers 1-3, layer gradients 3-1 (1 stays)
          for (uint32_t c = 0; c < 2; ++c) {
            if (!(ok = tc::mbar_wait(&sm.half[c], ph, kWaitNs))) break;
            const uint32_t at = 2u * rank + c;
            if (e < 5) tc::bulk_s2s(peer_act + at * kMlpChunk, sm.act + at * kMlpChunk, kMlpChunk, peer_bar + 8u * c);
            tc::tma_store_3d(e < 3 ? &tmH : &tmZ, sm.act + at * kMlpChunk, (int)at * 64, row0, e < 3 ? e : 5 - e);
          }
          ph ^= 1u;
          tc::bulk_commit();
          tc::bulk_wait_read<0>();
          if (!ok) break;
          tc::mbar_arrive(&sm.stored);
          if (e == 5) tc::mbar_arrive(&sm.act_free);
        }
      }
      tc::bulk_wait_all();
      if (!ok) sm.fail = 1;
    }
    __syncwarp();
  } else {
    if (lane == 0) {
      // ---- weight copies and MMAs ----
      bool ok = tc::mbar_wait(&sm.fixed, 0u, kWaitNs);
      const uint32_t act = tc::smem_u32(sm.act);
      constexpr uint32_t id128 = tc::idesc_bf16(128, 128), id16 = tc::idesc_bf16(128, kMlpOut);
      uint32_t ph_half = 0u, ph_peer = 0u, n_fill[2] = {1u, 1u}, n_full[2] = {0u, 0u};
      // one 64-column chunk: four K = 16 steps
      auto chunk = [&](uint32_t d, uint32_t x, uint32_t w, uint32_t idesc, bool fresh) {
        const uint64_t ad = tc::smem_desc_sw128(x), bd = tc::smem_desc_sw128(w);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) tc::mma_bf16(d, ad + 2u * kk, bd + 2u * kk, idesc, fresh && kk == 0 ? 0u : 1u);
      };
      // a layer from the activations and weights of 64-column chunks of w_stride bytes.  Columns in ascending order in
      // both CTAs: the first CTA starts with its own half, the second waits for the first one's.  The second CTA too
      // waits for its own first chunk before its first MMA: in the back-propagation that MMA overwrites the derivatives
      // which this CTA's epilogue has read by the time it hands that chunk over, and the peer's chunk says nothing
      // about them.  (The chunk is there well before the peer's copy.)
      auto layer = [&](uint32_t d, uint32_t w, uint32_t w_stride, uint32_t idesc) {
        for (int c = 0; c < 2; ++c) tc::mbar_expect_tx(&sm.peer[c], kMlpChunk);
        if (!(ok = tc::mbar_wait(&sm.half[0], ph_half, kWaitNs))) return;
        for (uint32_t c = 0; c < 4; ++c) {
          ok = c / 2 == rank ? tc::mbar_wait(&sm.half[c & 1], ph_half, kWaitNs)
                             : tc::mbar_wait_cluster(&sm.peer[c & 1], ph_peer, kWaitNs);
          if (!ok) return;
          tc::fence_after_sync();
          chunk(d, act + c * kMlpChunk, w + c * w_stride, idesc, c == 0);
        }
        ph_half ^= 1u;
        ph_peer ^= 1u;
        tc::mma_commit_both(&sm.layer);
      };
      auto buffered = [&](int b, uint32_t d) {
        ok = ok && tc::mbar_wait(&sm.full[b], n_full[b] & 1u, kWaitNs);
        ++n_full[b];
        if (ok) layer(d, tc::smem_u32(sm.buf[b]), kMlpChunk, id128);
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
        buffered(0, tmem + 128u);
        if (!ok) break;
        buffered(1, tmem + 256u);
        if (!ok) break;
        refill(0, true);  // layer 3 waited for layer 2's epilogue, and so for its MMAs: W2 has been read
        layer(tmem + 384u, tc::smem_u32(sm.w4), kMlpW4Chunk, id16);
        if (!ok) break;
        refill(1, true);
        if (!(ok = tc::mbar_wait(&sm.dy, (uint32_t)(ti & 1), kWaitNs))) break;
        tc::fence_after_sync();
        tc::mma_bf16(tmem + 384u, tc::smem_desc(act, 128u, 256u), tc::smem_desc(tc::smem_u32(sm.w4t), 128u, 256u), id128,
                     0u);
        tc::mma_commit_both(&sm.layer);
        buffered(0, tmem + 256u);
        if (!ok) break;
        buffered(1, tmem + 128u);
        if (!ok) break;
        if (more) refill(0, false);
        ph_half ^= 1u;  // the last layer gradient is only stored; the wait for `tile` covers it
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

// ---- weight gradients --------------------------------------------------------------------------------------
constexpr int kWgStages = 4, kWgEpiWarps = 8, kWgThreads = 32 * (2 + kWgEpiWarps);
constexpr uint32_t kWgBox = 64 * 128;           // 64 rows of the batch x 64 columns (128-byte swizzled)
constexpr uint32_t kWgStage = 6 * kWgBox;       // A: 128 columns; B: up to 256
constexpr uint32_t kWgSmem = kWgStages * kWgStage + 1024;

struct WgradArgs {
  uint64_t B;
  int k_hidden, k_first, k_last;  // batch slices of dW2 and dW3, of dW1, of dW4
  float* grad;
  int* err;
};

// Descriptor of an MN-major operand: boxes of 64 columns (the M or N dimension) x 64 rows (K), 128-byte swizzled;
// the next 64 columns one box further, the next 8 rows 1024 bytes.
__device__ __forceinline__ uint64_t wg_desc_mn(uint32_t saddr) {
  uint64_t d = tc::smem_desc_sw128(saddr);
  d &= ~((uint64_t)0x3FFFu << 16);
  return d | (uint64_t)(kWgBox >> 4) << 16;
}

__global__ void __launch_bounds__(kWgThreads, 1)
    mlp_wgrad_kernel(WgradArgs a, const __grid_constant__ CUtensorMap tmH, const __grid_constant__ CUtensorMap tmZ,
                     const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmY,
                     const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmW2,
                     const __grid_constant__ CUtensorMap tmW3) {
  extern __shared__ unsigned char wg_raw[];
  __shared__ __align__(8) uint64_t full[kWgStages], empty[kWgStages], acc_full;
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* ring = wg_raw + ((1024u - (tc::smem_u32(wg_raw) & 1023u)) & 1023u);
  // this CTA's item: layer gradient `job` (3, 2, 1: dW3, dW2, dW1; 4: dW4), rows m0 .. m0 + 127, slice of the batch
  int job, m0, slice, slices;
  {
    int i = blockIdx.x;
    if (i < 4 * a.k_hidden) {
      slices = a.k_hidden;
      job = i < 2 * slices ? 3 : 2;
      i -= job == 3 ? 0 : 2 * slices;
    } else if (i < 4 * a.k_hidden + 2 * a.k_first) {
      slices = a.k_first;
      job = 1;
      i -= 4 * a.k_hidden;
    } else {
      slices = a.k_last;
      job = 4;
      i -= 4 * a.k_hidden + 2 * a.k_first;
    }
    m0 = i < slices ? 0 : 128;
    slice = i < slices ? i : i - slices;
  }
  const int total = (int)((a.B + 63) / 64), per = (total + slices - 1) / slices;
  const int first = slice * per, last = first + per < total ? first + per : total;
  if (first >= last) return;  // (the whole CTA)
  launch_dependents();  // Adam's CTAs fit beside this launch's and wait there
  const int count = last - first;
  const int n_cols = job == 4 ? kMlpOut : (job == 1 ? kMlpIn : kMlpHidden);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kWgStages; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], 1);
    }
    tc::mbar_init(&acc_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
  }
  __syncwarp();
  if (warp == 0) {
    tc::tmem_alloc(&s_tmem, 256);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = s_tmem;
  wait_previous();
  if (warp == 0) {
    if (lane == 0) {
      // ---- loads ----
      const uint32_t bytes = 2 * kWgBox + (job == 4 ? kMlpOut * 128u : (uint32_t)n_cols * 128u);
      bool ok = true;
      int q = 0;
      for (; q < count; ++q) {
        const int s = q % kWgStages, u = q / kWgStages;
        if (u > 0 && !(ok = tc::mbar_wait(&empty[s], (uint32_t)(u - 1) & 1u, kWaitNs))) break;
        unsigned char* st = ring + s * kWgStage;
        const int b0 = (first + q) * 64;
        tc::mbar_expect_tx(&full[s], bytes);
        for (int k = 0; k < 2; ++k)
          tc::tma_load_3d(st + k * kWgBox, job == 4 ? &tmH : &tmZ, m0 + 64 * k, b0, job == 4 ? 2 : job - 1, &full[s]);
        if (job == 4) {
          tc::tma_load_2d(st + 2 * kWgBox, &tmY, b0, 0, &full[s]);
        } else if (job == 1) {
          tc::tma_load_2d(st + 2 * kWgBox, &tmX, 0, b0, &full[s]);
        } else {
          for (int k = 0; k < 4; ++k) tc::tma_load_3d(st + (2 + k) * kWgBox, &tmH, 64 * k, b0, job - 2, &full[s]);
        }
      }
      if (!ok) {  // the loads in flight finish before the memory goes
        s_fail = 1;
        for (int p = q > kWgStages ? q - kWgStages : 0; p < q; ++p)
          tc::mbar_wait(&full[p % kWgStages], (uint32_t)(p / kWgStages) & 1u, kWaitNs);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      // ---- MMAs: A MN-major; B MN-major, but dY, which is stored transposed, K-major ----
      const uint32_t idesc = tc::idesc_bf16(128, (uint32_t)n_cols) | 1u << 15 | (job == 4 ? 0u : 1u << 16);
      bool ok = true;
      for (int q = 0; q < count; ++q) {
        const int s = q % kWgStages, u = q / kWgStages;
        if (!(ok = tc::mbar_wait(&full[s], (uint32_t)u & 1u, kWaitNs))) break;
        tc::fence_after_sync();
        const uint32_t st = tc::smem_u32(ring + s * kWgStage);
        const uint64_t ad = wg_desc_mn(st);
        const uint64_t bd = job == 4 ? tc::smem_desc_sw128(st + 2 * kWgBox) : wg_desc_mn(st + 2 * kWgBox);
        const uint32_t bstep = job == 4 ? 2u : 128u;  // 16 rows of the batch: 32 bytes K-major, 2048 MN-major
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) tc::mma_bf16(tmem, ad + 128u * kk, bd + bstep * kk, idesc, (q | kk) ? 1u : 0u);
        tc::mma_commit(&empty[s]);
      }
      if (!ok) {  // before the epilogue can see the barrier
        *reinterpret_cast<volatile int*>(&s_fail) = 1;
        __threadfence_block();
      }
      tc::mma_commit(&acc_full);
      if (!ok) tc::mbar_wait(&acc_full, 0u, kWaitNs);
    }
    __syncwarp();
  } else {
    // ---- the partial product into the gradient ----
    const int q = warp & 3, half = (warp - 2) >> 2;
    const bool ok = __all_sync(0xffffffffu, tc::mbar_wait(&acc_full, 0u, kWaitNs)) &&
                    *reinterpret_cast<volatile int*>(&s_fail) == 0;
    tc::fence_after_sync();
    const uint32_t acc = tmem + ((uint32_t)(q * 32) << 16);
    if (ok && job == 4) {
      if (half == 0) {
        float v[16];
        tc::tmem_ld16(acc, v);
#pragma unroll
        for (int o = 0; o < kMlpOut; ++o) atomicAdd(a.grad + kOffW4 + o * kMlpHidden + m0 + q * 32 + lane, v[o]);
      }
    } else if (ok) {
      // 32 x 32 boxes, staged where the operands were (every MMA has read them), added by the TMA engine
      unsigned char* stg = ring + (warp - 2) * 4 * 4096;
      const int boxes = n_cols / 64;  // per half
      for (int k = 0; k < boxes; ++k) {
        const int n0 = (half * boxes + k) * 32;
        unsigned char* box = stg + k * 4096;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float v[16];
          tc::tmem_ld16(acc + (uint32_t)(n0 + 16 * c), v);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            *reinterpret_cast<float4*>(box + lane * 128 + (((4 * c + i) ^ (lane & 7)) << 4)) =
                make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
        tc::fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          tc::tma_reduce_add_2d(job == 3 ? &tmW3 : (job == 2 ? &tmW2 : &tmW1), box, n0, m0 + q * 32);
          tc::bulk_commit();
        }
      }
      if (lane == 0) tc::bulk_wait_all();
      __syncwarp();
    }
    if (!ok && lane == 0) s_fail = 1;
  }
  tc::fence_before_sync();
  __syncthreads();
  if (s_fail && threadIdx.x == 0 && a.err) atomicCAS(a.err, 0, ERR_MMA_TIMEOUT);
  __syncwarp();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
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
  if (e == cudaSuccess) e = cudaFuncSetAttribute(mlp_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem);
  if (e != cudaSuccess) return e;
  // H and dZ [3][B][256], X [B][64], dY^T [16][ldY]; the FP32 gradients
  CUtensorMap st_h, st_z, ld_h, ld_z, ld_x, ld_y, w[3];
  constexpr auto kBf16 = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  constexpr auto kSw = CU_TENSOR_MAP_SWIZZLE_128B;
  const cuuint64_t hd[3] = {kMlpHidden, a.B, 3}, hs[2] = {kMlpHidden * 2, a.B * kMlpHidden * 2};
  const cuuint64_t xd[2] = {kMlpIn, a.B}, xs[1] = {kMlpIn * 2}, yd[2] = {a.B, kMlpOut}, ys[1] = {a.ldY * 2};
  const cuuint32_t st_box[3] = {64, 128, 1}, ld_box[3] = {64, 64, 1}, y_box[2] = {64, kMlpOut}, w_box[2] = {32, 32};
  bool ok = encode_map(&st_h, kBf16, 3, a.H, hd, hs, st_box, kSw) && encode_map(&st_z, kBf16, 3, a.dZ, hd, hs, st_box, kSw) &&
            encode_map(&ld_h, kBf16, 3, a.H, hd, hs, ld_box, kSw) && encode_map(&ld_z, kBf16, 3, a.dZ, hd, hs, ld_box, kSw) &&
            encode_map(&ld_x, kBf16, 2, a.Xb, xd, xs, ld_box, kSw) && encode_map(&ld_y, kBf16, 2, a.dYt, yd, ys, y_box, kSw);
  for (int l = 0; l < 3; ++l) {
    const int K = l == 0 ? kMlpIn : kMlpHidden, off = l == 0 ? kOffW1 : (l == 1 ? kOffW2 : kOffW3);
    const cuuint64_t wd[2] = {(cuuint64_t)K, kMlpHidden}, ws[1] = {(cuuint64_t)K * 4};
    ok = ok && encode_map(&w[l], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, a.grad + off, wd, ws, w_box, kSw);
  }
  if (!ok) return cudaErrorInvalidValue;
  const uint64_t tiles = (a.B + 127) / 128, cap = (uint64_t)(n_sm > 1 ? n_sm / 2 : 1);
  e = launch_path(a.chained != 0, mlp_train_kernel, 2u * (unsigned)(tiles < cap ? tiles : cap), kTrainThreads, smem, stream, a,
                  st_h, st_z);
  count_launch();
  if (e != cudaSuccess) return e;
  // One item per SM.  An item of dW2 or dW3 loads 48 KB per 64 rows and adds 128 KB, one of dW1 24 and 32 KB, one of
  // dW4 18 and 8 KB: 28, 12 and 8 slices of 152 items make them about equal at 8192 rows.
  const int stages = (int)((a.B + 63) / 64);
  auto share = [&](int part) {
    const int k = n_sm * part / 152;
    return k < 1 ? 1 : (k < stages ? k : stages);
  };
  const WgradArgs g{a.B, share(28), share(12), share(8), a.grad, a.err};
  e = launch_overlapped(mlp_wgrad_kernel, (unsigned)(4 * g.k_hidden + 2 * g.k_first + 2 * g.k_last), kWgThreads, kWgSmem,
                        stream, g, ld_h, ld_z, ld_x, ld_y, w[0], w[1], w[2]);
  count_launch();
  return e;
}

}  // namespace fpt
