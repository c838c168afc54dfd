// k_infer.cu -- fused inference of the learned start on CTA pairs (tcgen05, cta_group::2).
//
// The network's BF16 weights are 303 KB, more than one SM's shared memory; streamed for every 128-path
// tile they made a chain of 19 copies, MMA groups and waits per tile that took 3.6 times as long as the
// MMAs (0.61 ns per path, tensor pipe 17 % busy).  A pair of SMs holds them once: with cta_group::2 each CTA of
// the pair supplies half of B's rows, so half of every layer's outputs (152 KB with the output layer
// padded to 32 columns) stays in each CTA's shared memory for the whole launch, beside its own 64 KB of
// activations, and nothing is streamed.
//
// Per pair and step, 256 paths (128 per CTA).  Roles: four warps form the features of the next 128 paths
// and write the starts of the last 128, one thread of the pair's first CTA issues every MMA (M = 256, N = 256;
// K = 16 steps in the order of the columns), sixteen warps run the epilogues of the hidden layers.  The two accumulators use all 512 TMEM columns: layer l + 1
// accumulates into one while the epilogue of layer l reads the other.  An epilogue hands over its layer in
// 64-column chunks, and the MMAs of the next layer run on each chunk as soon as both CTAs have written it;
// only the last chunk's four MMAs are exposed.  The next features go into the first activation chunk as
// soon as the output layer has read it.
//
// Hand-overs to the first CTA, whose thread issues the MMAs: the warps of each CTA arrive on its own barriers, and a thread
// of the second CTA, which has seen their arrivals, passes them on by a 16-byte bulk copy that completes on the first CTA's
// barrier.  That completion releases at cluster scope and holds no thread up.  (4 M city paths: the writers' own
// arrivals on the remote barrier with a cluster-scope release 2135 us, one thread that passes them on with such
// arrivals 1740, a thread per barrier 1685, the copies 1418.  Remote arrivals that release to the writers' own CTA
// only, 1364, are not ordered for the other CTA's thread by the memory model.)
//
// Measured on 4 M city paths of orders 1-5: 2580 -> 1418 us (0.35 ns per path; the same bits).  What bounds it now
// is the epilogues: 768 tanh per path at 16 a clock and SM are 6144 cycles per 128 paths (the MMAs 4900), and three
// times per tile the last chunk's MMAs and the hand-overs (about 1200 cycles) are exposed: 12,600
// cycles in all.  The rest of the GELU runs in packed FP32 pairs, five instructions for two values.
//
// Every wait is bounded; a role that runs out of time marks its CTA failed and leaves its loop, the others
// follow by their own limits, and the pair meets at its last barrier before it frees its TMEM.
#include <cuda_bf16.h>

#include "fpt_kernels.h"
#include "mlp.h"
#include "mlp_device.cuh"
#include "tc.cuh"

namespace fpt {

constexpr int kInferEpiWarps = 16;                          // four per 32-lane quarter of TMEM
constexpr int kInferFeatWarps = 4;                          // one thread per path of the CTA's 128
constexpr int kInferThreads = 32 * (kInferEpiWarps + kInferFeatWarps + 1);
static_assert(kMlpTileW4 + 4 * kMlpW4Chunk == kMlpHalfBytes, "weights of one CTA");

struct InferSmem {
  unsigned char w[kMlpHalfBytes];
  unsigned char act[4 * kMlpChunk];
  float half_bias[3 * 256];   // of the hidden layers
  float bias4[16];
  uint64_t weights;           // this CTA's weights have arrived
  uint64_t weights_pair;      // first CTA: the second's have
  // activation chunk c is written, the features are: by this CTA's warps; in the first CTA, by the second's too
  uint64_t chunk[4];
  uint64_t feat;
  uint64_t out_read;          // first CTA: the output layer's accumulator has been read in both CTAs
  uint64_t layer, out;        // MMAs of a hidden layer / of the output layer are done
  uint64_t chunk0;            // the output layer has read activation chunk 0
  uint64_t drain;
  uint32_t tmem;
  int fail;
  uint4 word[5];              // of the hand-overs (chunks, features); never read
};
static_assert(sizeof(InferSmem) <= 227 * 1024, "one CTA per SM");

// Path source, fixed per launch: kSrcEnum, an exhaustive batch's enumeration of order n; kSrcRec, records of
// orders up to kMaxBfgsOrder (the ids and the order in the record); kSrcRecDecode, records of longer
// sequences (ids decoded from the global index).
enum { kSrcEnum = 0, kSrcRec = 1, kSrcRecDecode = 2 };

template <int kSrc>
__device__ __forceinline__ void infer_fetch(const BatchDev& B, int n, const PathRec* list, uint64_t j, PathDesc& d) {
  if constexpr (kSrc == kSrcEnum) {
    decode_exhaustive_order(B, n, j, d);
  } else {
    load_rec(list, j, d);
    if constexpr (kSrc == kSrcRecDecode) decode_global(B, d.g, d);
  }
}

// One 64-column chunk of a pair's MMAs: four K = 16 steps (32 bytes, 2 in the descriptors' address field).
__device__ __forceinline__ void mma_chunk(uint32_t d_tmem, uint32_t a, uint32_t b, uint32_t idesc, bool fresh) {
  const uint64_t ad = tc::smem_desc_sw128(a), bd = tc::smem_desc_sw128(b);
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) tc::mma_bf16_pair(d_tmem, ad + 2u * kk, bd + 2u * kk, idesc, fresh && kk == 0 ? 0u : 1u);
}

// BF16 GELU of two accumulator values plus bias, in packed FP32 instructions: with h = z / 2 = acc / 2 + bias / 2,
// u = h (2 K0 + 8 K0 K1 h^2) and gelu = h + h tanh(u).  The factors are powers of two, so every step rounds as
// gelu()'s does, with one product less.
__device__ __forceinline__ uint32_t gelu_pair(uint32_t v0, uint32_t v1, uint64_t half_bias) {
  const uint64_t half = tc::splat2(0.5f), k8 = tc::splat2(8.f * kGeluK01), k2 = tc::splat2(2.f * kGeluK0);
  const uint64_t h = tc::fma2(tc::pack2(v0, v1), half, half_bias);
  const uint64_t u = tc::mul2(h, tc::fma2(k8, tc::mul2(h, h), k2));
  float u0, u1;
  tc::unpack2(u, u0, u1);
  const uint64_t th = tc::pack2(__float_as_uint(tanh_approx(u0)), __float_as_uint(tanh_approx(u1)));
  float y0, y1;
  tc::unpack2(tc::fma2(h, th, h), y0, y1);
  const __nv_bfloat162 p = __floats2bfloat162_rn(y0, y1);
  return *reinterpret_cast<const uint32_t*>(&p);
}

// A bounded wait of a whole warp for a commit of the pair's MMAs: true only if every lane saw the phase complete (the lanes
// stay together for the warp-wide instructions that follow).
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, tc::mbar_wait_cluster(bar, parity, kWaitNs));
}

template <int kSrc>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kInferThreads, 1)
    mlp_infer_kernel(SceneDev S, BatchDev B, int n, const PathRec* __restrict__ list, uint64_t count, float inv_scale,
                     const __nv_bfloat16* __restrict__ wt, const float* __restrict__ params, float* T, int n_fill,
                     int* err) {
  extern __shared__ __align__(1024) unsigned char infer_smem[];
  InferSmem& sm = *reinterpret_cast<InferSmem*>(infer_smem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = tc::cluster_rank();
  const uint32_t n_pairs = gridDim.x >> 1, pair = blockIdx.x >> 1;
  const uint64_t n_tiles = (count + 255) / 256;  // per pair and step: 256 paths
  const uint64_t my_tiles = pair < n_tiles ? (n_tiles - pair + n_pairs - 1) / n_pairs : 0;
  if (tid == 0) {
    tc::mbar_init(&sm.weights, 1);
    tc::mbar_init(&sm.weights_pair, 1);
    const uint32_t other = rank == 0 ? 1u : 0u;  // the second CTA's hand-over
    for (int c = 0; c < 4; ++c) tc::mbar_init(&sm.chunk[c], kInferEpiWarps + other);
    tc::mbar_init(&sm.feat, kInferFeatWarps + other);
    tc::mbar_init(&sm.out_read, 2 * kInferFeatWarps);
    tc::mbar_init(&sm.layer, 1);
    tc::mbar_init(&sm.out, 1);
    tc::mbar_init(&sm.chunk0, 1);
    tc::mbar_init(&sm.drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sm.fail = 0;
    const char* src = reinterpret_cast<const char*>(wt) + rank * kMlpHalfBytes;
    tc::mbar_expect_tx(&sm.weights, kMlpHalfBytes);
    for (uint32_t o = 0; o < kMlpHalfBytes; o += kMlpChunk)
      tc::bulk_g2s(sm.w + o, src + o, o + kMlpChunk <= kMlpHalfBytes ? kMlpChunk : kMlpHalfBytes - o,
                   &sm.weights);
  }
  for (int i = tid; i < 256; i += blockDim.x) {
    sm.half_bias[i] = 0.5f * params[kOffB1 + i];
    sm.half_bias[256 + i] = 0.5f * params[kOffB2 + i];
    sm.half_bias[512 + i] = 0.5f * params[kOffB3 + i];
  }
  if (tid < 16) sm.bias4[tid] = params[kOffB4 + tid];
  __syncwarp();
  if (warp == 0) {
    tc::tmem_alloc_pair(&sm.tmem, 512);
    tc::tmem_relinquish_pair();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::cluster_sync();  // the peer's barriers are initialised before anything arrives on them
  tc::fence_after_sync();
  const uint32_t tmem = sm.tmem;

  if (warp < kInferEpiWarps) {
    // ---- epilogues of the hidden layers ----
    const uint32_t rg = warp & 3, part = warp >> 2;  // TMEM lane quarter; which 16 columns of a chunk
    const uint32_t row = rg * 32 + lane;
    const uint32_t lane_addr = tmem + ((rg * 32u) << 16) + part * 16u;
    uint4* const dst0 = reinterpret_cast<uint4*>(sm.act + tc::sw128_offset(row, part * 16u));
    uint4* const dst1 = reinterpret_cast<uint4*>(sm.act + tc::sw128_offset(row, part * 16u + 8u));
    auto hand_over = [&](int c) {
      tc::fence_async_smem();
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sm.chunk[c]);
    };
    uint32_t ph_layer = 0u;
    bool ok = true;
    for (uint64_t ti = 0; ti < my_tiles && ok; ++ti) {
#pragma unroll 1
      for (int l = 0; l < 3; ++l) {
        ok = warp_wait(&sm.layer, ph_layer);
        if (!ok) break;
        ph_layer ^= 1u;
        tc::fence_after_sync();
        const uint32_t acc = lane_addr + (l & 1 ? 256u : 0u);
        const float* bias = sm.half_bias + l * 256 + part * 16;
        uint32_t v[2][16];
        tc::tmem_ld16_issue(acc, v[0]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t(&x)[16] = v[c & 1];
          tc::tmem_ld16_wait(x);
          if (c < 3) tc::tmem_ld16_issue(acc + (c + 1) * 64u, v[(c + 1) & 1]);
          const ulonglong2* bp = reinterpret_cast<const ulonglong2*>(bias + c * 64);
          uint32_t w[8];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const ulonglong2 b2 = bp[k];
            w[2 * k] = gelu_pair(x[4 * k], x[4 * k + 1], b2.x);
            w[2 * k + 1] = gelu_pair(x[4 * k + 2], x[4 * k + 3], b2.y);
            // chunk c - 1 is handed over only now: its stores have completed, so the fence does not wait for them
            if (k == 1 && c > 0) hand_over(c - 1);
          }
          dst0[c * (kMlpChunk / 16)] = make_uint4(w[0], w[1], w[2], w[3]);
          dst1[c * (kMlpChunk / 16)] = make_uint4(w[4], w[5], w[6], w[7]);
          if (c == 3) hand_over(3);
        }
      }
    }
    if (!ok) sm.fail = 1;
  } else if (warp < kInferEpiWarps + kInferFeatWarps) {
    // ---- a thread per path: features of tile ti while the layers of tile ti - 1 run, then that tile's starts ----
    const int row = tid - 32 * kInferEpiWarps;
    const uint32_t out_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 256u;
    uint64_t g = 0;      // the path of tile ti - 1: global index,
    uint32_t info = 0u;  // order | (sequence usable) << 8 | edge mask << 16 (order 0: no path)
    bool ok = true;
    for (uint64_t ti = 0; ti <= my_tiles; ++ti) {
      const uint64_t j = (pair + ti * n_pairs) * 256 + rank * 128 + row;
      uint4 f[kMlpIn / 8];
      uint64_t g_new = 0;
      uint32_t info_new = 0u;
#pragma unroll
      for (int k = 0; k < kMlpIn / 8; ++k) f[k] = make_uint4(0u, 0u, 0u, 0u);
      if (ti < my_tiles && j < count) {
        PathDesc d;
        infer_fetch<kSrc>(B, n, list, j, d);
        path_features(S, d, inv_scale, reinterpret_cast<__nv_bfloat16*>(f), nullptr);
        g_new = d.g;
        info_new = (uint32_t)d.n | (d.flags & ST_INVALID ? 0u : 1u << 8) | (edge_mask(S, d) << 16);
      }
      // the previous tile's output layer has read the chunk (waited for after the last tile too, so that no arrival
      // is on its way to a CTA that has left)
      if (ti > 0 && !(ok = warp_wait(&sm.chunk0, (uint32_t)(ti - 1) & 1u))) break;
      if (ti < my_tiles) {
#pragma unroll
        for (int k = 0; k < kMlpIn / 8; ++k)
          *reinterpret_cast<uint4*>(sm.act + tc::sw128_offset(row, k * 8)) = f[k];
        tc::fence_async_smem();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&sm.feat);
      }
      if (ti > 0) {
        if (!(ok = warp_wait(&sm.out, (uint32_t)(ti - 1) & 1u))) break;
        tc::fence_after_sync();
        float v[16];
        tc::tmem_ld16(out_addr, v);
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive_remote_relaxed(tc::map_rank(&sm.out_read, 0));
        if (info & 0xFFu) {
          float y[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) y[i] = v[i] + sm.bias4[i];
          float2* To = reinterpret_cast<float2*>(T) + g * (uint64_t)B.n_max;
          const int np = (int)(info & 0xFFu);
          write_start(np, (info >> 8) & 1u, info >> 16, y, To);
          for (int s = np; s < n_fill; ++s) To[s] = make_float2(0.f, 0.f);
        }
      }
      g = g_new;
      info = info_new;
    }
    if (!ok) sm.fail = 1;
  } else {
    if (lane == 0) {
      bool ok = tc::mbar_wait(&sm.weights, 0u, kWaitNs);
      if (rank == 1) {
        // ---- the second CTA's hand-overs, passed on in the order in which they come (the next tile's features follow the
        // output layer's first chunk).  The first CTA waits for each of them before it leaves. ----
        if (ok) tc::mbar_arrive_remote(tc::map_rank(&sm.weights_pair, 0));
        const uint32_t words = tc::map_rank(sm.word, 0), chunks = tc::map_rank(sm.chunk, 0);
        const uint32_t feat = tc::map_rank(&sm.feat, 0);
        uint32_t ph_chunk = 0u;
        auto pass_features = [&](uint64_t ti) {
          ok = ok && tc::mbar_wait(&sm.feat, (uint32_t)ti & 1u, kWaitNs);
          if (ok) tc::signal_remote(words + 4u * sizeof(uint4), sm.word + 4, feat);
        };
        if (my_tiles > 0) pass_features(0);
        for (uint64_t ti = 0; ti < my_tiles && ok; ++ti) {
          for (int l = 1; l < 4; ++l) {
            for (int c = 0; c < 4 && ok; ++c) {
              ok = tc::mbar_wait(&sm.chunk[c], ph_chunk, kWaitNs);
              if (ok) tc::signal_remote(words + c * (uint32_t)sizeof(uint4), sm.word + c, chunks + 8u * c);
            }
            ph_chunk ^= 1u;
          }
          if (ti + 1 < my_tiles) pass_features(ti + 1);
        }
      } else {
        // ---- the pair's MMAs ----
        ok = ok && tc::mbar_wait_cluster(&sm.weights_pair, 0u, kWaitNs);
        const uint32_t w = tc::smem_u32(sm.w), act = tc::smem_u32(sm.act);
        constexpr uint32_t id256 = tc::idesc_bf16(256, 256), id32 = tc::idesc_bf16(256, 32);
        uint32_t ph_chunk = 0u, ph_feat = 0u;
        for (uint64_t ti = 0; ti < my_tiles && ok; ++ti) {
          tc::mbar_expect_tx(&sm.feat, tc::kSignalBytes);
          if (!(ok = tc::mbar_wait_cluster(&sm.feat, ph_feat, kWaitNs))) break;
          ph_feat ^= 1u;
          tc::fence_after_sync();
          mma_chunk(tmem, act, w, id256, true);
          tc::mma_commit_pair(&sm.layer);
          // layer 2 goes into the accumulator the last tile's output layer used
          if (ti > 0 && !(ok = tc::mbar_wait_cluster(&sm.out_read, (uint32_t)(ti - 1) & 1u, kWaitNs))) break;
          for (int l = 1; l < 4 && ok; ++l) {
            const uint32_t acc = tmem + (l & 1 ? 256u : 0u);
            const uint32_t wl = w + (l == 1 ? kMlpTileW2 : (l == 2 ? kMlpTileW3 : kMlpTileW4));
            const uint32_t wc = l < 3 ? kMlpChunk : kMlpW4Chunk;
            for (int c = 0; c < 4; ++c) tc::mbar_expect_tx(&sm.chunk[c], tc::kSignalBytes);
            for (int c = 0; c < 4; ++c) {
              if (!(ok = tc::mbar_wait_cluster(&sm.chunk[c], ph_chunk, kWaitNs))) break;
              tc::fence_after_sync();
              mma_chunk(acc, act + c * kMlpChunk, wl + c * wc, l < 3 ? id256 : id32, c == 0);
              if (l == 3 && c == 0) tc::mma_commit_pair(&sm.chunk0);
            }
            if (!ok) break;
            ph_chunk ^= 1u;
            tc::mma_commit_pair(l < 3 ? &sm.layer : &sm.out);
          }
        }
        if (ok && my_tiles > 0) ok = tc::mbar_wait_cluster(&sm.out_read, (uint32_t)(my_tiles - 1) & 1u, kWaitNs);
        if (!ok) {  // let the MMAs in flight finish before the TMEM goes
          tc::mma_commit_pair(&sm.drain);
          tc::mbar_wait(&sm.drain, 0u, kWaitNs);
        }
      }
      if (!ok) sm.fail = 1;
    }
    __syncwarp();
  }
  tc::fence_before_sync();
  __syncthreads();
  if (sm.fail && tid == 0 && err) atomicCAS(err, 0, ERR_MMA_TIMEOUT);
  tc::cluster_sync();  // no arrival or MMA of the peer reaches a CTA that has left
  if (warp == 0) tc::tmem_dealloc_pair(tmem, 512);
}

cudaError_t launch_mlp_infer(const SceneDev& S, const BatchDev& B, int n, const PathRec* list, uint64_t count,
                             float inv_scale, const __nv_bfloat16* wt, const float* params, float* T, int n_fill,
                             int* err, cudaStream_t stream, int n_sm) {
  if (!count) return cudaSuccess;
  auto kern = list == nullptr ? mlp_infer_kernel<kSrcEnum>
                              : (n > kMaxBfgsOrder ? mlp_infer_kernel<kSrcRecDecode> : mlp_infer_kernel<kSrcRec>);
  const int smem = (int)sizeof(InferSmem);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const uint64_t tiles = (count + 255) / 256, cap = (uint64_t)(n_sm > 1 ? n_sm / 2 : 1);
  const unsigned grid = 2u * (unsigned)(tiles < cap ? tiles : cap);
  kern<<<grid, kInferThreads, smem, stream>>>(S, B, n, list, count, inv_scale, wt, params, T, n_fill, err);
  count_launch();
  return cudaGetLastError();
}

}  // namespace fpt
