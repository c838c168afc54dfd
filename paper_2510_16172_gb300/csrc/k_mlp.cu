// k_mlp.cu -- tensor-core (tcgen05) kernels of the learned warm start.
//
// A small MLP (3 hidden layers of 256, GELU) maps the geometry of a candidate
// sequence (TX, RX and the first four objects) to starting parameters t for
// the solver.  Weights are BF16, accumulation FP32 in tensor memory,
// activations are rounded to BF16 between layers.
//
// GEMMs D[M x N] = sum_k A(m, k) B(n, k), N <= 256, K in chunks of 64, for the unfused forward pass.  Operands whose
// rows are contiguous and 16-byte aligned go to gemm_ws_kernel: persistent, one CTA per SM over 128-row tiles, the
// chunks loaded by TMA into a three-stage ring (128-byte swizzled K-major tiles), one thread issuing the MMAs
// into two TMEM accumulators, twelve epilogue warps staging the outputs in shared memory for TMA tensor stores.
// Other strides take gemm_kernel, one tile per CTA with the operands gathered element by element.  Epilogues: plain
// store (+ bias); bias + GELU with a BF16 activation.  Inference is fused in k_infer.cu, training in k_train.cu.
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include "fpt_kernels.h"
#include "mlp.h"
#include "mlp_device.cuh"
#include "tc.cuh"

namespace fpt {

constexpr int kGemmKC = 64;                  // K per chunk

// Gather rows [r0, r0 + 128) x k [k0, k0 + 64) of a strided bf16 matrix into a
// 128 x 64 K-major tile (zero outside rows < R, k < K).
__device__ __forceinline__ void load_tile(unsigned char* tile, const __nv_bfloat16* src, long long s_r, long long s_k,
                                          int R, int K, int r0, int k0, int rows) {
  const bool vec = (s_k == 1) && ((s_r & 7) == 0) && ((reinterpret_cast<uintptr_t>(src) & 15) == 0);
  if (vec) {
    // 16-byte chunks: (row, group of 8 along k)
    for (int idx = threadIdx.x; idx < rows * (kGemmKC / 8); idx += blockDim.x) {
      const int r = idx / (kGemmKC / 8), kg = idx % (kGemmKC / 8);
      const int gr = r0 + r, gk = k0 + kg * 8;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (gr < R && gk + 8 <= K) {
        v = *reinterpret_cast<const uint4*>(src + (long long)gr * s_r + gk);
      } else if (gr < R && gk < K) {
        __nv_bfloat16 e[8];
        for (int q = 0; q < 8; ++q) e[q] = gk + q < K ? src[(long long)gr * s_r + gk + q] : __float2bfloat16(0.f);
        v = *reinterpret_cast<uint4*>(e);
      }
      *reinterpret_cast<uint4*>(tile + tc::kmajor_offset(r, kg * 8, kGemmKC)) = v;
    }
  } else {
    // element gather, consecutive threads along rows (coalesced when rows are contiguous)
    for (int idx = threadIdx.x; idx < rows * kGemmKC; idx += blockDim.x) {
      const int r = idx % rows, k = idx / rows;
      const int gr = r0 + r, gk = k0 + k;
      __nv_bfloat16 v = __float2bfloat16(0.f);
      if (gr < R && gk < K) v = src[(long long)gr * s_r + (long long)gk * s_k];
      *reinterpret_cast<__nv_bfloat16*>(tile + tc::kmajor_offset(r, k, kGemmKC)) = v;
    }
  }
}

// 16 bytes global -> shared, asynchronous (cp.async), the bytes past src_bytes (0..16) zero-filled.
__device__ __forceinline__ void cp_async16(void* dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(dst)), "l"(src), "r"(src_bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory");
}

// Rows [r0, r0 + rows) x k [k0, k0 + 64) of a row-major bf16 matrix whose rows start on 16-byte
// boundaries into the K-major tile layout, with asynchronous 16-byte copies (zero outside rows < R,
// k < K).  Consecutive threads take consecutive 16-byte pieces of a row: a warp reads four whole rows.
__device__ __forceinline__ void load_tile_async(unsigned char* tile, const __nv_bfloat16* src, long long s_r, int R,
                                                int K, int r0, int k0, int rows) {
  for (int idx = threadIdx.x; idx < rows * (kGemmKC / 8); idx += blockDim.x) {
    const int r = idx / (kGemmKC / 8), kg = idx % (kGemmKC / 8);
    const int gr = r0 + r, gk = k0 + kg * 8;
    const int valid = gr < R ? min(max(K - gk, 0), 8) : 0;
    const __nv_bfloat16* p = valid ? src + (long long)gr * s_r + gk : src;
    cp_async16(tile + tc::kmajor_offset(r, kg * 8, kGemmKC), p, (uint32_t)valid * 2u);
  }
}

// Operands that the pipelined path takes: unit stride along k, rows 16-byte aligned.
__host__ __device__ inline bool gemm_vectorised(const GemmArgs& g) {
  const bool a = g.sak == 1 && (g.sam % 8) == 0 && (reinterpret_cast<uintptr_t>(g.A) & 15) == 0;
  const bool b = g.sbk == 1 && (g.sbn % 8) == 0 && (reinterpret_cast<uintptr_t>(g.B) & 15) == 0;
  return a && b;
}

constexpr int kGemmStages = 2;                                      // K chunks in flight
constexpr int kGemmTileA = 128 * kGemmKC * 2;                       // 16 KB
constexpr int kGemmStageBytes = kGemmTileA + 256 * kGemmKC * 2;     // A + B (N <= 256): 48 KB
constexpr int kGemmSmem = kGemmStages * kGemmStageBytes;            // 96 KB: two CTAs per SM
// Epilogue staging: each warp's 32 accumulator rows, 64 columns at a time, in a private slab of the
// (by then idle) pipeline buffers; rows padded to 65 floats so that both the row-wise and the
// column-wise passes hit 32 different banks.
constexpr int kEpiCols = 64, kEpiStride = kEpiCols + 1;
static_assert(4 * 32 * kEpiStride * 4 <= kGemmSmem, "epilogue slabs");

// Epilogue of one warp's 32 accumulator rows (TMEM lanes 32 w .. 32 w + 31, matrix rows mrow0 ..).  Per
// 64-column slab: (a) the accumulator (+ bias) goes from TMEM to the warp's staging slab, lane = row;
// (b) row by row, consecutive lanes on consecutive columns, the output is formed and stored (coalesced).
__device__ __forceinline__ void gemm_epilogue_staged(const GemmArgs& g, uint32_t tmem_warp, int mrow0, int lane,
                                                     int n_pad, float* slab) {
  for (int c0 = 0; c0 < n_pad; c0 += kEpiCols) {
    const int cols = min(kEpiCols, n_pad - c0);
    for (int cc = 0; cc < cols; cc += 16) {
      float v[16];
      tc::tmem_ld16(tmem_warp + (uint32_t)(c0 + cc), v);
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int n = c0 + cc + q;
        float x = v[q];
        if (g.bias && n < g.N) x += g.bias[n];
        slab[lane * kEpiStride + cc + q] = x;
      }
    }
    __syncwarp();
    for (int r = 0; r < 32; ++r) {
      const int m = mrow0 + r;
      if (m >= g.M) break;  // r is the same for the whole warp
      for (int cc = lane; cc < cols; cc += 32) {
        const int n = c0 + cc;
        if (n >= g.N) continue;
        const float x = slab[r * kEpiStride + cc];
        if (g.op == EPI_STORE)
          g.C[(long long)m * g.scm + (long long)n * g.scn] = x;
        else
          g.H[(long long)m * g.shm + (long long)n * g.shn] = __float2bfloat16(gelu(x));
      }
    }
    __syncwarp();
  }
}

__global__ void __launch_bounds__(128) gemm_kernel(GemmArgs g) {
  extern __shared__ __align__(1024) unsigned char gemm_smem[];
  __shared__ __align__(8) uint64_t bar[kGemmStages];
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * 128;
  const int n_pad = (g.N + 15) & ~15;
  const uint32_t ncols = n_pad <= 32 ? 32 : (n_pad <= 64 ? 64 : (n_pad <= 128 ? 128 : 256));
  const int n_chunks = (g.K + kGemmKC - 1) / kGemmKC;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kGemmStages; ++s) tc::mbar_init(&bar[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
  }
  if (warp == 0) {
    tc::tmem_alloc(&s_tmem, ncols);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = s_tmem;
  const uint32_t idesc = tc::idesc_bf16(128, n_pad);
  auto stage_a = [&](int s) { return gemm_smem + s * kGemmStageBytes; };
  auto stage_b = [&](int s) { return gemm_smem + s * kGemmStageBytes + kGemmTileA; };
  auto issue = [&](int c) {  // one thread: the four MMAs of chunk c, then its commit
    const int s = c % kGemmStages;
    tc::fence_after_sync();
    const uint32_t a0 = tc::smem_u32(stage_a(s)), b0 = tc::smem_u32(stage_b(s));
#pragma unroll
    for (int kk = 0; kk < kGemmKC / 16; ++kk) {
      const uint64_t ad = tc::smem_desc(a0 + kk * 256, 128, (kGemmKC / 8) * 128);
      const uint64_t bd = tc::smem_desc(b0 + kk * 256, 128, (kGemmKC / 8) * 128);
      tc::mma_bf16(tmem, ad, bd, idesc, (c | kk) ? 1u : 0u);
    }
    tc::mma_commit(&bar[s]);
  };
  // chunk c's MMAs have completed: its stage barrier's phase number c / kGemmStages.  A thread whose
  // bounded wait runs out sets s_fail, which every thread reads only after the next barrier.
  auto wait_chunk = [&](int c) {
    if (tc::mbar_wait(&bar[c % kGemmStages], (uint32_t)((c / kGemmStages) & 1), kWaitNs)) return true;
    atomicExch(&s_fail, 1);
    return false;
  };
  if (gemm_vectorised(g)) {
    // pipelined: chunks load (cp.async, one commit group per chunk) kGemmStages - 1 ahead of the MMAs
    for (int c = 0; c < kGemmStages - 1; ++c) {
      if (c < n_chunks) {
        load_tile_async(stage_a(c), g.A, g.sam, g.M, g.K, m0, c * kGemmKC, 128);
        load_tile_async(stage_b(c), g.B, g.sbn, g.N, g.K, 0, c * kGemmKC, n_pad);
      }
      cp_async_commit();
    }
    for (int c = 0; c < n_chunks; ++c) {
      cp_async_wait<kGemmStages - 2>();  // this thread's copies of chunk c (group c) have landed
      tc::fence_async_smem();
      __syncthreads();
      if (s_fail) break;  // the same value for every thread after the barrier
      if (threadIdx.x == 0) issue(c);
      // refill the stage of chunk c - 1 with chunk c + kGemmStages - 1 once chunk c - 1's MMAs, queued ahead
      // of chunk c's, have read it
      const int cn = c + kGemmStages - 1;
      if (cn < n_chunks && (c == 0 || wait_chunk(c - 1))) {
        const int sn = cn % kGemmStages;
        load_tile_async(stage_a(sn), g.A, g.sam, g.M, g.K, m0, cn * kGemmKC, 128);
        load_tile_async(stage_b(sn), g.B, g.sbn, g.N, g.K, 0, cn * kGemmKC, n_pad);
      }
      cp_async_commit();
    }
    cp_async_wait<0>();
  } else {
    // element gathers from arbitrary strides: one stage, each chunk waited for before the next
    for (int c = 0; c < n_chunks; ++c) {
      load_tile(stage_a(0), g.A, g.sam, g.sak, g.M, g.K, m0, c * kGemmKC, 128);
      load_tile(stage_b(0), g.B, g.sbn, g.sbk, g.N, g.K, 0, c * kGemmKC, n_pad);
      tc::fence_async_smem();
      __syncthreads();
      if (threadIdx.x == 0) {
        const int s = c % kGemmStages;
        tc::fence_after_sync();
        const uint32_t a0 = tc::smem_u32(stage_a(0)), b0 = tc::smem_u32(stage_b(0));
#pragma unroll
        for (int kk = 0; kk < kGemmKC / 16; ++kk) {
          const uint64_t ad = tc::smem_desc(a0 + kk * 256, 128, (kGemmKC / 8) * 128);
          const uint64_t bd = tc::smem_desc(b0 + kk * 256, 128, (kGemmKC / 8) * 128);
          tc::mma_bf16(tmem, ad, bd, idesc, (c | kk) ? 1u : 0u);
        }
        tc::mma_commit(&bar[s]);
      }
      wait_chunk(c);  // the tile is reused by the next chunk
      tc::fence_after_sync();
      __syncthreads();
      if (s_fail) break;
    }
  }
  __syncthreads();
  if (n_chunks > 0 && !s_fail) wait_chunk(n_chunks - 1);  // the last commit: every MMA has completed
  tc::fence_after_sync();
  __syncthreads();
  if (s_fail) {
    if (threadIdx.x == 0 && g.err) atomicCAS(g.err, 0, ERR_MMA_TIMEOUT);
    // give MMAs still in flight a (bounded) chance to finish before TMEM is freed
    if (n_chunks > 0) tc::mbar_wait(&bar[(n_chunks - 1) % kGemmStages], (uint32_t)(((n_chunks - 1) / kGemmStages) & 1),
                                    kWaitNs);
  } else if (n_chunks > 0) {
    // epilogue: warp w owns TMEM lanes (rows) 32 w .. 32 w + 31; the pipeline buffers are idle now
    float* slab = reinterpret_cast<float*>(gemm_smem) + warp * 32 * kEpiStride;
    gemm_epilogue_staged(g, tmem + ((uint32_t)(warp * 32) << 16), m0 + warp * 32, lane, n_pad, slab);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, ncols);
}

// ---- persistent warp-specialised GEMM (TMA operands) -------------------------------------------------
// One CTA per SM walks the 128-row tiles.  Warp 0 (one thread) loads each 64-wide K chunk
// of A (128 rows) and B (n_pad rows) with one TMA tile load per operand into a ring of kWsStages stages,
// in the 128-byte swizzled K-major layout; rows past M or N and k past K arrive as zeros.  Warp 1 (one
// thread) issues four 128 x n_pad x 16 MMAs per chunk into one of two TMEM accumulators (columns 0-255,
// 256-511), releases the chunk's stage by a commit to `empty` and announces a finished tile by a commit
// to `acc_full`.  Warps 2-13 are the epilogue: three warps per 32-lane quarter of TMEM (a warp may read the
// quarter given by its index mod 4), each on every third group of 16 columns, one output row per lane.
// Each 32 x 16 group is staged in shared memory and written by TMA tensor stores (full lines, no
// per-lane store traffic); outputs whose strides a tensor map cannot describe are stored by the lanes.
// The warps hand the accumulator back through `acc_empty`, so the MMAs of the tile after next may start
// while this tile's epilogue runs.  Every wait is bounded; a timeout sets the CTA's fail flag, which every
// role polls and leaves on.
constexpr int kWsStages = 3;  // operand ring
constexpr int kWsEpiWarps = 12;
constexpr int kWsGroupStride = kWsEpiWarps / 4;  // epilogue warps per 32-lane quarter of TMEM
constexpr int kWsThreads = 32 * (2 + kWsEpiWarps);
constexpr int kWsTileA = 128 * 128;                       // 128 rows x 128 bytes
constexpr int kWsStageBytes = kWsTileA + 256 * 128;       // + B, up to 256 rows: 48 KB
// the ring, two 2 KB output staging buffers per epilogue warp, slack to align the ring to 1024 bytes
constexpr int kWsSmem = kWsStages * kWsStageBytes + kWsEpiWarps * 2 * 2048 + 1024;

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

// Which accesses may take 16 bytes (unit stride along n, row strides and bases aligned).
struct EpiVec {
  bool c, h, bias;
};
__device__ __forceinline__ bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
__device__ __forceinline__ EpiVec epi_vec(const GemmArgs& g) {
  EpiVec v;
  v.c = g.scn == 1 && g.scm % 4 == 0 && aligned16(g.C);
  v.h = g.shn == 1 && g.shm % 8 == 0 && aligned16(g.H);
  v.bias = aligned16(g.bias);
  return v;
}

__device__ __forceinline__ void store16_f32(float* p, const float (&x)[16], bool vec, int nv, long long sn) {
  if (vec) {
    float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (i < nv) p[i * sn] = x[i];
  }
}
__device__ __forceinline__ void store16_bf16(__nv_bfloat16* p, const float (&x)[16], bool vec, int nv, long long sn) {
  if (vec) {
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const __nv_bfloat162 b2 = __floats2bfloat162_rn(x[2 * i], x[2 * i + 1]);
      w[i] = *reinterpret_cast<const uint32_t*>(&b2);
    }
    uint4* q = reinterpret_cast<uint4*>(p);
    q[0] = make_uint4(w[0], w[1], w[2], w[3]);
    q[1] = make_uint4(w[4], w[5], w[6], w[7]);
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (i < nv) p[i * sn] = __float2bfloat16(x[i]);
  }
}

// Staging of one warp's 32 x 16 output group for the TMA tensor stores (two buffers per warp, used in
// turn): the FP32 box in the 64-byte swizzled layout (row r, 16-byte chunk c at r 64 + 16 (c ^ (r / 2 mod 4))),
// the BF16 box in the 32-byte swizzled layout (r 32 + 16 (c ^ (r / 4 mod 2))).  Consecutive lanes (rows) hit
// different banks in both.
constexpr int kStgBytes = 2048;

// One warp's share of a finished 128 x n_pad accumulator: its lane quarter, column groups j0, j0 + kWsGroupStride, ...
// m = this lane's output row, mrow0 = the warp's first row.  The output goes out through a TMA store of the
// staged group when its tensor map exists (`tma`), else with this lane's own stores.  gi counts the warp's
// groups (it picks the staging buffer).
template <int OP>
__device__ __forceinline__ void ws_epilogue(const GemmArgs& g, const EpiVec& ev, uint32_t tacc, int m, int mrow0,
                                            int j0, int n_groups, const CUtensorMap* out, bool tma, unsigned char* stg,
                                            int& gi) {
  const int lane = lane_id();
  const bool row = m < g.M;
  for (int j = j0; j < n_groups; j += kWsGroupStride) {
    const int n0 = 16 * j;
    const int nv = min(16, g.N - n0);
    const bool full = nv == 16;
    float x[16];
    __syncwarp();
    tc::tmem_ld16(tacc + (uint32_t)n0, x);
    if (g.bias) {
      if (full && ev.bias) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 b = __ldg(reinterpret_cast<const float4*>(g.bias + n0) + i);
          x[4 * i] += b.x;
          x[4 * i + 1] += b.y;
          x[4 * i + 2] += b.z;
          x[4 * i + 3] += b.w;
        }
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (i < nv) x[i] += g.bias[n0 + i];
      }
    }
    if (OP == EPI_BIAS_GELU) {
#pragma unroll
      for (int i = 0; i < 16; ++i) x[i] = gelu(x[i]);
    }
    if (!tma) {  // this lane's own stores
      if (row && OP == EPI_STORE)
        store16_f32(g.C + (long long)m * g.scm + (long long)n0 * g.scn, x, full && ev.c, nv, g.scn);
      if (row && OP == EPI_BIAS_GELU)
        store16_bf16(g.H + (long long)m * g.shm + (long long)n0 * g.shn, x, full && ev.h, nv, g.shn);
      continue;
    }
    // the staged group: wait until the engine has read this buffer's previous group, fill it, store it
    unsigned char* buf = stg + (gi & 1) * kStgBytes;
    ++gi;
    if (lane == 0) tc::bulk_wait_read<1>();
    __syncwarp();
    if (OP == EPI_STORE) {
      unsigned char* cb = buf + lane * 64;
      const int sw = (lane >> 1) & 3;
#pragma unroll
      for (int c = 0; c < 4; ++c)
        *reinterpret_cast<float4*>(cb + 16 * (c ^ sw)) = make_float4(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
    } else {
      unsigned char* hb = buf + lane * 32;
      const int sw = (lane >> 2) & 1;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const __nv_bfloat162 b2 = __floats2bfloat162_rn(x[8 * c + 2 * i], x[8 * c + 2 * i + 1]);
          w[i] = *reinterpret_cast<const uint32_t*>(&b2);
        }
        *reinterpret_cast<uint4*>(hb + 16 * (c ^ sw)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    tc::fence_async_smem();
    __syncwarp();
    if (lane == 0 && mrow0 < g.M) {
      tc::tma_store_2d(out, buf, n0, mrow0);
      tc::bulk_commit();
    }
  }
}

__global__ void __launch_bounds__(kWsThreads, 1)
    gemm_ws_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ CUtensorMap tmOut, int tma_out, GemmArgs g, int m_tiles) {
  extern __shared__ unsigned char ws_raw[];
  __shared__ __align__(8) uint64_t full[kWsStages], empty[kWsStages], acc_full[2], acc_empty[2];
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;
  __shared__ int s_last_q;             // the MMA thread's last committed chunk (-1: none)
  __shared__ int s_armed[kWsStages];  // each stage's last phase handed to the TMA engine (-1: none)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned all = 0xffffffffu;
  const int n_pad = (g.N + 15) & ~15;
  unsigned char* ring = ws_raw + ((1024u - (tc::smem_u32(ws_raw) & 1023u)) & 1023u);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kWsStages; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], 1);
      s_armed[s] = -1;
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&acc_full[b], 1);
      tc::mbar_init(&acc_empty[b], kWsEpiWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
    s_last_q = -1;
  }
  if (warp == 0) {
    tc::tmem_alloc(&s_tmem, 512);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = s_tmem;
  auto stage_a = [&](int s) { return ring + s * kWsStageBytes; };
  auto stage_b = [&](int s) { return ring + s * kWsStageBytes + kWsTileA; };
  auto failed = [&]() { return *reinterpret_cast<volatile int*>(&s_fail) != 0; };

  if (warp == 0) {
    // ---- TMA producer ----
    if (lane == 0) {
      const uint32_t tx_bytes = (uint32_t)(128 + n_pad) * 128u;
      int q = 0;
      bool ok = true;
      for (int item = blockIdx.x; ok && item < m_tiles; item += gridDim.x) {
        for (int k0 = 0; k0 < g.K; k0 += kGemmKC, ++q) {
          const int s = q % kWsStages, u = q / kWsStages;
          if (u > 0) {  // the stage's previous chunk has been read by its MMAs
            ok = !failed() && tc::mbar_wait(&empty[s], (uint32_t)((u - 1) & 1), kWaitNs);
            if (!ok) break;
          }
          tc::mbar_expect_tx(&full[s], tx_bytes);
          s_armed[s] = u;
          tc::tma_load_2d(stage_a(s), &tmA, k0, item * 128, &full[s]);
          tc::tma_load_2d(stage_b(s), &tmB, k0, 0, &full[s]);
        }
      }
      if (!ok) atomicExch(&s_fail, 1);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---- MMA issuer ----
    if (lane == 0) {
      int q = 0, i = 0;
      bool ok = true;
      const uint32_t idesc = tc::idesc_bf16(128, (uint32_t)n_pad);
      for (int item = blockIdx.x; ok && item < m_tiles; item += gridDim.x, ++i) {
        const int b = i & 1, v = i >> 1;
        if (v > 0) ok = !failed() && tc::mbar_wait(&acc_empty[b], (uint32_t)((v - 1) & 1), kWaitNs);
        if (!ok) break;
        tc::fence_after_sync();
        const uint32_t d = tmem + (uint32_t)(b * 256);
        for (int k0 = 0, c = 0; k0 < g.K; k0 += kGemmKC, ++q, ++c) {
          const int s = q % kWsStages, u = q / kWsStages;
          ok = !failed() && tc::mbar_wait(&full[s], (uint32_t)(u & 1), kWaitNs);
          if (!ok) break;
          tc::fence_after_sync();
          const uint64_t ad = tc::smem_desc_sw128(tc::smem_u32(stage_a(s)));
          const uint64_t bd = tc::smem_desc_sw128(tc::smem_u32(stage_b(s)));
#pragma unroll
          for (int kk = 0; kk < kGemmKC / 16; ++kk)
            tc::mma_bf16(d, ad + 2u * kk, bd + 2u * kk, idesc, (c | kk) ? 1u : 0u);
          tc::mma_commit(&empty[s]);
          s_last_q = q;
        }
        if (!ok) break;
        tc::mma_commit(&acc_full[b]);
      }
      if (!ok) atomicExch(&s_fail, 1);
    }
    __syncwarp();
  } else {
    // ---- epilogue ----
    const int quarter = warp & 3;            // the TMEM lanes this warp may read
    const int j0 = (warp - 2) >> 2;          // its column groups: j0, j0 + kWsGroupStride, ...
    const int n_groups = n_pad / 16;
    const EpiVec ev = epi_vec(g);
    unsigned char* stg = ring + kWsStages * kWsStageBytes + (warp - 2) * 2 * kStgBytes;
    int gi = 0;
    int i = 0;
    for (int item = blockIdx.x; item < m_tiles; item += gridDim.x, ++i) {
      const int b = i & 1, v = i >> 1;
      const bool ok = __all_sync(all, !failed() && tc::mbar_wait(&acc_full[b], (uint32_t)(v & 1), kWaitNs));
      if (!ok) {
        if (lane == 0) atomicExch(&s_fail, 1);
        break;
      }
      tc::fence_after_sync();
      const uint32_t tacc = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * 256);
      const int mrow0 = item * 128 + quarter * 32;
      const int m = mrow0 + lane;
      if (g.op == EPI_STORE)
        ws_epilogue<EPI_STORE>(g, ev, tacc, m, mrow0, j0, n_groups, &tmOut, tma_out != 0, stg, gi);
      else
        ws_epilogue<EPI_BIAS_GELU>(g, ev, tacc, m, mrow0, j0, n_groups, &tmOut, tma_out != 0, stg, gi);
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&acc_empty[b]);
    }
    // every TMA store of this warp has completed before its staging buffers go away
    if (lane == 0) tc::bulk_wait_all();
    __syncwarp();
  }
  tc::fence_before_sync();
  __syncthreads();
  if (s_fail && threadIdx.x == 0) {
    if (g.err) atomicCAS(g.err, 0, ERR_MMA_TIMEOUT);
    // let the copies and MMAs already issued finish (bounded) before shared and tensor memory go away
    for (int s = 0; s < kWsStages; ++s)
      if (s_armed[s] >= 0) tc::mbar_wait(&full[s], (uint32_t)(s_armed[s] & 1), kWaitNs);
    const int q = s_last_q;
    if (q >= 0) tc::mbar_wait(&empty[q % kWsStages], (uint32_t)((q / kWsStages) & 1), kWaitNs);
  }
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link against the driver library).
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }();
  return fn;
}

// A tiled tensor map of `rank` dimensions (dims innermost first, strides in bytes for dimensions 1..),
// elements outside the tensor read as zero and are not written.
bool encode_map(CUtensorMap* map, CUtensorMapDataType type, int rank, const void* base, const cuuint64_t* dims,
                const cuuint64_t* strides, const cuuint32_t* box, CUtensorMapSwizzle swizzle) {
  const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc || (reinterpret_cast<uintptr_t>(base) & 15) != 0) return false;
  for (int d = 0; d + 1 < rank; ++d)
    if (strides[d] % 16 != 0) return false;
  const cuuint32_t elem[3] = {1, 1, 1};
  return enc(map, type, (cuuint32_t)rank, const_cast<void*>(base), dims, strides, box, elem,
             CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The {k, row} view of a row-major BF16 matrix (rows x K, row stride ld elements) in 64 x box_rows boxes
// with 128-byte swizzling.
static bool encode_operand(CUtensorMap* map, const __nv_bfloat16* base, int rows, int K, long long ld, int box_rows) {
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2u};
  const cuuint32_t box[2] = {(cuuint32_t)kGemmKC, (cuuint32_t)box_rows};
  return encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

// Tensor map of the epilogue's output (32-row x 16-column boxes, laid out as the staging buffers are), if it has one.
static bool encode_output(const GemmArgs& g, CUtensorMap* map) {
  const bool f32 = g.op == EPI_STORE;
  if ((f32 ? g.scn : g.shn) != 1) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)g.N, (cuuint64_t)g.M};
  const cuuint64_t strides[1] = {f32 ? (cuuint64_t)g.scm * 4u : (cuuint64_t)g.shm * 2u};
  const cuuint32_t box[2] = {16, 32};
  return f32 ? encode_map(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, g.C, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_64B)
             : encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, g.H, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_32B);
}

cudaError_t launch_gemm(const GemmArgs& g, cudaStream_t stream) {
  if (g.N < 1 || g.N > 256 || g.M < 1 || g.K < 1) return cudaErrorInvalidValue;
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGemmSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_ws_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWsSmem);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  if (gemm_vectorised(g)) {
    const int n_pad = (g.N + 15) & ~15;
    CUtensorMap tmA, tmB;
    if (encode_operand(&tmA, g.A, g.M, g.K, g.sam, 128) && encode_operand(&tmB, g.B, g.N, g.K, g.sbn, n_pad)) {
      // persistent: one CTA per SM over the row tiles
      const int m_tiles = (g.M + 127) / 128;
      int dev = 0, n_sm = 0;
      cudaError_t e = cudaGetDevice(&dev);
      if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess) return e;
      CUtensorMap out{};
      const int tma_out = encode_output(g, &out);
      gemm_ws_kernel<<<m_tiles < n_sm ? m_tiles : n_sm, kWsThreads, kWsSmem, stream>>>(tmA, tmB, out, tma_out, g, m_tiles);
      count_launch();
      return cudaGetLastError();
    }
  }
  gemm_kernel<<<(g.M + 127) / 128, 128, kGemmSmem, stream>>>(g);
  count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// features, Adam, learned start
// ---------------------------------------------------------------------------

__global__ void mlp_features_kernel(SceneDev S, BatchDev B, float inv_scale, __nv_bfloat16* X, float* G) {
  for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < B.n_paths;
       k += (uint64_t)gridDim.x * blockDim.x) {
    PathDesc d;
    decode_global(B, k, d);
    path_features(S, d, inv_scale, X + k * kMlpIn, G ? G + k * 12 : nullptr);
  }
}

// One Adam step; the updated weights' BF16 copies go straight into every layout that reads them, and one thread
// adds the batch's loss to its epoch's mean.
__global__ void adam_kernel(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                            float* __restrict__ g, float lr, float c1, float c2, __nv_bfloat16* __restrict__ wb,
                            __nv_bfloat16* __restrict__ wt, __nv_bfloat16* __restrict__ wtT, float* __restrict__ loss,
                            float* hist, float hist_w, int clear) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  // Not only the gradient and the loss, the weights and moments too are loaded after the wait.  The last step's Adam has
  // completed by the time this one is launched, but that its writes are visible here is promised only by this grid's own
  // wait.  (Loaded before it, while the weight gradients ran, they slowed those down: one epoch of 524,288
  // samples 2.30 ms, 2.22 so.)
  wait_previous();
  launch_dependents();  // the next step's CTAs set up and gather their rows
  if (i == 0 && hist) *hist += hist_w * *loss;
  if (i == 0 && clear) *loss = 0.f;
  if (i >= kMlpParams) return;
  const float gi = g[i], m0 = m[i], v0 = v[i], w0 = w[i];
  if (clear) g[i] = 0.f;
  const float mi = 0.9f * m0 + 0.1f * gi;
  const float vi = 0.999f * v0 + 0.001f * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float wi = w0 - lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
  w[i] = wi;
  const __nv_bfloat16 b = __float2bfloat16(wi);
  wb[i] = b;
  tile_weight(i, b, wt, wtT);
}

__global__ void mlp_tile_weights_kernel(const __nv_bfloat16* __restrict__ wb, __nv_bfloat16* __restrict__ wt,
                                        __nv_bfloat16* __restrict__ wtT) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < kMlpParams) tile_weight(i, wb[i], wt, wtT);
}

__global__ void to_bf16_kernel(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    dst[i] = __float2bfloat16(src[i]);
}

static unsigned grid_1d(uint64_t n, int threads, int cap) {
  uint64_t g = (n + threads - 1) / threads;
  return (unsigned)(g < (uint64_t)cap ? (g ? g : 1) : (uint64_t)cap);
}

cudaError_t launch_mlp_features(const SceneDev& S, const BatchDev& B, float inv_scale, __nv_bfloat16* X, float* G,
                                cudaStream_t stream) {
  if (!B.n_paths) return cudaSuccess;
  mlp_features_kernel<<<grid_1d(B.n_paths, 128, 4096), 128, 0, stream>>>(S, B, inv_scale, X, G);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_adam(float* w, float* m, float* v, float* g, float lr, float c1, float c2, __nv_bfloat16* wb,
                        __nv_bfloat16* wt, __nv_bfloat16* wtT, float* loss, float* hist, float hist_w, int clear,
                        cudaStream_t stream) {
  const cudaError_t e = launch_overlapped(adam_kernel, (kMlpParams + 255) / 256, 256, 0, stream, w, m, v, g, lr, c1, c2, wb,
                                          wt, wtT, loss, hist, hist_w, clear);
  count_launch();
  return e;
}

cudaError_t launch_mlp_tile_weights(const __nv_bfloat16* wb, __nv_bfloat16* wt, __nv_bfloat16* wtT,
                                    cudaStream_t stream) {
  mlp_tile_weights_kernel<<<(kMlpParams + 255) / 256, 256, 0, stream>>>(wb, wt, wtT);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_to_bf16(const float* src, __nv_bfloat16* dst, int n, cudaStream_t stream) {
  to_bf16_kernel<<<grid_1d(n, 256, 1024), 256, 0, stream>>>(src, dst, n);
  count_launch();
  return cudaGetLastError();
}

// Check of the bounded waits that every tensor-core kernel here relies on.  Thread 0 initialises an
// mbarrier that expects one arrival; unless `arrive` is set, nothing ever arrives on it, so its phase
// never completes.  The wait gives up after `limit_ns` and records ERR_MMA_TIMEOUT in the error word,
// the same path a GEMM or inference CTA takes when an MMA or a TMA copy does not complete.
// `elapsed` (optional) receives the nanoseconds the wait took.
__global__ void bounded_wait_check_kernel(uint32_t limit_ns, int arrive, int* err, unsigned long long* elapsed) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x != 0) return;
  tc::mbar_init(&bar, 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if (arrive) tc::mbar_arrive(&bar);
  const uint64_t t0 = tc::global_ns();
  const bool ok = tc::mbar_wait(&bar, 0u, limit_ns);
  const uint64_t t1 = tc::global_ns();
  if (!ok && err) atomicCAS(err, 0, ERR_MMA_TIMEOUT);
  if (elapsed) *elapsed = (unsigned long long)(t1 - t0);
}

cudaError_t launch_bounded_wait_check(uint32_t limit_ns, int arrive, int* err, unsigned long long* elapsed,
                                      cudaStream_t stream) {
  if (limit_ns < 1 || limit_ns > kWaitNs) return cudaErrorInvalidValue;
  bounded_wait_check_kernel<<<1, 32, 0, stream>>>(limit_ns, arrive, err, elapsed);
  count_launch();
  return cudaGetLastError();
}

}  // namespace fpt
