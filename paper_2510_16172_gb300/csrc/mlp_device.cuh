// mlp_device.cuh -- device code shared by the network's kernels (k_mlp.cu, k_infer.cu, k_train.cu): GELU,
// column sums, the features of a path, the starting parameters from the network's outputs, the order of the
// training samples, the weights' layouts.
#pragma once

#include <cuda_bf16.h>

#include "fpt_device.cuh"
#include "mlp.h"
#include "tc.cuh"

namespace fpt {

constexpr uint32_t kWaitNs = 1000000000u;   // mbarrier waits give up after 1 s
constexpr int ERR_MMA_TIMEOUT = 3;

// GELU in its tanh form (Hendrycks and Gimpel, arXiv:1606.08415):
//   gelu(z) = z/2 (1 + tanh(u)),  u = sqrt(2/pi) (z + 0.044715 z^3),
// with the hardware tanh approximation (PTX tanh.approx.f32, relative error
// about 2^-11, below the BF16 rounding that follows every activation).  One
// MUFU operation per activation: the epilogues of the inference kernel
// evaluate 768 of them per path.
__device__ __forceinline__ float tanh_approx(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// u = z (K0 + K0 K1 z^2) and gelu = h + h tanh(u) with h = z/2: six operations.
constexpr float kGeluK0 = 0.79788456080286536f;  // sqrt(2 / pi)
constexpr float kGeluK1 = 0.044715f;
constexpr float kGeluK01 = 0.0356774081363001f;  // K0 K1
__device__ __forceinline__ float gelu(float z) {
  const float h = 0.5f * z;
  return fmaf(h, tanh_approx(z * fmaf(kGeluK01, z * z, kGeluK0)), h);
}

// Sum of x[i] over the warp's 32 lanes for each of the 16 columns i: a transposing butterfly (16 shuffles).
// Returns the sum of column ((lane >> 1) & 8) | ((lane >> 1) & 4) | ((lane >> 1) & 2) | ((lane >> 1) & 1),
// i.e. column lane / 2 in bit-reversed halves: lane bits 4, 3, 2, 1 select column bits 3, 2, 1, 0.
__device__ __forceinline__ float warp_colsum16(const float (&x)[16], int lane) {
  float a[8], b[4], c[2];
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4, h2 = lane & 2;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float send = h16 ? x[i] : x[i + 8];
    const float keep = h16 ? x[i + 8] : x[i];
    a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float send = h8 ? a[i] : a[i + 4];
    const float keep = h8 ? a[i + 4] : a[i];
    b[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float send = h4 ? b[i] : b[i + 2];
    const float keep = h4 ? b[i + 2] : b[i];
    c[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  const float d = (h2 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, h2 ? c[0] : c[1], 2);
  return d + __shfl_xor_sync(0xffffffffu, d, 1);
}
__device__ __forceinline__ int warp_colsum16_column(int lane) {
  return ((lane >> 1) & 8) | ((lane >> 1) & 4) | ((lane >> 1) & 2) | ((lane >> 1) & 1);
}

// 64 features of one path (see include/fpt.h): origin o = (TX + RX)/2, scale S;
// per interaction the orthogonal projections of TX and RX onto the object's
// affine hull in its own parameters, their distances to it, the first basis
// length, and the distance-weighted combination of the two projections.  Also
// the per-slot Gram matrix A^T A / S^2 (g11, g12, g22) of the loss.
__device__ __forceinline__ void path_features(const SceneDev& S, const PathDesc& d, float inv_scale,
                                              __nv_bfloat16* f, float* G) {
  float tx[3], rx[3], o[3];
  float txl[3], rxl[3];
  load_pair3(S.tx32 + kEnd32 * d.tx, tx, txl);
  load_pair3(S.rx32 + kEnd32 * d.rx, rx, rxl);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    tx[c] += txl[c];
    rx[c] += rxl[c];
    o[c] = 0.5f * (tx[c] + rx[c]);
  }
  float v[kMlpIn], gram[12];
#pragma unroll
  for (int k = 0; k < kMlpIn; ++k) v[k] = 0.f;
#pragma unroll
  for (int k = 0; k < 12; ++k) gram[k] = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    v[c] = (tx[c] - o[c]) * inv_scale;
    v[3 + c] = (rx[c] - o[c]) * inv_scale;
  }
  const bool valid = !(d.flags & ST_INVALID);
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    if (s < d.n && valid) {
      const bool edge = S.aux[kAux * d.ids[s] + 2] != 0.f;
      float b[3], bl[3], a1[3], a2[3];
      load_rec32(S.rec32 + kRec32 * d.ids[s], b, bl, a1, a2);
#pragma unroll
      for (int c = 0; c < 3; ++c) b[c] += bl[c];
      const float g11 = a1[0] * a1[0] + a1[1] * a1[1] + a1[2] * a1[2];
      const float g12 = a1[0] * a2[0] + a1[1] * a2[1] + a1[2] * a2[2];
      const float g22 = a2[0] * a2[0] + a2[1] * a2[1] + a2[2] * a2[2];
      const float det = g11 * g22 - g12 * g12;
      float tau[2][2], dist[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float* pt = q == 0 ? tx : rx;
        float rr[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) rr[c] = pt[c] - b[c];
        const float c1 = a1[0] * rr[0] + a1[1] * rr[1] + a1[2] * rr[2];
        const float c2 = a2[0] * rr[0] + a2[1] * rr[1] + a2[2] * rr[2];
        if (edge) {
          tau[q][0] = c1 / g11;
          tau[q][1] = 0.f;
        } else {
          tau[q][0] = (g22 * c1 - g12 * c2) / det;
          tau[q][1] = (g11 * c2 - g12 * c1) / det;
        }
        float e2 = 0.f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float e = rr[c] - tau[q][0] * a1[c] - tau[q][1] * a2[c];
          e2 += e * e;
        }
        dist[q] = sqrtf(e2) * inv_scale;
      }
      const int base = 6 + 11 * s;
      v[base] = 1.f;
      v[base + 1] = edge ? 1.f : 0.f;
      v[base + 2] = tau[0][0];
      v[base + 3] = tau[0][1];
      v[base + 4] = tau[1][0];
      v[base + 5] = tau[1][1];
      v[base + 6] = dist[0];
      v[base + 7] = dist[1];
      v[base + 8] = sqrtf(g11) * inv_scale;
      const float dsum = dist[0] + dist[1];
#pragma unroll
      for (int k = 0; k < 2; ++k)
        v[base + 9 + k] = dsum > 0.f ? (dist[1] * tau[0][k] + dist[0] * tau[1][k]) / dsum
                                     : 0.5f * (tau[0][k] + tau[1][k]);
      const float is2 = inv_scale * inv_scale;
      gram[3 * s] = g11 * is2;
      gram[3 * s + 1] = g12 * is2;
      gram[3 * s + 2] = g22 * is2;
    }
  }
#pragma unroll
  for (int k = 0; k < kMlpIn; k += 8) {
    __nv_bfloat16 e[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) e[q] = __float2bfloat16(v[k + q]);
    *reinterpret_cast<uint4*>(f + k) = *reinterpret_cast<uint4*>(e);
  }
  if (G)
#pragma unroll
    for (int k = 0; k < 12; ++k) G[k] = gram[k];
}

// Starting parameters of a path of order n from the network's outputs y (slots 1-4; an edge's
// second parameter -- bit s of `edges` -- and the later slots start at 1/2, and so does an output
// that is not finite or beyond 1e3, and every slot of an invalid sequence).  The slot loop runs over
// compile-time indices so that y stays in registers.
__device__ __forceinline__ void write_start(int n, bool use, unsigned edges, const float (&y)[8], float2* To) {
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    if (s < n) {
      float t0 = 0.5f, t1 = 0.5f;
      if (use) {
        if (isfinite(y[2 * s]) && fabsf(y[2 * s]) < 1e3f) t0 = y[2 * s];
        if (!((edges >> s) & 1u) && isfinite(y[2 * s + 1]) && fabsf(y[2 * s + 1]) < 1e3f) t1 = y[2 * s + 1];
      }
      To[s] = make_float2(t0, t1);
    }
  }
  for (int s = 4; s < n; ++s) To[s] = make_float2(0.5f, 0.5f);
}

// bit s: slot s (s < 4) of the path is an edge
__device__ __forceinline__ unsigned edge_mask(const SceneDev& S, const PathDesc& d) {
  unsigned m = 0;
#pragma unroll
  for (int s = 0; s < 4; ++s)
    if (s < d.n && S.aux[kAux * d.ids[s] + 2] != 0.f) m |= 1u << s;
  return m;
}

// Training data order: a seeded pseudo-random permutation of [0, n) per epoch, evaluated index by index
// (a four-round Feistel network on 2h-bit words, 2^(2h) >= n, with cycle walking back into [0, n)).
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

__device__ __forceinline__ uint64_t feistel(uint64_t x, int h, uint64_t key) {
  const uint64_t mask = (1ULL << h) - 1ULL;
  uint64_t l = x >> h, r = x & mask;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint64_t f = mix64(r ^ (key + 0x9E3779B97F4A7C15ULL * (uint64_t)(k + 1))) & mask;
    const uint64_t nl = r;
    r = l ^ f;
    l = nl;
  }
  return (l << h) | r;
}

// Position k of the permutation of [0, n) drawn by `key` (n >= 1).  The walk stays on k's cycle of the
// Feistel permutation, which holds k itself, so it returns a value below n; the bound only guards the loop.
__device__ __forceinline__ uint64_t perm_index(uint64_t k, uint64_t n, int h, uint64_t key) {
  uint64_t x = k;
  for (int i = 0; i < (1 << 20); ++i) {
    x = feistel(x, h, key);
    if (x < n) return x;
  }
  return k;
}

// Places of flat parameter i in the fused kernels' weight layouts (mlp.h) and its BF16 value there; biases have
// none.  fwd: outputs by rows, split by output; the output layer in both halves.  back: the transposes of
// layers 2-4, split by input.
__device__ __forceinline__ void tile_weight(int i, __nv_bfloat16 v, __nv_bfloat16* fwd, __nv_bfloat16* back) {
  uint32_t first, back_first = 0;
  int off, K;
  if (i < kOffB1) {
    off = kOffW1; K = kMlpIn; first = 0;
  } else if (i >= kOffW2 && i < kOffB2) {
    off = kOffW2; K = kMlpHidden; first = kMlpTileW2; back_first = kMlpTileW2t;
  } else if (i >= kOffW3 && i < kOffB3) {
    off = kOffW3; K = kMlpHidden; first = kMlpTileW3; back_first = kMlpTileW3t;
  } else if (i >= kOffW4 && i < kOffB4) {
    const int r = (i - kOffW4) >> 8, k = (i - kOffW4) & 255;
    const uint32_t byte = kMlpTileW4 + (uint32_t)(k >> 6) * kMlpW4Chunk + tc::sw128_offset(r, k & 63);
    fwd[byte / 2] = v;
    fwd[(kMlpHalfBytes + byte) / 2] = v;
    back[((uint32_t)(k >> 7) * kMlpHalfTBytes + kMlpTileW4t + tc::kmajor_offset(k & 127, r, kMlpOut)) / 2] = v;
    return;
  } else {
    return;
  }
  const int r = (i - off) / K, k = (i - off) % K;
  fwd[((uint32_t)(r >> 7) * kMlpHalfBytes + first + (uint32_t)(k >> 6) * kMlpChunk +
       tc::sw128_offset(r & 127, k & 63)) / 2] = v;
  if (K == kMlpHidden)
    back[((uint32_t)(k >> 7) * kMlpHalfTBytes + back_first + (uint32_t)(r >> 6) * kMlpChunk +
          tc::sw128_offset(k & 127, r & 63)) / 2] = v;
}

}  // namespace fpt
