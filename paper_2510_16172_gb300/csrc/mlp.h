// mlp.h -- host/device interface of the tensor-core kernels of the learned warm start.
#pragma once

#include <cstdint>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "fpt_kernels.h"

namespace fpt {

constexpr int kMlpIn = 64, kMlpHidden = 256, kMlpOut = 16;
// offsets of the parameter blocks in the flat FP32 vector
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + 256 * 64, kOffW2 = kOffB1 + 256, kOffB2 = kOffW2 + 256 * 256,
              kOffW3 = kOffB2 + 256, kOffB3 = kOffW3 + 256 * 256, kOffW4 = kOffB3 + 256, kOffB4 = kOffW4 + 16 * 256,
              kMlpParams = kOffB4 + 16;

enum EpilogueOp { EPI_STORE = 0, EPI_BIAS_GELU = 1 };

// D[M x N] = sum_k A(m, k) B(n, k); A(m, k) = A[m * sam + k * sak], B(n, k) = B[n * sbn + k * sbk].
struct GemmArgs {
  int M, N, K;
  const __nv_bfloat16* A;
  long long sam, sak;
  const __nv_bfloat16* B;
  long long sbn, sbk;
  int op;                 // EpilogueOp
  const float* bias;      // [N] or null
  float* C;               // EPI_STORE: FP32 output, D (+ bias)
  long long scm, scn;
  __nv_bfloat16* H;       // EPI_BIAS_GELU: BF16 activation
  long long shm, shn;
  int* err;               // device error word (MMA completion timeout)
};

// A tiled tensor map (false where the base or a stride does not allow one).
bool encode_map(CUtensorMap* map, CUtensorMapDataType type, int rank, const void* base, const cuuint64_t* dims,
                const cuuint64_t* strides, const cuuint32_t* box, CUtensorMapSwizzle swizzle);
cudaError_t launch_gemm(const GemmArgs& g, cudaStream_t stream);
// Features (and Gram entries, if G) of every path of a batch, by global index.
cudaError_t launch_mlp_features(const SceneDev& S, const BatchDev& B, float inv_scale, __nv_bfloat16* X, float* G,
                                cudaStream_t stream);
// One Adam step, with the BF16 copies of the parameters (plain and as launch_mlp_tile_weights lays them out); with
// hist, also *hist += hist_w * *loss; with clear, g and *loss are zero afterwards.
cudaError_t launch_adam(float* w, float* m, float* v, float* g, float lr, float c1, float c2, __nv_bfloat16* wb,
                        __nv_bfloat16* wt, __nv_bfloat16* wtT, float* loss, float* hist, float hist_w, int clear,
                        cudaStream_t stream);
cudaError_t launch_to_bf16(const float* src, __nv_bfloat16* dst, int n, cudaStream_t stream);
// The weights as the fused kernels' CTA pairs read them (k_infer.cu, k_train.cu): CTA r of a pair holds outputs
// 128 r .. 128 r + 127 of the hidden layers in chunks of 64 inputs, and the whole output layer; transposed, for the
// back-propagation, inputs 128 r .. 128 r + 127.  Chunks of 64 columns are K-major in the 128-byte swizzled layout
// (tc.cuh, sw128_offset, read through smem_desc_sw128); only the transposed output layer, 16 columns, is in core
// matrices (kmajor_offset, smem_desc).
constexpr uint32_t kMlpChunk = 128 * 64 * 2;   // 128 rows x 64 columns
constexpr uint32_t kMlpW4Chunk = 16 * 64 * 2;  // the output layer's 16 rows
constexpr uint32_t kMlpTileW2 = kMlpChunk, kMlpTileW3 = 5 * kMlpChunk, kMlpTileW4 = 9 * kMlpChunk;
constexpr uint32_t kMlpHalfBytes = 9 * kMlpChunk + 4 * kMlpW4Chunk;
constexpr uint32_t kMlpTileW3t = 0, kMlpTileW2t = 4 * kMlpChunk, kMlpTileW4t = 8 * kMlpChunk;
constexpr uint32_t kMlpHalfTBytes = 8 * kMlpChunk + 128 * 16 * 2;
// both from the BF16 parameter copy
cudaError_t launch_mlp_tile_weights(const __nv_bfloat16* wb, __nv_bfloat16* wt, __nv_bfloat16* wtT,
                                    cudaStream_t stream);
// Loss and gradient of B rows (two launches).  Row i is sample perm(first + i) of n when n > 0 (perm = the seeded
// permutation of [0, n) drawn by key), else sample i.  grad and loss are added to.  Scratch: the rows' features
// [B][64], hidden activations and gradients at the hidden layers' outputs [3][B][256], transposed gradient at the
// outputs [16][ldY] (ldY >= B, a multiple of 8).
struct TrainArgs {
  const __nv_bfloat16* X;
  const float* T;
  const float* G;
  uint64_t B, n, first, key;
  const __nv_bfloat16 *wt, *wtT;
  const float* params;
  __nv_bfloat16 *Xb, *H, *dZ, *dYt;
  uint64_t ldY;
  float *grad, *loss;
  int* err;
  int chained;           // the previous launch on the stream is the last step's Adam, which left grad and loss at zero
  int h, vec_x, vec_tg;  // set by the launch: half the permutation's bits, 16-byte alignment of X, of T and G
};
cudaError_t launch_mlp_train(const TrainArgs& a, cudaStream_t stream, int n_sm);
// The learned start of `count` paths: of order n of an exhaustive batch (list == nullptr), or of a list of
// records, all of orders up to kMaxBfgsOrder (n any of them) or all above (n > kMaxBfgsOrder).  Slots from a
// path's order to n_fill are set to zero.
cudaError_t launch_mlp_infer(const SceneDev& S, const BatchDev& B, int n, const PathRec* list, uint64_t count,
                             float inv_scale, const __nv_bfloat16* wt, const float* params, float* T, int n_fill,
                             int* err, cudaStream_t stream, int n_sm);
// One CTA waits, for at most `limit_ns` (1 ns .. 1 s), on an mbarrier that receives an arrival only
// when `arrive` != 0; a wait that runs out sets *err (if 0) to the MMA-timeout code.  `elapsed`
// (device, optional) receives the wait's duration in nanoseconds of the global timer.
cudaError_t launch_bounded_wait_check(uint32_t limit_ns, int arrive, int* err, unsigned long long* elapsed,
                                      cudaStream_t stream);

}  // namespace fpt
