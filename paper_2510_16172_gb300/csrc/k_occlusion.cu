// k_occlusion.cu -- obstruction test of solved paths against the scene's planar objects.
//
// Sec. I: a candidate ray is discarded when it is obstructed, as well as when an
// interaction point falls outside its object (the validity bit).  For segment j
// of a path of order n, from x_j to x_{j+1} (x_0 = TX, x_{n+1} = RX), every
// planar object other than the objects at the segment's two ends is tested: the
// segment is blocked when its ends lie on opposite sides of the object's plane,
// each more than `tol` metres from it, and the crossing point lies in the closed
// parallelogram.  Edges (lines) block nothing.  One thread per path; the
// occluders' records (centred origin, unit normal and the dual basis that gives
// the in-plane coordinates u = d1 . (h - b), v = d2 . (h - b)) are staged in
// shared memory and every thread of a warp walks them in the same order.  Per occluder the signed distances of all
// n + 2 points are formed once, each serving the two segments that meet there, and only the segments that cross
// the plane go on to the crossing point; the kernel is bound by instruction issue (8.4 M canyon paths, 0.55 M of
// them tested, select and test together: 144 -> 95 us).  When
// only paths with given status bits are tested (typically the few per cent
// that are valid and solved), a first kernel lists them and writes zero for
// the rest, so that the test kernel's warps run full.
#include "fpt_kernels.h"

namespace fpt {

// List the paths of a slice that hold the status bits (local indices); zero the others' masks.  A CTA
// takes kOccSelPer consecutive local indices per thread and appends its chunk in index order with a
// single atomic on the list counter, which one atomic per warp would turn into a serial hot spot.
constexpr int kOccSelThreads = 256, kOccSelPer = 16, kOccSelChunk = kOccSelThreads * kOccSelPer;
__global__ void __launch_bounds__(kOccSelThreads) occlusion_select_kernel(BatchDev B, int n, const PathRec* list,
                                                                          uint64_t n_local,
                                                                          const uint8_t* __restrict__ status,
                                                                          uint8_t mask, uint16_t* __restrict__ blocked,
                                                                          uint32_t* __restrict__ sel,
                                                                          unsigned* __restrict__ sel_count) {
  for (uint64_t c0 = (uint64_t)blockIdx.x * kOccSelChunk; c0 < n_local; c0 += (uint64_t)gridDim.x * kOccSelChunk) {
    const uint64_t j0 = c0 + (uint64_t)threadIdx.x * kOccSelPer;
    unsigned bits = 0;
    SliceWalk walk;
    bool whole = false;  // the thread's 16 statuses read with one load, its 16 masks cleared with two stores
    if (list == nullptr && j0 + kOccSelPer <= n_local) {
      // exhaustive batch: 16 consecutive paths of one TX/RX pair, on 16-byte boundaries.  The masks of the listed
      // paths are cleared too; the test kernel writes them afterwards.
      SliceWalk w0;
      const uint64_t g0 = w0.next(B, n, j0);
      whole = w0.left + 1 >= (uint64_t)kOccSelPer &&
              ((reinterpret_cast<uintptr_t>(status + g0) | reinterpret_cast<uintptr_t>(blocked + g0)) & 15u) == 0;
      if (whole) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(status + g0));
        const uint32_t wd[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < kOccSelPer; ++k) {
          const uint8_t st = (uint8_t)(wd[k >> 2] >> (8 * (k & 3)));
          bits |= (!(st & ST_SKIP) && (st & mask) == mask ? 1u : 0u) << k;
        }
        uint4* out = reinterpret_cast<uint4*>(blocked + g0);
        out[0] = out[1] = make_uint4(0u, 0u, 0u, 0u);
      }
    }
#pragma unroll 4
    for (int k = 0; k < kOccSelPer && !whole; ++k) {
      const uint64_t j = j0 + k;
      if (j >= n_local) break;
      // the solver wrote the sequence's REPEAT / INVALID_INPUT bits into its status
      const uint64_t g = list != nullptr ? slice_global(B, n, list, j) : walk.next(B, n, j);
      const uint8_t st = status[g];
      const bool take = !(st & ST_SKIP) && (st & mask) == mask;
      if (!take) blocked[g] = 0;
      bits |= (take ? 1u : 0u) << k;
    }
    cta_append_ordered<kOccSelThreads>(bits, j0, sel, sel_count);
  }
}

// Occluder records in shared memory: three 16-byte words each (origin, normal, d1, d2), the ids behind them.
constexpr int kOccWords = kOcc - 1;
static_assert(kOccWords == 12, "three 16-byte words");

// Test the order-N paths of a slice (sel == nullptr) or the listed ones.
template <int N>
__global__ void __launch_bounds__(kThreads) occlusion_kernel(SceneDev S, BatchDev B, const PathRec* list,
                                                             uint64_t n_local, const float* __restrict__ T,
                                                             const uint32_t* __restrict__ sel,
                                                             const unsigned* __restrict__ sel_count,
                                                             const float* __restrict__ occ, int n_occ, float tol,
                                                             uint16_t* __restrict__ blocked) {
  extern __shared__ __align__(16) float s_occ[];
  for (int k = threadIdx.x; k < n_occ * kOcc; k += blockDim.x) {
    const int o = k / kOcc, f = k % kOcc;
    s_occ[f < kOccWords ? o * kOccWords + f : n_occ * kOccWords + o] = occ[k];
  }
  __syncthreads();
  constexpr unsigned kAll = (2u << N) - 1u;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t n_iter = sel ? (uint64_t)*sel_count : n_local;
  for (uint64_t k0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k0 < n_iter; k0 += stride) {
    const uint64_t j = sel ? (uint64_t)sel[k0] : k0;
    PathDesc d;
    fetch_path_n<N>(B, list, j, d);
    unsigned bits = 0;  // blocked segments
    if (!(d.flags & ST_SKIP)) {
      // the points x_0 .. x_{n+1}, relative to the scene centre
      const float2* Tp = reinterpret_cast<const float2*>(T) + d.g * (uint64_t)B.n_max;
      float x[N + 2][3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        x[0][c] = S.tx32[kEnd32 * d.tx + c] + S.tx32[kEnd32 * d.tx + 3 + c];
        x[N + 1][c] = S.rx32[kEnd32 * d.rx + c] + S.rx32[kEnd32 * d.rx + 3 + c];
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const float* r = S.rec32 + kRec32 * d.ids[i];
        const float2 t = Tp[i];
#pragma unroll
        for (int c = 0; c < 3; ++c) x[i + 1][c] = fmaf(r[9 + c], t.y, fmaf(r[6 + c], t.x, r[c] + r[3 + c]));
      }
      for (int k = 0; k < n_occ && bits != kAll; ++k) {
        const float4* o = reinterpret_cast<const float4*>(s_occ + kOccWords * k);
        const float4 o0 = o[0], o1 = o[1];  // origin (3), normal (3), d1, d2
        float dist[N + 2];
#pragma unroll
        for (int i = 0; i < N + 2; ++i)
          dist[i] = fmaf(o1.y, x[i][2] - o0.z, fmaf(o1.x, x[i][1] - o0.y, o0.w * (x[i][0] - o0.x)));
        // segments whose ends lie on opposite sides, each more than tol away, not blocked yet
        unsigned cross = 0;
#pragma unroll
        for (int i = 0; i <= N; ++i)
          if (fminf(dist[i], dist[i + 1]) < -tol && fmaxf(dist[i], dist[i + 1]) > tol) cross |= 1u << i;
        cross &= ~bits;
        if (!cross) continue;
        const int id = __float_as_int(s_occ[kOccWords * n_occ + k]);
#pragma unroll
        for (int i = 0; i < N; ++i)
          if (d.ids[i] == id) cross &= ~(3u << i);  // an object blocks neither segment that ends on it
        const float4 o2 = o[2];
#pragma unroll
        for (int i = 0; i <= N; ++i) {
          if (!((cross >> i) & 1u)) continue;
          const float pb0 = x[i][0] - o0.x, pb1 = x[i][1] - o0.y, pb2 = x[i][2] - o0.z;
          const float qb0 = x[i + 1][0] - o0.x, qb1 = x[i + 1][1] - o0.y, qb2 = x[i + 1][2] - o0.z;
          const float s = dist[i] / (dist[i] - dist[i + 1]);
          const float h0 = fmaf(s, qb0 - pb0, pb0), h1 = fmaf(s, qb1 - pb1, pb1), h2 = fmaf(s, qb2 - pb2, pb2);
          const float u = fmaf(o2.x, h2, fmaf(o1.w, h1, o1.z * h0));
          const float v = fmaf(o2.w, h2, fmaf(o2.z, h1, o2.y * h0));
          if (u >= 0.f && u <= 1.f && v >= 0.f && v <= 1.f) bits |= 1u << i;
        }
      }
    }
    blocked[d.g] = (uint16_t)bits;
  }
}

template <int N>
cudaError_t launch_occlusion_n(const SceneDev& S, const BatchDev& B, const PathRec* list, uint64_t n_local,
                               const float* T, const uint32_t* sel, const unsigned* sel_count, const float* occ,
                               int n_occ, float tol, uint16_t* blocked, cudaStream_t stream, int n_sm) {
  const size_t smem = (size_t)n_occ * kOcc * sizeof(float);
  if (smem > kMaxSmemBytes) return cudaErrorInvalidValue;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(occlusion_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  // a listed launch strides over the list; a full grid covers the largest list
  unsigned grid = 0;
  const cudaError_t e = strided_grid(occlusion_kernel<N>, kThreads, smem, n_local, n_sm, grid);
  if (e != cudaSuccess || grid == 0) return e;
  occlusion_kernel<N><<<grid, kThreads, smem, stream>>>(S, B, list, n_local, T, sel, sel_count, occ, n_occ, tol, blocked);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_occlusion(const SceneDev& S, const BatchDev& B, int n, const PathRec* list, uint64_t n_local,
                             const float* T, const uint8_t* status, uint8_t mask, const float* occ, int n_occ,
                             float tol, uint16_t* blocked, uint32_t* sel, unsigned* sel_count, cudaStream_t stream,
                             int n_sm) {
  const bool listed = status != nullptr && mask != 0;
  if (listed) {
    if (!sel || !sel_count) return cudaErrorInvalidValue;
    const uint64_t want = (n_local + kOccSelChunk - 1) / kOccSelChunk;
    const unsigned g = (unsigned)(want < (uint64_t)n_sm * 8 ? want : (uint64_t)n_sm * 8);
    if (g == 0) return cudaSuccess;
    occlusion_select_kernel<<<g, kOccSelThreads, 0, stream>>>(B, n, list, n_local, status, mask, blocked, sel,
                                                              sel_count);
    count_launch();
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  switch (n) {
#define FPT_OCC_CASE(K) \
  case K:               \
    return launch_occlusion_n<K>(S, B, list, n_local, T, listed ? sel : nullptr, listed ? sel_count : nullptr, occ, n_occ, tol, blocked, stream, n_sm);
    FPT_OCC_CASE(1)
    FPT_OCC_CASE(2)
    FPT_OCC_CASE(3)
    FPT_OCC_CASE(4)
    FPT_OCC_CASE(5)
    FPT_OCC_CASE(6)
    FPT_OCC_CASE(7)
    FPT_OCC_CASE(8)
    FPT_OCC_CASE(9)
    FPT_OCC_CASE(10)
#undef FPT_OCC_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fpt
