// fpt_api.cu -- host implementation of the C ABI declared in include/fpt.h.
//
// Owns contexts (device, stream, error word, workspace), scenes (object
// records built in FP64 on the host, recentred, split into FP32 hi/lo parts
// and uploaded) and batches (candidate-sequence descriptions; seeded and
// explicit batches are bucketed by order on the device once, so that every
// solver launch is specialised to one order).
#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <new>
#include <utility>
#include <vector>

#include "fpt.h"
#include "fpt_kernels.h"
#include "mlp.h"

using namespace fpt;

// Streams over which the BFGS pattern launches of one order are spread (a
// build-time tuning constant: more streams overlap the launches' tails, but
// co-resident kernels share each SM's instruction cache).
#ifndef FPT_SIDE_STREAMS
#define FPT_SIDE_STREAMS 4
#endif

// Device scratch of a context, grown when a call needs more (reserve).
struct Scratch {
  void* p = nullptr;
  size_t cap = 0;         // bytes
  bool captured = false;  // a stream capture has recorded launches that use it
};

struct fpt_ctx {
  int device = 0;
  int n_sm = 0;
  cudaStream_t stream = nullptr;
  int* d_err = nullptr;                    // device error word
  Scratch gacc;                            // backward accumulators (FP64)
  Scratch tape;                            // per-step state of fpt_backward_unrolled
  unsigned long long* d_count = nullptr;   // counters for reductions
  unsigned char* d_ctl = nullptr;          // launch counters of the orders (OrderCtl), cleared once per call
  static constexpr int kSide = FPT_SIDE_STREAMS;  // streams for the independent pattern launches of one order
  cudaStream_t side[kSide] = {};           // created by the first call that needs them (side_streams)
  cudaEvent_t fork_ev = nullptr;
  cudaEvent_t join_ev[kSide] = {};
  // orders of one call that run side by side: the first on `stream`, the others dealt over these
  static constexpr int kOrderStreams = 4;
  cudaStream_t ostream[kOrderStreams] = {};
  cudaEvent_t ofork_ev = nullptr;
  cudaEvent_t ojoin_ev[kOrderStreams] = {};
  Scratch rescue;                          // path lists: FP64 polish, FP64 adjoint, second polish pass
  Scratch step;                            // first Newton steps of the second polish pass's paths
  std::vector<void*> kept;                 // outgrown scratch that captured graphs use
  unsigned* d_dropped = nullptr;           // paths the last backward left out (fpt_backward_dropped)
  fpt_mlp* init_mlp = nullptr;             // network for init_mode = 1
  int acc_flush_tiles = 64;                // backward sums: CTA tiles between flushes of the FP32 partial sums
  int acc_smem = 1;                        // backward sums: 1 = FP32 partial sums per CTA, 0 = straight to FP64
  char msg[512] = "ok";
  // kernel timing
  bool prof = false;
  std::vector<cudaEvent_t> ev_pool;
  std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> ev_pending;
  double prof_ms[FPT_K_COUNT] = {0, 0, 0, 0, 0};
  uint64_t prof_kernels[FPT_K_COUNT] = {0, 0, 0, 0, 0};
};

// Launch counters of one order, in context memory; a call clears the counters of all orders with one memset
// before its first launch.
struct OrderCtl {
  unsigned long long work[40];  // path counters of the lane-refill solver: one per pattern, 32: the small buckets
  unsigned polish64, adjoint64, stepped;  // entries of the polish's lists: FP64 polish, FP64 adjoint, second pass
  unsigned backward64, selected;          // entries of the backward's lists: FP64 adjoint, paths with a cotangent
  unsigned pad[3];
};
constexpr size_t kCtlBytes = (kMaxOrder + 1) * sizeof(OrderCtl);

// Event pair around the launches of one call when timing is on; counts the kernels launched in between.
struct ProfScope {
  fpt_ctx* ctx;
  int cls;
  uint64_t k0 = 0;
  cudaEvent_t a = nullptr, b = nullptr;
  static cudaEvent_t take(fpt_ctx* c) {
    cudaEvent_t e = nullptr;
    if (!c->ev_pool.empty()) {
      e = c->ev_pool.back();
      c->ev_pool.pop_back();
    } else if (cudaEventCreate(&e) != cudaSuccess) {
      e = nullptr;
    }
    return e;
  }
  ProfScope(fpt_ctx* c, int k) : ctx(c), cls(k) {
    if (!ctx->prof) return;
    k0 = tl_kernel_launches;
    a = take(ctx);
    b = take(ctx);
    if (a) cudaEventRecord(a, ctx->stream);
  }
  ~ProfScope() {
    if (!ctx->prof) return;
    ctx->prof_kernels[cls] += tl_kernel_launches - k0;
    if (!a || !b) return;
    cudaEventRecord(b, ctx->stream);
    ctx->ev_pending.push_back({cls, {a, b}});
  }
};

struct fpt_scene {
  fpt_ctx* ctx = nullptr;
  int n_obj = 0;
  std::vector<uint8_t> types;
  double centre[3] = {0, 0, 0};
  float* d_rec32 = nullptr;
  double* d_rec64 = nullptr;
  float* d_aux = nullptr;
  float* d_reclo = nullptr;
  int n_tx = 0, n_rx = 0;
  float* d_tx32 = nullptr;
  float* d_rx32 = nullptr;
  double* d_tx64 = nullptr;
  double* d_rx64 = nullptr;
  float* d_occ = nullptr;  // planar objects as occluders (kOcc floats each)
  int n_occ = 0;
  uint8_t* d_types = nullptr;      // object types and occluder slots (-1: edge), for records built on the device
  int32_t* d_occ_slot = nullptr;
  int tx_cap = 0, rx_cap = 0;      // endpoints the device buffers hold
  std::vector<int32_t> h_occ_slot;
  // host sources of the asynchronous uploads, kept until the device buffers are freed (cudaFree
  // waits for the device, so no copy from them is still pending when they go)
  std::vector<float> h_rec32, h_aux, h_reclo, h_occ, h_tx32, h_rx32;
  std::vector<double> h_rec64, h_tx64, h_rx64;
};

struct fpt_batch {
  fpt_ctx* ctx = nullptr;
  BatchDev dev{};
  int32_t* d_alphabet = nullptr;
  int32_t* d_type_pos = nullptr;  // alphabet positions of the reflectors, then of the edges
  std::vector<uint8_t> types;     // object types of the scene the batch was built for
  std::vector<int32_t> h_alphabet, h_type_pos;  // host sources of the uploads (as in fpt_scene)
  // (order, pattern) buckets of seeded / explicit batches (built on first use)
  bool bucketed = false;
  PathRec* d_lists = nullptr;
  uint64_t count[kPatternKeys] = {0};
  uint64_t start[kPatternKeys] = {0};
  // per order: the buckets too small for a pattern launch sit together at the end of the order's range
  uint64_t small_start[kMaxOrder + 1] = {0};
  uint64_t small_count[kMaxOrder + 1] = {0};
};

// Smallest bucket worth its own pattern launch: about four paths per resident lane.
static uint64_t min_pattern_bucket(const fpt_ctx* ctx) { return (uint64_t)ctx->n_sm * 4 * 128 * 4; }

static fpt_status fail(fpt_ctx* ctx, fpt_status st, const char* fmt, ...) {
  if (ctx) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(ctx->msg, sizeof(ctx->msg), fmt, ap);
    va_end(ap);
  }
  return st;
}

#define CUDA_OR_FAIL(ctx, call)                                                                    \
  do {                                                                                             \
    cudaError_t e_ = (call);                                                                       \
    if (e_ != cudaSuccess)                                                                         \
      return fail((ctx), FPT_ECUDA, "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
  } while (0)

struct fpt_mlp {
  fpt_ctx* ctx = nullptr;
  float scale = 1.f;
  uint64_t seed = 0;
  int64_t step = 0;
  float* d_w = nullptr;          // FP32 master parameters
  float* d_m = nullptr;          // Adam moments
  float* d_v = nullptr;
  float* d_g = nullptr;          // gradient
  __nv_bfloat16* d_wb = nullptr;  // BF16 copy used by the tensor cores
  __nv_bfloat16* d_wt = nullptr;   // the weights as the fused kernels read them (mlp.h),
  __nv_bfloat16* d_wtT = nullptr;  // and their transposes
  float* d_loss = nullptr;       // the batch's loss, behind the gradient (cleared with it)
  float* d_hist = nullptr;       // fpt_mlp_train: per-epoch mean losses
  size_t hist_cap = 0;
  // activations of two layers for a forward pass of up to cap rows, where those of a training batch do not serve
  Scratch fwd;
  uint64_t cap = 0;
  // operands of the weight gradients dW = dZ^T act for a training batch of up to train_cap rows: activations and
  // gradients of the three hidden layers, features, transposed gradient at the outputs
  Scratch train;
  uint64_t train_cap = 0;
  __nv_bfloat16* H() const { return static_cast<__nv_bfloat16*>(train.p); }
  __nv_bfloat16* dZ() const { return H() + 3 * train_cap * kMlpHidden; }
  __nv_bfloat16* Xb() const { return dZ() + 3 * train_cap * kMlpHidden; }
  __nv_bfloat16* dYt() const { return Xb() + train_cap * kMlpIn; }
};

static SceneDev scene_dev(const fpt_scene* s) {
  SceneDev d{};
  d.n_obj = s->n_obj;
  d.rec32 = s->d_rec32;
  d.rec64 = s->d_rec64;
  d.aux = s->d_aux;
  d.n_tx = s->n_tx;
  d.n_rx = s->n_rx;
  d.tx32 = s->d_tx32;
  d.rx32 = s->d_rx32;
  d.tx64 = s->d_tx64;
  d.rx64 = s->d_rx64;
  d.reclo = s->d_reclo;
  for (int c = 0; c < 3; ++c) {
    d.centre[c] = s->centre[c];
    d.centre_hi[c] = (float)s->centre[c];
    d.centre_lo[c] = (float)(s->centre[c] - (double)d.centre_hi[c]);
  }
  return d;
}

extern "C" {

void fpt_default_params(fpt_solve_params* p) {
  if (!p) return;
  std::memset(p, 0, sizeof(*p));
  p->max_iters = 64;
  p->fp_iters = 1;
  p->polish = 1;
  p->fixed_iters = 0;
  p->tol_step = 1e-4f;
  p->solved_tol = 1e-5f;
  p->deg_tol = 1e-3f;
  p->cond_fp64 = 1e-4f;
  p->init_mode = 0;
  p->polish_fp64 = 0;
  p->refill = 8;
  p->specialize = 1;
  p->polish_radius = 0.1f;
}

fpt_status fpt_create(fpt_ctx** out, int device, void* cuda_stream) {
  if (!out) return FPT_EINVAL;
  *out = nullptr;
  fpt_ctx* ctx = new (std::nothrow) fpt_ctx();
  if (!ctx) return FPT_ENOMEM;
  ctx->device = device;
  ctx->stream = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e = cudaSetDevice(device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&ctx->n_sm, cudaDevAttrMultiProcessorCount, device);
  if (e == cudaSuccess) e = cudaMalloc(&ctx->d_err, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(ctx->d_err, 0, sizeof(int));
  static_assert(kPatternKeys <= 128, "pattern counters");
  if (e == cudaSuccess) e = cudaMalloc(&ctx->d_count, 128 * sizeof(unsigned long long));
  if (e == cudaSuccess) e = cudaMalloc(&ctx->d_ctl, kCtlBytes);
  for (int k = 0; k < fpt_ctx::kSide && e == cudaSuccess; ++k)
    e = cudaEventCreateWithFlags(&ctx->join_ev[k], cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->fork_ev, cudaEventDisableTiming);
  for (int k = 0; k < fpt_ctx::kOrderStreams && e == cudaSuccess; ++k) {
    e = cudaStreamCreateWithFlags(&ctx->ostream[k], cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->ojoin_ev[k], cudaEventDisableTiming);
  }
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->ofork_ev, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaMalloc(&ctx->d_dropped, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemset(ctx->d_dropped, 0, sizeof(unsigned));
  // the fixed array of fpt_backward_noalloc: its address on this device, looked up again for every context
  if (e == cudaSuccess) e = noalloc_lookup(device);
  if (e != cudaSuccess) {
    fpt_destroy(ctx);
    return FPT_ECUDA;
  }
  *out = ctx;
  return FPT_OK;
}

void fpt_destroy(fpt_ctx* ctx) {
  if (!ctx) return;
  cudaSetDevice(ctx->device);
  for (auto& p : ctx->ev_pending) {
    cudaEventDestroy(p.second.first);
    cudaEventDestroy(p.second.second);
  }
  for (cudaEvent_t e : ctx->ev_pool) cudaEventDestroy(e);
  cudaFree(ctx->d_err);
  cudaFree(ctx->d_count);
  cudaFree(ctx->d_ctl);
  for (int k = 0; k < fpt_ctx::kSide; ++k) {
    if (ctx->side[k]) cudaStreamDestroy(ctx->side[k]);
    if (ctx->join_ev[k]) cudaEventDestroy(ctx->join_ev[k]);
  }
  if (ctx->fork_ev) cudaEventDestroy(ctx->fork_ev);
  for (int k = 0; k < fpt_ctx::kOrderStreams; ++k) {
    if (ctx->ostream[k]) cudaStreamDestroy(ctx->ostream[k]);
    if (ctx->ojoin_ev[k]) cudaEventDestroy(ctx->ojoin_ev[k]);
  }
  if (ctx->ofork_ev) cudaEventDestroy(ctx->ofork_ev);
  cudaFree(ctx->d_dropped);
  for (const Scratch* s : {&ctx->gacc, &ctx->rescue, &ctx->step, &ctx->tape}) cudaFree(s->p);
  for (void* p : ctx->kept) cudaFree(p);
  delete ctx;
}

fpt_status fpt_set_stream(fpt_ctx* ctx, void* cuda_stream) {
  if (!ctx) return FPT_EINVAL;
  // no synchronisation here (the call is legal inside a stream capture): the caller orders the old
  // stream's work, uploads included, before the new stream's
  ctx->stream = static_cast<cudaStream_t>(cuda_stream);
  return FPT_OK;
}

const char* fpt_last_error(const fpt_ctx* ctx) { return ctx ? ctx->msg : "null context"; }

fpt_status fpt_set_accumulation(fpt_ctx* ctx, int32_t flush_tiles, int32_t smem) {
  if (!ctx) return FPT_EINVAL;
  if (flush_tiles < 1 || (smem != 0 && smem != 1))
    return fail(ctx, FPT_EINVAL, "fpt_set_accumulation: flush_tiles must be >= 1 and smem 0 or 1");
  ctx->acc_flush_tiles = flush_tiles;
  ctx->acc_smem = smem;
  return FPT_OK;
}

fpt_status fpt_sync(fpt_ctx* ctx) {
  if (!ctx) return FPT_EINVAL;
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  int err = 0;
  CUDA_OR_FAIL(ctx, cudaMemcpy(&err, ctx->d_err, sizeof(int), cudaMemcpyDeviceToHost));
  if (err) {
    CUDA_OR_FAIL(ctx, cudaMemset(ctx->d_err, 0, sizeof(int)));
    return fail(ctx, FPT_EDEVICE, "device error code %d", err);
  }
  return FPT_OK;
}

// ---------------------------------------------------------------------------
// scene
// ---------------------------------------------------------------------------
static void split(double x, float& hi, float& lo) {
  hi = (float)x;
  lo = (float)(x - (double)hi);
}

fpt_status fpt_scene_upload(fpt_ctx* ctx, const uint8_t* types, const double* verts, int32_t n_obj,
                            fpt_scene** out) {
  if (!ctx || !types || !verts || !out) return fail(ctx, FPT_EINVAL, "null argument");
  *out = nullptr;
  if (n_obj < 1 || n_obj > 65535) return fail(ctx, FPT_EINVAL, "n_obj %d outside [1, 65535]", n_obj);
  double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int k = 0; k < n_obj; ++k) {
    if (types[k] != FPT_QUAD && types[k] != FPT_EDGE) return fail(ctx, FPT_EINVAL, "object %d: bad type", k);
    const int nv = types[k] == FPT_QUAD ? 3 : 2;
    for (int v = 0; v < nv; ++v)
      for (int c = 0; c < 3; ++c) {
        double x = verts[9 * k + 3 * v + c];
        if (!std::isfinite(x)) return fail(ctx, FPT_EINVAL, "object %d: non-finite vertex", k);
        lo[c] = x < lo[c] ? x : lo[c];
        hi[c] = x > hi[c] ? x : hi[c];
      }
  }
  fpt_scene* s = new (std::nothrow) fpt_scene();
  if (!s) return FPT_ENOMEM;
  s->ctx = ctx;
  s->n_obj = n_obj;
  s->types.assign(types, types + n_obj);
  for (int c = 0; c < 3; ++c) s->centre[c] = 0.5 * (lo[c] + hi[c]);
  std::vector<float>& rec32 = s->h_rec32;
  std::vector<float>& aux = s->h_aux;
  std::vector<float>& reclo = s->h_reclo;
  std::vector<double>& rec64 = s->h_rec64;
  rec32.assign((size_t)n_obj * kRec32, 0.f);
  aux.assign((size_t)n_obj * kAux, 0.f);
  reclo.assign((size_t)n_obj * kRecLo, 0.f);
  rec64.assign((size_t)n_obj * kRec64, 0.0);
  for (int k = 0; k < n_obj; ++k) {
    const double* v = verts + 9 * k;
    double b[3], a1[3], a2[3];
    for (int c = 0; c < 3; ++c) {
      b[c] = v[c] - s->centre[c];
      a1[c] = v[3 + c] - v[c];
      a2[c] = types[k] == FPT_QUAD ? v[6 + c] - v[c] : 0.0;
    }
    double n1 = std::sqrt(a1[0] * a1[0] + a1[1] * a1[1] + a1[2] * a1[2]);
    double n2 = std::sqrt(a2[0] * a2[0] + a2[1] * a2[1] + a2[2] * a2[2]);
    double cx = a1[1] * a2[2] - a1[2] * a2[1], cy = a1[2] * a2[0] - a1[0] * a2[2], cz = a1[0] * a2[1] - a1[1] * a2[0];
    double area = std::sqrt(cx * cx + cy * cy + cz * cz);
    if (types[k] == FPT_QUAD && area < 1e-9) {
      delete s;
      return fail(ctx, FPT_EINVAL, "object %d: zero-area plane", k);
    }
    if (types[k] == FPT_EDGE && n1 < 1e-9) {
      delete s;
      return fail(ctx, FPT_EINVAL, "object %d: zero-length edge", k);
    }
    for (int c = 0; c < 3; ++c) {
      rec64[kRec64 * k + c] = b[c];
      rec64[kRec64 * k + 3 + c] = a1[c];
      rec64[kRec64 * k + 6 + c] = a2[c];
      split(b[c], rec32[kRec32 * k + c], rec32[kRec32 * k + 3 + c]);
      split(a1[c], rec32[kRec32 * k + 6 + c], reclo[kRecLo * k + c]);
      split(a2[c], rec32[kRec32 * k + 9 + c], reclo[kRecLo * k + 3 + c]);
    }
    // side heights for the boundary distance: distance between the sides t1 = 0, 1 is area/|a2|
    aux[kAux * k + 0] = types[k] == FPT_QUAD ? (float)(area / n2) : (float)n1;
    aux[kAux * k + 1] = types[k] == FPT_QUAD ? (float)(area / n1) : 0.f;
    aux[kAux * k + 2] = types[k] == FPT_EDGE ? 1.f : 0.f;
    aux[kAux * k + 3] = 0.f;
  }
  // occluder records of the planar objects: centred origin, unit normal, dual basis of (a1, a2)
  std::vector<float>& occ = s->h_occ;
  for (int k = 0; k < n_obj; ++k) {
    if (types[k] != FPT_QUAD) continue;
    const double* v = verts + 9 * k;
    double b[3], a1[3], a2[3];
    for (int c = 0; c < 3; ++c) {
      b[c] = v[c] - s->centre[c];
      a1[c] = v[3 + c] - v[c];
      a2[c] = v[6 + c] - v[c];
    }
    double nv[3] = {a1[1] * a2[2] - a1[2] * a2[1], a1[2] * a2[0] - a1[0] * a2[2], a1[0] * a2[1] - a1[1] * a2[0]};
    const double nn = std::sqrt(nv[0] * nv[0] + nv[1] * nv[1] + nv[2] * nv[2]);
    const double g11 = a1[0] * a1[0] + a1[1] * a1[1] + a1[2] * a1[2];
    const double g12 = a1[0] * a2[0] + a1[1] * a2[1] + a1[2] * a2[2];
    const double g22 = a2[0] * a2[0] + a2[1] * a2[1] + a2[2] * a2[2];
    const double det = g11 * g22 - g12 * g12;
    for (int c = 0; c < 3; ++c) occ.push_back((float)b[c]);
    for (int c = 0; c < 3; ++c) occ.push_back((float)(nv[c] / nn));
    for (int c = 0; c < 3; ++c) occ.push_back((float)((g22 * a1[c] - g12 * a2[c]) / det));
    for (int c = 0; c < 3; ++c) occ.push_back((float)((g11 * a2[c] - g12 * a1[c]) / det));
    int32_t id = k;
    float idf;
    std::memcpy(&idf, &id, sizeof(idf));
    occ.push_back(idf);
  }
  s->n_occ = (int)(occ.size() / kOcc);
  s->h_occ_slot.assign(n_obj, -1);
  for (int k = 0, q = 0; k < n_obj; ++k)
    if (types[k] == FPT_QUAD) s->h_occ_slot[k] = q++;
  cudaError_t e = cudaSetDevice(ctx->device);
  if (e == cudaSuccess) e = cudaMalloc(&s->d_types, (size_t)n_obj);
  if (e == cudaSuccess) e = cudaMalloc(&s->d_occ_slot, (size_t)n_obj * sizeof(int32_t));
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(s->d_types, s->types.data(), (size_t)n_obj, cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(s->d_occ_slot, s->h_occ_slot.data(), (size_t)n_obj * sizeof(int32_t), cudaMemcpyHostToDevice,
                        ctx->stream);
  if (e == cudaSuccess && s->n_occ) e = cudaMalloc(&s->d_occ, occ.size() * sizeof(float));
  if (e == cudaSuccess && s->n_occ)
    e = cudaMemcpyAsync(s->d_occ, occ.data(), occ.size() * sizeof(float), cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess) e = cudaMalloc(&s->d_rec32, rec32.size() * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&s->d_rec64, rec64.size() * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&s->d_aux, aux.size() * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&s->d_reclo, reclo.size() * sizeof(float));
  // copies on the context's stream, ordered before every later call on it, with no wait for the
  // device; their host sources live in the scene until it is freed
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(s->d_reclo, reclo.data(), reclo.size() * sizeof(float), cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(s->d_rec32, rec32.data(), rec32.size() * sizeof(float), cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(s->d_rec64, rec64.data(), rec64.size() * sizeof(double), cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(s->d_aux, aux.data(), aux.size() * sizeof(float), cudaMemcpyHostToDevice, ctx->stream);
  if (e != cudaSuccess) {
    fpt_scene_free(s);
    return fail(ctx, FPT_ECUDA, "scene upload: %s", cudaGetErrorString(e));
  }
  *out = s;
  return FPT_OK;
}

fpt_status fpt_scene_upload_device(fpt_ctx* ctx, const uint8_t* types, const float* verts, int32_t n_obj,
                                   const double* centre, fpt_scene** out) {
  if (!ctx || !types || !verts || !out) return fail(ctx, FPT_EINVAL, "null argument");
  *out = nullptr;
  if (n_obj < 1 || n_obj > 65535) return fail(ctx, FPT_EINVAL, "n_obj %d outside [1, 65535]", n_obj);
  for (int k = 0; k < n_obj; ++k)
    if (types[k] != FPT_QUAD && types[k] != FPT_EDGE) return fail(ctx, FPT_EINVAL, "object %d: bad type", k);
  if (centre)
    for (int c = 0; c < 3; ++c)
      if (!std::isfinite(centre[c])) return fail(ctx, FPT_EINVAL, "non-finite centre");
  fpt_scene* s = new (std::nothrow) fpt_scene();
  if (!s) return FPT_ENOMEM;
  s->ctx = ctx;
  s->n_obj = n_obj;
  s->types.assign(types, types + n_obj);
  for (int c = 0; c < 3; ++c) s->centre[c] = centre ? centre[c] : 0.0;
  s->h_occ_slot.assign(n_obj, -1);
  int n_occ = 0;
  for (int k = 0; k < n_obj; ++k)
    if (types[k] == FPT_QUAD) s->h_occ_slot[k] = n_occ++;
  s->n_occ = n_occ;
  cudaError_t e = cudaSetDevice(ctx->device);
  if (e == cudaSuccess) e = cudaMalloc(&s->d_types, (size_t)n_obj);
  if (e == cudaSuccess) e = cudaMalloc(&s->d_occ_slot, (size_t)n_obj * sizeof(int32_t));
  if (e == cudaSuccess && n_occ) e = cudaMalloc(&s->d_occ, (size_t)n_occ * kOcc * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&s->d_rec32, (size_t)n_obj * kRec32 * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&s->d_rec64, (size_t)n_obj * kRec64 * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&s->d_aux, (size_t)n_obj * kAux * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&s->d_reclo, (size_t)n_obj * kRecLo * sizeof(float));
  // the type tables' host sources stay in the scene until it is freed
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(s->d_types, s->types.data(), (size_t)n_obj, cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(s->d_occ_slot, s->h_occ_slot.data(), (size_t)n_obj * sizeof(int32_t), cudaMemcpyHostToDevice,
                        ctx->stream);
  if (e == cudaSuccess)
    e = launch_object_records(n_obj, s->d_types, s->d_occ_slot, verts, s->centre, s->d_rec32, s->d_reclo, s->d_rec64,
                              s->d_aux, s->d_occ, ctx->d_err, ctx->stream);
  if (e != cudaSuccess) {
    fpt_scene_free(s);
    return fail(ctx, FPT_ECUDA, "device scene upload: %s", cudaGetErrorString(e));
  }
  *out = s;
  return FPT_OK;
}

void fpt_scene_free(fpt_scene* s) {
  if (!s) return;
  cudaFree(s->d_rec32);
  cudaFree(s->d_rec64);
  cudaFree(s->d_aux);
  cudaFree(s->d_reclo);
  cudaFree(s->d_tx32);
  cudaFree(s->d_rx32);
  cudaFree(s->d_tx64);
  cudaFree(s->d_rx64);
  cudaFree(s->d_occ);
  cudaFree(s->d_types);
  cudaFree(s->d_occ_slot);
  delete s;
}

// Upload points (recentred, FP32 pairs and FP64) asynchronously on `stream`.  h32 / h64 hold the host
// sources until the next upload or the scene's release; the old device buffers are freed first
// (cudaFree waits for the device), so no copy from the old sources is pending when they are refilled.
static cudaError_t upload_points(const double* p, int n, const double* centre, float** d32, double** d64,
                                 std::vector<float>& h32, std::vector<double>& h64, cudaStream_t stream) {
  cudaFree(*d32);
  cudaFree(*d64);
  *d32 = nullptr;
  *d64 = nullptr;
  h32.assign((size_t)n * kEnd32, 0.f);
  h64.assign((size_t)n * 3, 0.0);
  for (int i = 0; i < n; ++i)
    for (int c = 0; c < 3; ++c) {
      double x = p[3 * i + c] - centre[c];
      h64[3 * i + c] = x;
      split(x, h32[kEnd32 * i + c], h32[kEnd32 * i + 3 + c]);
    }
  cudaError_t e = cudaMalloc(d32, h32.size() * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(d64, h64.size() * sizeof(double));
  if (e == cudaSuccess) e = cudaMemcpyAsync(*d32, h32.data(), h32.size() * sizeof(float), cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(*d64, h64.data(), h64.size() * sizeof(double), cudaMemcpyHostToDevice, stream);
  return e;
}

fpt_status fpt_set_endpoints(fpt_scene* s, const double* tx, int32_t n_tx, const double* rx, int32_t n_rx) {
  if (!s || !tx || !rx) return FPT_EINVAL;
  fpt_ctx* ctx = s->ctx;
  if (n_tx < 1 || n_rx < 1) return fail(ctx, FPT_EINVAL, "need at least one TX and one RX");
  for (int i = 0; i < 3 * n_tx; ++i)
    if (!std::isfinite(tx[i])) return fail(ctx, FPT_EINVAL, "non-finite TX");
  for (int i = 0; i < 3 * n_rx; ++i)
    if (!std::isfinite(rx[i])) return fail(ctx, FPT_EINVAL, "non-finite RX");
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  CUDA_OR_FAIL(ctx, upload_points(tx, n_tx, s->centre, &s->d_tx32, &s->d_tx64, s->h_tx32, s->h_tx64, ctx->stream));
  CUDA_OR_FAIL(ctx, upload_points(rx, n_rx, s->centre, &s->d_rx32, &s->d_rx64, s->h_rx32, s->h_rx64, ctx->stream));
  s->n_tx = s->tx_cap = n_tx;
  s->n_rx = s->rx_cap = n_rx;
  return FPT_OK;
}

// Device buffers for n endpoints: kept when they already hold n, reallocated otherwise (cudaFree waits
// for the device, so a pending copy from an earlier host upload into the old buffer has finished).
static cudaError_t endpoint_buffers(int n, int* cap, float** d32, double** d64) {
  if (n <= *cap && *d32 && *d64) return cudaSuccess;
  cudaFree(*d32);
  cudaFree(*d64);
  *d32 = nullptr;
  *d64 = nullptr;
  *cap = 0;
  cudaError_t e = cudaMalloc(d32, (size_t)n * kEnd32 * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(d64, (size_t)n * 3 * sizeof(double));
  if (e == cudaSuccess) *cap = n;
  return e;
}

fpt_status fpt_set_endpoints_device(fpt_scene* s, const float* tx, int32_t n_tx, const float* rx, int32_t n_rx) {
  if (!s || !tx || !rx) return s ? fail(s->ctx, FPT_EINVAL, "null argument") : FPT_EINVAL;
  fpt_ctx* ctx = s->ctx;
  if (n_tx < 1 || n_rx < 1) return fail(ctx, FPT_EINVAL, "need at least one TX and one RX");
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  CUDA_OR_FAIL(ctx, endpoint_buffers(n_tx, &s->tx_cap, &s->d_tx32, &s->d_tx64));
  CUDA_OR_FAIL(ctx, endpoint_buffers(n_rx, &s->rx_cap, &s->d_rx32, &s->d_rx64));
  CUDA_OR_FAIL(ctx, launch_endpoint_records(tx, n_tx, s->centre, s->d_tx32, s->d_tx64, ctx->d_err, ctx->stream));
  CUDA_OR_FAIL(ctx, launch_endpoint_records(rx, n_rx, s->centre, s->d_rx32, s->d_rx64, ctx->d_err, ctx->stream));
  s->n_tx = n_tx;
  s->n_rx = n_rx;
  return FPT_OK;
}

fpt_status fpt_scene_update_vertices(fpt_scene* s, const float* verts) {
  if (!s || !verts) return s ? fail(s->ctx, FPT_EINVAL, "null argument") : FPT_EINVAL;
  fpt_ctx* ctx = s->ctx;
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  CUDA_OR_FAIL(ctx, launch_object_records(s->n_obj, s->d_types, s->d_occ_slot, verts, s->centre, s->d_rec32,
                                          s->d_reclo, s->d_rec64, s->d_aux, s->d_occ, ctx->d_err, ctx->stream));
  return FPT_OK;
}

// ---------------------------------------------------------------------------
// batches
// ---------------------------------------------------------------------------
static fpt_status make_alphabet(fpt_ctx* ctx, const fpt_scene* s, const int32_t* alphabet, int32_t n_alpha,
                                fpt_batch* b) {
  std::vector<int32_t>& a = b->h_alphabet;
  a.clear();
  if (alphabet) {
    if (n_alpha < 1) return fail(ctx, FPT_EINVAL, "empty alphabet");
    a.assign(alphabet, alphabet + n_alpha);
    for (int32_t o : a)
      if (o < 0 || o >= s->n_obj) return fail(ctx, FPT_EINVAL, "alphabet id %d out of range", o);
  } else {
    for (int k = 0; k < s->n_obj; ++k) a.push_back(k);
  }
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  CUDA_OR_FAIL(ctx, cudaMalloc(&b->d_alphabet, a.size() * sizeof(int32_t)));
  CUDA_OR_FAIL(ctx, cudaMemcpyAsync(b->d_alphabet, a.data(), a.size() * sizeof(int32_t), cudaMemcpyHostToDevice,
                                    ctx->stream));
  b->dev.alphabet = b->d_alphabet;
  b->dev.n_alpha = (int)a.size();
  // positions of the reflectors, then of the edges: the exhaustive enumeration by pattern
  std::vector<int32_t>& pos = b->h_type_pos;
  pos.clear();
  for (int pass = 0; pass < 2; ++pass)
    for (size_t k = 0; k < a.size(); ++k)
      if ((s->types[a[k]] == FPT_QUAD) == (pass == 0)) pos.push_back((int32_t)k);
  b->dev.n_alpha_quad = 0;
  for (int32_t o : a) b->dev.n_alpha_quad += s->types[o] == FPT_QUAD;
  CUDA_OR_FAIL(ctx, cudaMalloc(&b->d_type_pos, pos.size() * sizeof(int32_t)));
  CUDA_OR_FAIL(ctx, cudaMemcpyAsync(b->d_type_pos, pos.data(), pos.size() * sizeof(int32_t), cudaMemcpyHostToDevice,
                                    ctx->stream));
  b->dev.type_pos = b->d_type_pos;
  b->types = s->types;
  return FPT_OK;
}

// Reciprocals of the exhaustive decoders' divisors (FastDiv).
static void set_reciprocals(BatchDev& d) {
  d.fd_rx = make_fastdiv((uint64_t)d.n_rx);
  d.fd_alpha = make_fastdiv((uint64_t)d.n_alpha);
  d.fd_quad = make_fastdiv((uint64_t)d.n_alpha_quad);
  d.fd_edge = make_fastdiv((uint64_t)(d.n_alpha - d.n_alpha_quad));
  for (int n = 0; n <= kMaxOrder; ++n) d.fd_kpow[n] = make_fastdiv(d.kpow[n]);
  const uint64_t range = d.hi >= d.lo ? (uint64_t)(d.hi - d.lo + 1) : 1u;
  d.fd_alpha1 = make_fastdiv(d.n_alpha > 1 ? (uint64_t)(d.n_alpha - 1) : 1u);
  d.fd_range = make_fastdiv(range);
  d.fd_pp = make_fastdiv(d.per_pair);
  auto t32 = [](uint64_t m) { return m >= 1 && m <= 65535 ? (uint32_t)((1ull << 32) % m) : 0u; };
  d.t32_alpha = t32((uint64_t)d.n_alpha);
  d.t32_alpha1 = t32(d.n_alpha > 1 ? (uint64_t)(d.n_alpha - 1) : 1u);
  d.t32_range = t32(range);
}

static fpt_status check_orders(fpt_ctx* ctx, int lo, int hi) {
  if (lo < 1 || hi > kMaxOrder || lo > hi) return fail(ctx, FPT_EINVAL, "orders [%d, %d] outside [1, %d]", lo, hi, kMaxOrder);
  return FPT_OK;
}

fpt_status fpt_batch_exhaustive(fpt_ctx* ctx, const fpt_scene* s, const int32_t* alphabet, int32_t n_alpha,
                                int32_t lo, int32_t hi, fpt_batch** out) {
  if (!ctx || !s || !out) return fail(ctx, FPT_EINVAL, "null argument");
  *out = nullptr;
  if (s->n_tx < 1 || s->n_rx < 1) return fail(ctx, FPT_EINVAL, "scene has no endpoints");
  fpt_status st = check_orders(ctx, lo, hi);
  if (st != FPT_OK) return st;
  fpt_batch* b = new (std::nothrow) fpt_batch();
  if (!b) return FPT_ENOMEM;
  b->ctx = ctx;
  st = make_alphabet(ctx, s, alphabet, n_alpha, b);
  if (st != FPT_OK) {
    fpt_batch_free(b);
    return st;
  }
  BatchDev& d = b->dev;
  d.mode = BATCH_EXHAUSTIVE;
  d.lo = lo;
  d.hi = hi;
  d.n_max = hi;
  d.n_tx = s->n_tx;
  d.n_rx = s->n_rx;
  // K^n and per-pair offsets; refuse sizes that overflow 64-bit indexing
  const double K = d.n_alpha;
  double total = 0;
  for (int n = lo; n <= hi; ++n) total += std::pow(K, n);
  if (total * (double)s->n_tx * (double)s->n_rx > 9.0e18) {
    fpt_batch_free(b);
    return fail(ctx, FPT_EINVAL, "batch too large for 64-bit path indices");
  }
  d.kpow[0] = 1;
  for (int n = 1; n <= kMaxOrder; ++n) d.kpow[n] = n <= hi ? d.kpow[n - 1] * (uint64_t)d.n_alpha : 0;
  // offset[n] = sum_{m = lo}^{n-1} K^m: first index of order n inside a pair
  uint64_t acc = 0;
  for (int n = 0; n <= kMaxOrder + 1; ++n) {
    d.offset[n] = acc;
    if (n >= lo && n <= hi && n <= kMaxOrder) acc += d.kpow[n];
  }
  d.per_pair = acc;
  d.n_paths = acc * (uint64_t)s->n_tx * (uint64_t)s->n_rx;
  set_reciprocals(d);
  *out = b;
  return FPT_OK;
}

fpt_status fpt_batch_seeded(fpt_ctx* ctx, const fpt_scene* s, const int32_t* alphabet, int32_t n_alpha, uint64_t seed,
                            uint64_t per_pair, int32_t lo, int32_t hi, fpt_batch** out) {
  if (!ctx || !s || !out) return fail(ctx, FPT_EINVAL, "null argument");
  *out = nullptr;
  if (s->n_tx < 1 || s->n_rx < 1) return fail(ctx, FPT_EINVAL, "scene has no endpoints");
  fpt_status st = check_orders(ctx, lo, hi);
  if (st != FPT_OK) return st;
  if (per_pair < 1) return fail(ctx, FPT_EINVAL, "per_pair must be >= 1");
  fpt_batch* b = new (std::nothrow) fpt_batch();
  if (!b) return FPT_ENOMEM;
  b->ctx = ctx;
  st = make_alphabet(ctx, s, alphabet, n_alpha, b);
  if (st == FPT_OK && b->dev.n_alpha < 2 && hi > 1) st = fail(ctx, FPT_EINVAL, "seeded batches need >= 2 objects");
  if (st != FPT_OK) {
    fpt_batch_free(b);
    return st;
  }
  BatchDev& d = b->dev;
  d.mode = BATCH_SEEDED;
  d.lo = lo;
  d.hi = hi;
  d.n_max = hi;
  d.n_tx = s->n_tx;
  d.n_rx = s->n_rx;
  d.seed = seed;
  d.per_pair = per_pair;
  d.n_paths = per_pair * (uint64_t)s->n_tx * (uint64_t)s->n_rx;
  set_reciprocals(b->dev);
  *out = b;
  return FPT_OK;
}

fpt_status fpt_batch_explicit(fpt_ctx* ctx, const fpt_scene* s, const int32_t* ids_dev, const uint8_t* order_dev,
                              const int32_t* tx_idx_dev, const int32_t* rx_idx_dev, uint64_t n, int32_t n_max,
                              fpt_batch** out) {
  // an empty batch (n = 0) is legal and its device arrays may be NULL
  if (!ctx || !s || !out || (n > 0 && (!ids_dev || !order_dev || !tx_idx_dev || !rx_idx_dev)))
    return fail(ctx, FPT_EINVAL, "null argument");
  *out = nullptr;
  if (n_max < 1 || n_max > kMaxOrder) return fail(ctx, FPT_EINVAL, "n_max %d outside [1, %d]", n_max, kMaxOrder);
  if (s->n_tx < 1 || s->n_rx < 1) return fail(ctx, FPT_EINVAL, "scene has no endpoints");
  fpt_batch* b = new (std::nothrow) fpt_batch();
  if (!b) return FPT_ENOMEM;
  b->ctx = ctx;
  BatchDev& d = b->dev;
  d.mode = BATCH_EXPLICIT;
  d.n_alpha = s->n_obj;  // ids are object ids, checked against the object count
  d.lo = 1;
  d.hi = n_max;
  d.n_max = n_max;
  d.n_tx = s->n_tx;
  d.n_rx = s->n_rx;
  d.n_paths = n;
  d.per_pair = 1;
  d.ids = ids_dev;
  d.order = order_dev;
  d.tx_idx = tx_idx_dev;
  d.rx_idx = rx_idx_dev;
  b->types = s->types;
  set_reciprocals(b->dev);
  *out = b;
  return FPT_OK;
}

fpt_status fpt_batch_size(const fpt_batch* b, uint64_t* n_paths, int32_t* n_max) {
  if (!b) return FPT_EINVAL;
  if (n_paths) *n_paths = b->dev.n_paths;
  if (n_max) *n_max = b->dev.n_max;
  return FPT_OK;
}

void fpt_batch_free(fpt_batch* b) {
  if (!b) return;
  cudaFree(b->d_alphabet);
  cudaFree(b->d_type_pos);
  cudaFree(b->d_lists);
  delete b;
}

fpt_status fpt_enumerate(fpt_ctx* ctx, const fpt_batch* b, int32_t* ids, uint8_t* order, int32_t* tx_idx,
                         int32_t* rx_idx) {
  if (!ctx || !b) return fail(ctx, FPT_EINVAL, "null argument");
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  CUDA_OR_FAIL(ctx, launch_enumerate(b->dev, ids, order, tx_idx, rx_idx, ctx->stream, ctx->n_sm));
  return FPT_OK;
}

// Bucket a seeded/explicit batch by (order, pattern) (once per batch; synchronous).
static fpt_status ensure_buckets(fpt_ctx* ctx, fpt_batch* b, const SceneDev& S) {
  if (b->dev.mode == BATCH_EXHAUSTIVE || b->bucketed) return FPT_OK;
  unsigned long long h[kPatternKeys] = {0};
  CUDA_OR_FAIL(ctx, cudaMemsetAsync(ctx->d_count, 0, sizeof(h), ctx->stream));
  CUDA_OR_FAIL(ctx, launch_pattern_histogram(S, b->dev, ctx->d_count, ctx->stream, ctx->n_sm));
  CUDA_OR_FAIL(ctx, cudaMemcpyAsync(h, ctx->d_count, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
  CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  // layout: orders in sequence; inside an order, the buckets large enough for a pattern launch, then the
  // small ones together (the unified kernel takes them in one launch)
  const uint64_t min_bucket = min_pattern_bucket(ctx);
  uint64_t acc = 0;
  unsigned long long cur[kPatternKeys];
  for (int n = 1; n <= kMaxOrder; ++n) {
    for (int pass = 0; pass < 2; ++pass) {
      if (pass == 1) b->small_start[n] = acc;
      for (unsigned q = 0; q < (unsigned)n_patterns(n); ++q) {
        const int k = pattern_key(n, q);
        if ((h[k] >= min_bucket) != (pass == 0)) continue;
        b->start[k] = acc;
        b->count[k] = h[k];
        cur[k] = acc;
        acc += h[k];
      }
      if (pass == 1) b->small_count[n] = acc - b->small_start[n];
    }
  }
  if (acc != b->dev.n_paths) return fail(ctx, FPT_EDEVICE, "pattern histogram mismatch");
  CUDA_OR_FAIL(ctx, cudaMalloc(&b->d_lists, (acc ? acc : 1) * sizeof(PathRec)));
  CUDA_OR_FAIL(ctx, cudaMemcpyAsync(ctx->d_count, cur, sizeof(cur), cudaMemcpyHostToDevice, ctx->stream));
  CUDA_OR_FAIL(ctx, launch_pattern_scatter(S, b->dev, ctx->d_count, b->d_lists, ctx->stream, ctx->n_sm));
  CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  b->bucketed = true;
  return FPT_OK;
}

// Paths of order n in a batch: count and list (nullptr for exhaustive batches).
static uint64_t order_slice(const fpt_batch* b, int n, const PathRec** list) {
  if (b->dev.mode == BATCH_EXHAUSTIVE) {
    *list = nullptr;
    if (n < b->dev.lo || n > b->dev.hi) return 0;
    return b->dev.kpow[n] * (uint64_t)b->dev.n_tx * (uint64_t)b->dev.n_rx;
  }
  // the buckets of order n are contiguous; the order's range starts at its first bucket in the layout
  uint64_t first = b->small_start[n], c = 0;
  for (unsigned q = 0; q < (unsigned)n_patterns(n); ++q) {
    const int k = pattern_key(n, q);
    c += b->count[k];
    if (b->count[k] && b->start[k] < first) first = b->start[k];
  }
  *list = b->d_lists + first;
  return c;
}

// Whether the context's stream is being captured.
static bool capturing(const fpt_ctx* ctx) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(ctx->stream, &st) == cudaSuccess) return st != cudaStreamCaptureStatusNone;
  cudaGetLastError();
  return false;
}

// At least `bytes` of scratch for a call that may be part of a capture.  Scratch that a captured graph uses stays until the
// context is destroyed; other outgrown scratch is freed.  With must = false a shortage leaves the scratch as it was, and
// nothing is allocated inside a capture (most capture modes refuse that, and end).
static cudaError_t reserve(fpt_ctx* ctx, Scratch& s, size_t bytes, bool in_capture, bool must) {
  if (bytes > s.cap) {
    if (in_capture && !must) return cudaErrorMemoryAllocation;
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e == cudaErrorMemoryAllocation && must && !s.captured) {  // no room beside the old block
      cudaGetLastError();
      cudaFree(s.p);
      s = Scratch{};
      e = cudaMalloc(&p, bytes);
    }
    if (e != cudaSuccess) {
      if (!must) cudaGetLastError();
      return e;
    }
    if (s.captured) {
      try {
        ctx->kept.push_back(s.p);
      } catch (...) {  // (no exception leaves a C entry)
        cudaFree(p);
        return cudaErrorMemoryAllocation;
      }
    } else {
      cudaFree(s.p);
    }
    s = Scratch{p, bytes, false};
  }
  s.captured = s.captured || in_capture;
  return cudaSuccess;
}

// The backward accumulators (ensure_gacc).
static double* gacc(const fpt_ctx* ctx) { return static_cast<double*>(ctx->gacc.p); }

// Path scratch for `entries` paths (three uint32 lists of them) and `steps` floats of first Newton steps.
static cudaError_t reserve_paths(fpt_ctx* ctx, uint64_t entries, size_t steps, bool in_capture, bool must) {
  const cudaError_t e = reserve(ctx, ctx->rescue, 3 * entries * sizeof(uint32_t), in_capture, must);
  return e != cudaSuccess ? e : reserve(ctx, ctx->step, steps * sizeof(float), in_capture, must);
}

// One order's share of a call: its paths, the stream its kernels go to and its scratch.
struct OrderRun {
  int n;
  uint64_t cnt;
  const PathRec* list;
  cudaStream_t stream;
  uint32_t* lists;  // three lists of cnt entries
  float* step;      // 2 n cnt floats (nullptr when the call asked for none)
  OrderCtl* ctl;
};

// Largest batch whose orders run side by side.  The kernels of one order form a chain (BFGS, two polish passes,
// FP64 polish, select, adjoint, FP64 adjoint) whose later links, and every link of a small batch, leave
// most of the GPU idle; the orders touch different paths, so their chains can overlap.  Measured, one order
// after the other against side by side: 200,000 tiny-scene paths of orders 1-4 353 -> 174 us, 541,000 canyon
// paths of orders 1-3 651 -> 456 us, city batches of orders 1-5 with 8 M paths 5.70 -> 5.21 ms, 24 M 15.6 -> 14.8 ms,
// 48 M 29.0 -> 27.9 ms.  The gain shrinks as single kernels fill the GPU, while overlapped orders need
// their scratch side by side (12 + 8 n bytes per path of order n instead of the largest order's alone), which the
// context keeps: hence the second line, on those bytes (100 M city paths of orders 1-5: 3.6 GB, in turn 1.0).
constexpr uint64_t kOverlapMaxPaths = 1ull << 27;
constexpr size_t kOverlapMaxScratch = size_t(4) << 30;

// The orders of a call.  With overlap, the longest sequences come first (the longest chain) on the context's
// stream and the others on the order streams, each with its own scratch; else all on the context's stream
// in ascending order, sharing one scratch.  run(orders, body) forks, calls body for each order and joins.
struct OrderPlan {
  OrderRun runs[kMaxOrder];
  int count = 0;
  bool overlap = false;
  void run_in_turn(cudaStream_t stream) {
    overlap = false;
    for (int i = 0; i < count; ++i) runs[i].stream = stream;
  }
};

static fpt_status plan_orders(fpt_ctx* ctx, const fpt_batch* b, bool scratch, bool steps, OrderPlan& plan) {
  uint64_t sum = 0, most = 0;
  size_t step_sum = 0, step_most = 0;
  for (int n = 1; n <= kMaxOrder; ++n) {
    const PathRec* list;
    const uint64_t cnt = order_slice(b, n, &list);
    if (!cnt) continue;
    if (scratch && cnt > 0xFFFFFFFFull)  // the lists hold 32-bit path numbers
      return fail(ctx, FPT_EUNSUPPORTED, "more than 2^32 paths of one order");
    OrderRun& r = plan.runs[plan.count++];
    r = OrderRun{n, cnt, list, ctx->stream, nullptr, nullptr, reinterpret_cast<OrderCtl*>(ctx->d_ctl) + n};
    sum += cnt;
    most = cnt > most ? cnt : most;
    const size_t st = steps ? (size_t)2 * n * cnt : 0;
    step_sum += st;
    step_most = st > step_most ? st : step_most;
  }
  // kernel timing brackets the launches of one class on the context's stream: one order after the other
  plan.overlap = plan.count > 1 && sum <= kOverlapMaxPaths && !ctx->prof &&
                 (!scratch || 3 * sum * sizeof(uint32_t) + step_sum * sizeof(float) <= kOverlapMaxScratch);
  if (scratch && plan.count) {
    const bool in_capture = capturing(ctx);
    // no room side by side, or no scratch for it before a capture: one order after the other, as for large batches
    if (plan.overlap) plan.overlap = reserve_paths(ctx, sum, step_sum, in_capture, false) == cudaSuccess;
    if (!plan.overlap) CUDA_OR_FAIL(ctx, reserve_paths(ctx, most, step_most, in_capture, true));
  }
  if (plan.overlap)
    for (int i = 0, j = plan.count - 1; i < j; ++i, --j) std::swap(plan.runs[i], plan.runs[j]);
  uint64_t at = 0;
  size_t step_at = 0;
  for (int i = 0; i < plan.count; ++i) {
    OrderRun& r = plan.runs[i];
    if (scratch) {
      r.lists = static_cast<uint32_t*>(ctx->rescue.p) + 3 * at;
      r.step = steps ? static_cast<float*>(ctx->step.p) + step_at : nullptr;
    }
    if (plan.overlap) {
      if (i > 0) r.stream = ctx->ostream[(i - 1) % fpt_ctx::kOrderStreams];
      at += r.cnt;
      step_at += steps ? (size_t)2 * r.n * r.cnt : 0;
    }
  }
  return FPT_OK;
}

// (body as it is: a std::function of it would allocate, and could throw across the C entries)
extern "C++" {
template <class Body>
static fpt_status run_orders(fpt_ctx* ctx, const OrderPlan& plan, const Body& body) {
  const int used = !plan.overlap ? 0 : (plan.count - 1 < fpt_ctx::kOrderStreams ? plan.count - 1 : fpt_ctx::kOrderStreams);
  if (used) {
    CUDA_OR_FAIL(ctx, cudaEventRecord(ctx->ofork_ev, ctx->stream));
    for (int k = 0; k < used; ++k) CUDA_OR_FAIL(ctx, cudaStreamWaitEvent(ctx->ostream[k], ctx->ofork_ev, 0));
  }
  fpt_status st = FPT_OK;
  for (int i = 0; i < plan.count && st == FPT_OK; ++i) st = body(plan.runs[i]);
  // joined also after an error: later calls reuse the scratch, and a stream capture must end joined
  cudaError_t joined = cudaSuccess;
  for (int k = 0; k < used; ++k) {
    cudaError_t e = cudaEventRecord(ctx->ojoin_ev[k], ctx->ostream[k]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(ctx->stream, ctx->ojoin_ev[k], 0);
    if (joined == cudaSuccess) joined = e;
  }
  if (st == FPT_OK) CUDA_OR_FAIL(ctx, joined);
  return st;
}
}  // extern "C++"

// Paths of order n and interaction-type pattern q: count and list (nullptr for exhaustive batches).
static uint64_t pattern_slice(const fpt_batch* b, int n, unsigned q, const PathRec** list) {
  if (b->dev.mode == BATCH_EXHAUSTIVE) {
    *list = nullptr;
    if (n < b->dev.lo || n > b->dev.hi) return 0;
    uint64_t c = (uint64_t)b->dev.n_tx * (uint64_t)b->dev.n_rx;
    for (int i = 0; i < n; ++i)
      c *= (uint64_t)(((q >> i) & 1u) ? b->dev.n_alpha_quad : b->dev.n_alpha - b->dev.n_alpha_quad);
    return c;
  }
  *list = b->d_lists + b->start[pattern_key(n, q)];
  return b->count[pattern_key(n, q)];
}

static fpt_status check_scene_batch(fpt_ctx* ctx, const fpt_scene* s, const fpt_batch* b) {
  if (!ctx || !s || !b) return fail(ctx, FPT_EINVAL, "null argument");
  if (b->dev.n_tx != s->n_tx || b->dev.n_rx != s->n_rx)
    return fail(ctx, FPT_EINVAL, "batch was built for other endpoints");
  if (b->dev.mode == BATCH_EXPLICIT && b->dev.n_alpha != s->n_obj) return fail(ctx, FPT_EINVAL, "batch/scene mismatch");
  if (b->types != s->types) return fail(ctx, FPT_EINVAL, "batch was built for a scene with other object types");
  return FPT_OK;
}

// The implicit backward of one order's paths (fpt_backward, and fpt_solve_grad after its solve).
static fpt_status backward_order(fpt_ctx* ctx, const SceneDev& S, const fpt_batch* b, const OrderRun& r,
                                 const BackwardCfg& cfg, const float* T, const uint8_t* status, const float* dX,
                                 const float* dL) {
  ProfScope ps(ctx, FPT_K_BACKWARD);
  BackwardCfg cfg_n = cfg;
  cfg_n.sel = r.lists + 2 * r.cnt;  // the third list of the scratch (the polish's, free here)
  cfg_n.sel_count = &r.ctl->selected;
  CUDA_OR_FAIL(ctx, launch_backward(r.n, S, b->dev, cfg_n, r.cnt, r.list, T, status, dX, dL, gacc(ctx), r.stream,
                                    ctx->n_sm, r.lists, &r.ctl->backward64));
  return FPT_OK;
}

// Streams for the pattern launches of one order.  With one order at a time the order streams are idle and serve; orders
// side by side get streams of their own, created here once (a context whose batches never need them does not pay for
// them), or, where that is not possible (a stream capture, an error), the order streams too: that only
// adds dependencies.
static const cudaStream_t* side_streams(fpt_ctx* ctx, bool overlap) {
  static_assert(fpt_ctx::kSide <= fpt_ctx::kOrderStreams, "order streams in place of side streams");
  if (!overlap) return ctx->ostream;
  if (!ctx->side[fpt_ctx::kSide - 1]) {
    if (capturing(ctx)) return ctx->ostream;
    for (cudaStream_t& s : ctx->side)
      if (!s && cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) {
        s = nullptr;
        cudaGetLastError();
        return ctx->ostream;
      }
  }
  return ctx->side;
}

// BFGS of one order's paths.
static fpt_status bfgs_order(fpt_ctx* ctx, const SceneDev& S, const fpt_batch* b, const OrderRun& r, bool overlap,
                             const SolveCfg& sc, int specialize, float* T, uint8_t* status, uint8_t* iters) {
  ProfScope ps(ctx, FPT_K_BFGS);
  const int n = r.n;
  // pattern kernels pay off for buckets that fill the GPU several times over.  Seeded and explicit
  // batches keep an order's small buckets together, and the unified kernel takes them in one launch;
  // an exhaustive order with a small pattern runs the unified kernel throughout.
  const bool listed = b->dev.mode != BATCH_EXHAUSTIVE;
  const bool force = specialize == 2;
  bool by_pattern = specialize && sc.refill > 0 && n <= kMaxBfgsOrder;
  for (unsigned q = 0; by_pattern && !listed && !force && q < (1u << n); ++q) {
    const PathRec* qlist;
    const uint64_t qcnt = pattern_slice(b, n, q, &qlist);
    if (qcnt && qcnt < min_pattern_bucket(ctx)) by_pattern = false;
  }
  struct Launch {
    int pattern;
    uint64_t cnt;
    const PathRec* list;
    unsigned long long* work;
  };
  Launch todo[(1 << kMaxBfgsOrder) + 1];
  int count = 0;
  if (by_pattern) {
    for (unsigned q = 0; q < (1u << n); ++q) {
      const PathRec* qlist;
      const uint64_t qcnt = pattern_slice(b, n, q, &qlist);
      if (!qcnt || (listed && !force && qcnt < min_pattern_bucket(ctx))) continue;
      todo[count++] = {(int)q, qcnt, qlist, r.ctl->work + q};
    }
    if (listed && !force && b->small_count[n])
      todo[count++] = {-1, b->small_count[n], b->d_lists + b->small_start[n], r.ctl->work + 32};
  } else {
    todo[count++] = {-1, r.cnt, r.list, r.ctl->work + 32};
  }
  // the pattern launches of one order are independent: spread them over the side streams so that
  // each launch's tail overlaps the next one; each concurrent launch has its own work counter
  const int used = count < 2 ? 0 : (count < fpt_ctx::kSide ? count : fpt_ctx::kSide);
  const cudaStream_t* side = used ? side_streams(ctx, overlap) : nullptr;
  if (used) {
    CUDA_OR_FAIL(ctx, cudaEventRecord(ctx->fork_ev, r.stream));
    for (int k = 0; k < used; ++k) CUDA_OR_FAIL(ctx, cudaStreamWaitEvent(side[k], ctx->fork_ev, 0));
  }
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < count && e == cudaSuccess; ++i)
    e = launch_bfgs(n, todo[i].pattern, S, b->dev, sc, todo[i].cnt, todo[i].list, T, status, iters,
                    used ? side[i % used] : r.stream, ctx->n_sm, todo[i].work);
  // join every side stream that waited on the fork, also after an error (a stream capture must end joined)
  for (int k = 0; k < used; ++k) {
    const cudaError_t f = cudaEventRecord(ctx->join_ev[k], side[k]);
    const cudaError_t w = f == cudaSuccess ? cudaStreamWaitEvent(r.stream, ctx->join_ev[k], 0) : f;
    if (e == cudaSuccess) e = w;
  }
  CUDA_OR_FAIL(ctx, e);
  return FPT_OK;
}

// What fpt_solve_grad asks for after each order's solve.
struct BackwardAfter {
  BackwardCfg cfg;
  const float* dX;
  const float* dL;
};

// Solve of every order of the batch; with grad, the fused backward in the polish; with after, each order's
// adjoint kernels behind its solve on the same stream.
static fpt_status solve_impl(fpt_ctx* ctx, const fpt_scene* s, const fpt_batch* bc, const fpt_solve_params* prm,
                             float* T, float* X, float* L, uint8_t* status, uint8_t* iters, float* rho,
                             const GradCfg* grad, const BackwardAfter* after) {
  fpt_status st = check_scene_batch(ctx, s, bc);
  if (st != FPT_OK) return st;
  if (bc->dev.n_paths > 0 && (!T || !status)) return fail(ctx, FPT_EINVAL, "T_out and status_out are required");
  fpt_solve_params p;
  fpt_default_params(&p);
  if (prm) p = *prm;
  if (p.init_mode != 0 && p.init_mode != 1) return fail(ctx, FPT_EINVAL, "init_mode must be 0 or 1");
  if (p.init_mode == 1 && !ctx->init_mlp) return fail(ctx, FPT_EINVAL, "init_mode 1 needs fpt_set_init_mlp");
  if (p.max_iters < 0 || p.fp_iters < 1 || p.polish < 0 || p.polish > 2 || p.specialize < 0 || p.specialize > 2 ||
      !(p.kink_stop >= 0.f) || !(p.polish_radius >= 0.f))
    return fail(ctx, FPT_EINVAL, "bad solver parameters");
  fpt_batch* b = const_cast<fpt_batch*>(bc);
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  const SceneDev S = scene_dev(s);
  st = ensure_buckets(ctx, b, S);
  if (st != FPT_OK) return st;
  const float kink = p.kink_stop > 0.f ? p.kink_stop : 0.1f * p.deg_tol;
  SolveCfg sc{p.max_iters, p.fp_iters, p.fixed_iters, p.tol_step * p.tol_step, kink * kink,
              p.refill > 32 ? 32 : p.refill, p.init_mode == 1, kMaxChunk};
  // the polish needs its Newton step only to a modest relative accuracy: 100x looser pivot test than the adjoint
  PolishCfg pc{POLISH_SOLVE, p.polish, p.solved_tol, p.deg_tol, 1e-2f * p.cond_fp64, p.polish_fp64,
               p.polish_radius};
  OrderPlan plan;
  st = plan_orders(ctx, b, true, true, plan);
  if (st != FPT_OK) return st;
  if (b->dev.n_max > kMaxBfgsOrder) {
    // the kernels of orders 1-5 write the first five slots of a path; clear the rest
    CUDA_OR_FAIL(ctx, cudaMemsetAsync(T, 0, b->dev.n_paths * (uint64_t)b->dev.n_max * 2 * sizeof(float), ctx->stream));
    if (X) CUDA_OR_FAIL(ctx, cudaMemsetAsync(X, 0, b->dev.n_paths * (uint64_t)b->dev.n_max * 3 * sizeof(float), ctx->stream));
  }
  fpt_mlp* m = p.init_mode == 1 ? ctx->init_mlp : nullptr;
  CUDA_OR_FAIL(ctx, cudaMemsetAsync(ctx->d_ctl, 0, kCtlBytes, ctx->stream));
  return run_orders(ctx, plan, [&](const OrderRun& r) -> fpt_status {
    if (m) {
      // learned start: fused features -> network -> T on the tensor cores
      ProfScope ps(ctx, FPT_K_MLP);
      CUDA_OR_FAIL(ctx, launch_mlp_infer(S, b->dev, r.n, r.list, r.cnt, 1.f / m->scale, m->d_wt, m->d_w, T, 0, ctx->d_err,
                                         r.stream, ctx->n_sm));
    }
    fpt_status rs = bfgs_order(ctx, S, b, r, plan.overlap, sc, p.specialize, T, status, iters);
    if (rs != FPT_OK) return rs;
    {
      ProfScope ps(ctx, FPT_K_POLISH);
      GradCfg gc{};
      if (grad) {
        gc = *grad;
        gc.rescue_list = r.lists + r.cnt;
        gc.rescue_count = &r.ctl->adjoint64;
      }
      uint32_t* step_list = p.polish_all ? nullptr : r.lists + 2 * r.cnt;
      CUDA_OR_FAIL(ctx, launch_polish(r.n, S, b->dev, pc, r.cnt, r.list, T, X, L, status, rho, nullptr, nullptr,
                                      r.stream, ctx->n_sm, r.lists, &r.ctl->polish64, grad ? &gc : nullptr, step_list,
                                      &r.ctl->stepped, r.step));
    }
    if (!after) return FPT_OK;
    BackwardCfg cfg = after->cfg;
    cfg.chained = !ctx->prof;  // (kernel timing records events in between)
    return backward_order(ctx, S, b, r, cfg, T, status, after->dX, after->dL);
  });
}

fpt_status fpt_solve(fpt_ctx* ctx, const fpt_scene* s, const fpt_batch* bc, const fpt_solve_params* prm, float* T,
                     float* X, float* L, uint8_t* status, uint8_t* iters, float* rho) {
  return solve_impl(ctx, s, bc, prm, T, X, L, status, iters, rho, nullptr, nullptr);
}

// Context-owned FP64 gradient accumulators, sized for the scene and cleared.
static fpt_status ensure_gacc(fpt_ctx* ctx, const fpt_scene* s) {
  const size_t bytes = (size_t)(9 * s->n_obj + 3 * (s->n_tx + s->n_rx)) * sizeof(double);
  CUDA_OR_FAIL(ctx, reserve(ctx, ctx->gacc, bytes, capturing(ctx), true));
  CUDA_OR_FAIL(ctx, cudaMemsetAsync(ctx->gacc.p, 0, bytes, ctx->stream));
  return FPT_OK;
}

// The settings of a backward call on this context.
static BackwardCfg backward_cfg(fpt_ctx* ctx, uint8_t dl_mask) {
  fpt_solve_params p;
  fpt_default_params(&p);
  BackwardCfg cfg{p.cond_fp64, p.deg_tol, ctx->acc_smem, ctx->acc_flush_tiles, dl_mask};
  cfg.dropped = ctx->d_dropped;
  return cfg;
}

fpt_status fpt_solve_grad(fpt_ctx* ctx, const fpt_scene* s, const fpt_batch* bc, const fpt_solve_params* prm,
                          const float* dX, const float* dL, uint8_t dL_status_mask, float* T, float* X, float* L,
                          uint8_t* status, uint8_t* iters, float* rho, float* g_tx, float* g_rx,
                          float* g_vertices) {
  fpt_status st = check_scene_batch(ctx, s, bc);
  if (st != FPT_OK) return st;
  if (prm && prm->polish_fp64) return fail(ctx, FPT_EUNSUPPORTED, "fpt_solve_grad runs the double-float polish");
  if (prm && prm->polish < 1) return fail(ctx, FPT_EINVAL, "fpt_solve_grad needs polish >= 1");
  if (!status && bc->dev.n_paths > 0) return fail(ctx, FPT_EINVAL, "status_out is required");
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  st = ensure_gacc(ctx, s);
  if (st != FPT_OK) return st;
  CUDA_OR_FAIL(ctx, cudaMemsetAsync(ctx->d_dropped, 0, sizeof(unsigned), ctx->stream));
  if (!(prm && prm->fuse_adjoint)) {
    // the adjoint kernels after each order's solve, with the cotangents given here
    const BackwardAfter after{backward_cfg(ctx, dL ? (uint8_t)0 : dL_status_mask), dX, dL};
    st = solve_impl(ctx, s, bc, prm, T, X, L, status, iters, rho, nullptr, &after);
  } else {
    fpt_solve_params p;
    fpt_default_params(&p);
    GradCfg gc{};
    gc.dX = dX;
    gc.dL = dL;
    gc.dl_mask = dL ? (uint8_t)0 : dL_status_mask;
    gc.cond_adj = p.cond_fp64;
    gc.deg_tol = prm->deg_tol;
    gc.gacc = gacc(ctx);
    gc.flush_tiles = ctx->acc_flush_tiles;
    gc.acc_in_smem = ctx->acc_smem;
    gc.dropped = ctx->d_dropped;
    st = solve_impl(ctx, s, bc, prm, T, X, L, status, iters, rho, &gc, nullptr);
  }
  if (st != FPT_OK) return st;
  const SceneDev S = scene_dev(s);
  ProfScope ps(ctx, FPT_K_OTHER);
  CUDA_OR_FAIL(ctx, launch_backward_finalize(S, nullptr, gacc(ctx), g_tx, g_rx, g_vertices, ctx->stream));
  return FPT_OK;
}

fpt_status fpt_validity(fpt_ctx* ctx, const fpt_scene* s, const fpt_batch* bc, const float* T, uint8_t* mask,
                        float* bdist, float* rho) {
  fpt_status st = check_scene_batch(ctx, s, bc);
  if (st != FPT_OK) return st;
  if (!T && bc->dev.n_paths > 0) return fail(ctx, FPT_EINVAL, "T is required");
  fpt_batch* b = const_cast<fpt_batch*>(bc);
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  st = ensure_buckets(ctx, b, scene_dev(s));
  if (st != FPT_OK) return st;
  fpt_solve_params p;
  fpt_default_params(&p);
  const SceneDev S = scene_dev(s);
  PolishCfg pc{POLISH_VALIDITY, 0, p.solved_tol, p.deg_tol, 1e-2f * p.cond_fp64, 0};
  OrderPlan plan;
  st = plan_orders(ctx, b, true, false, plan);
  if (st != FPT_OK) return st;
  CUDA_OR_FAIL(ctx, cudaMemsetAsync(ctx->d_ctl, 0, kCtlBytes, ctx->stream));
  return run_orders(ctx, plan, [&](const OrderRun& r) -> fpt_status {
    ProfScope ps(ctx, FPT_K_POLISH);
    CUDA_OR_FAIL(ctx, launch_polish(r.n, S, b->dev, pc, r.cnt, r.list, const_cast<float*>(T), nullptr, nullptr, nullptr,
                                    rho, mask, bdist, r.stream, ctx->n_sm, r.lists, &r.ctl->polish64));
    return FPT_OK;
  });
}

fpt_status fpt_backward(fpt_ctx* ctx, const fpt_scene* s, const fpt_batch* bc, const float* T, const uint8_t* status,
                        const float* dX, const float* dL, uint8_t dL_status_mask, float* g_tx, float* g_rx,
                        float* g_vertices) {
  fpt_status st = check_scene_batch(ctx, s, bc);
  if (st != FPT_OK) return st;
  if (!T && bc->dev.n_paths > 0) return fail(ctx, FPT_EINVAL, "T is required");
  fpt_batch* b = const_cast<fpt_batch*>(bc);
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  st = ensure_buckets(ctx, b, scene_dev(s));
  if (st != FPT_OK) return st;
  st = ensure_gacc(ctx, s);
  if (st != FPT_OK) return st;
  const SceneDev S = scene_dev(s);
  if (!dL && dL_status_mask && !status && bc->dev.n_paths > 0)
    return fail(ctx, FPT_EINVAL, "dL_status_mask needs status");
  const BackwardCfg cfg = backward_cfg(ctx, dL ? (uint8_t)0 : dL_status_mask);
  OrderPlan plan;
  st = plan_orders(ctx, b, true, false, plan);
  if (st != FPT_OK) return st;
  CUDA_OR_FAIL(ctx, cudaMemsetAsync(ctx->d_dropped, 0, sizeof(unsigned), ctx->stream));
  CUDA_OR_FAIL(ctx, cudaMemsetAsync(ctx->d_ctl, 0, kCtlBytes, ctx->stream));
  st = run_orders(ctx, plan, [&](const OrderRun& r) { return backward_order(ctx, S, b, r, cfg, T, status, dX, dL); });
  if (st != FPT_OK) return st;
  {
    ProfScope ps(ctx, FPT_K_OTHER);
    CUDA_OR_FAIL(ctx, launch_backward_finalize(S, nullptr, gacc(ctx), g_tx, g_rx, g_vertices, ctx->stream));
  }
  return FPT_OK;
}

fpt_status fpt_backward_unrolled(fpt_ctx* ctx, const fpt_scene* s, const fpt_batch* bc, int32_t steps,
                                 int32_t fp_iters, const float* dX, const float* dL, float* T_out, uint8_t* status_out,
                                 float* g_tx, float* g_rx, float* g_vertices) {
  fpt_status st = check_scene_batch(ctx, s, bc);
  if (st != FPT_OK) return st;
  if (steps < 0 || steps > kUnrolledMaxSteps)
    return fail(ctx, FPT_EINVAL, "steps must be in [0, %d]", kUnrolledMaxSteps);
  if (fp_iters < 1 || fp_iters > kUnrolledMaxRounds) return fail(ctx, FPT_EINVAL, "fp_iters must be in [1, %d]",
                                                                 kUnrolledMaxRounds);
  fpt_batch* b = const_cast<fpt_batch*>(bc);
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  st = ensure_buckets(ctx, b, scene_dev(s));
  if (st != FPT_OK) return st;
  st = ensure_gacc(ctx, s);
  if (st != FPT_OK) return st;
  const SceneDev S = scene_dev(s);
  // tape for every resident thread of an order (at most 8 CTAs of kThreads per SM), within kUnrolledMaxTape bytes
  auto tape_floats = [&](const OrderRun& r) {
    uint64_t threads = ((r.cnt + kThreads - 1) / kThreads) * kThreads;
    const uint64_t resident = (uint64_t)ctx->n_sm * 8 * kThreads;
    if (threads > resident) threads = resident;
    const size_t need = unrolled_tape_floats(r.n, steps, threads), most = kUnrolledMaxTape / sizeof(float);
    return need > most ? most : need;
  };
  // Orders side by side where their tapes fit kUnrolledMaxTape together: the shorter orders run on the SMs that the
  // longest one's last, partly filled round of CTAs leaves idle.
  OrderPlan plan;
  st = plan_orders(ctx, b, false, false, plan);
  if (st != FPT_OK) return st;
  size_t sum = 0, most = 0;
  for (int i = 0; i < plan.count; ++i) {
    const size_t need = tape_floats(plan.runs[i]);
    sum += need;
    most = need > most ? need : most;
  }
  if (sum * sizeof(float) > kUnrolledMaxTape) plan.run_in_turn(ctx->stream);
  const bool in_capture = capturing(ctx);
  if (plan.overlap && reserve(ctx, ctx->tape, sum * sizeof(float), in_capture, false) != cudaSuccess)
    plan.run_in_turn(ctx->stream);  // no room side by side
  if (!plan.overlap) CUDA_OR_FAIL(ctx, reserve(ctx, ctx->tape, most * sizeof(float), in_capture, true));
  size_t at = 0;
  st = run_orders(ctx, plan, [&](const OrderRun& r) -> fpt_status {
    ProfScope ps(ctx, FPT_K_BACKWARD);
    const size_t need = tape_floats(r);
    CUDA_OR_FAIL(ctx, launch_unrolled(r.n, S, b->dev, steps, fp_iters, r.cnt, r.list, dX, dL, gacc(ctx),
                                      static_cast<float*>(ctx->tape.p) + at, need, T_out, status_out, r.stream, ctx->n_sm));
    if (plan.overlap) at += need;
    return FPT_OK;
  });
  if (st != FPT_OK) return st;
  {
    ProfScope ps(ctx, FPT_K_OTHER);
    CUDA_OR_FAIL(ctx, launch_backward_finalize(S, nullptr, gacc(ctx), g_tx, g_rx, g_vertices, ctx->stream));
  }
  return FPT_OK;
}

fpt_status fpt_occlusion(fpt_ctx* ctx, const fpt_scene* s, const fpt_batch* bc, const float* T, const uint8_t* status,
                         uint8_t status_mask, float tol, uint16_t* blocked_out) {
  fpt_status st = check_scene_batch(ctx, s, bc);
  if (st != FPT_OK) return st;
  if (bc->dev.n_paths > 0 && (!T || !blocked_out)) return fail(ctx, FPT_EINVAL, "T and blocked_out are required");
  if (status_mask && !status && bc->dev.n_paths > 0) return fail(ctx, FPT_EINVAL, "status_mask needs status");
  if (!(tol >= 0.f)) return fail(ctx, FPT_EINVAL, "tol must be >= 0");
  if ((size_t)s->n_occ * kOcc * sizeof(float) > kMaxSmemBytes)
    return fail(ctx, FPT_EUNSUPPORTED, "%d planar objects exceed the occluder table", s->n_occ);
  fpt_batch* b = const_cast<fpt_batch*>(bc);
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  st = ensure_buckets(ctx, b, scene_dev(s));
  if (st != FPT_OK) return st;
  const SceneDev S = scene_dev(s);
  const float t = tol > 0.f ? tol : 1e-4f;
  OrderPlan plan;
  st = plan_orders(ctx, b, true, false, plan);
  if (st != FPT_OK) return st;
  CUDA_OR_FAIL(ctx, cudaMemsetAsync(ctx->d_ctl, 0, kCtlBytes, ctx->stream));
  return run_orders(ctx, plan, [&](const OrderRun& r) -> fpt_status {
    ProfScope ps(ctx, FPT_K_OTHER);
    CUDA_OR_FAIL(ctx, launch_occlusion(S, b->dev, r.n, r.list, r.cnt, T, status, status_mask, s->d_occ, s->n_occ, t,
                                       blocked_out, r.lists, &r.ctl->selected, r.stream, ctx->n_sm));
    return FPT_OK;
  });
}

fpt_status fpt_backward_noalloc(fpt_ctx* ctx, const fpt_scene* s, const fpt_batch* b, const float* T,
                                const uint8_t* status, const float* dX, const float* dL, uint8_t dL_status_mask,
                                float* g_tx, float* g_rx, float* g_vertices) {
  fpt_status st = check_scene_batch(ctx, s, b);
  if (st != FPT_OK) return st;
  if (!T && b->dev.n_paths > 0) return fail(ctx, FPT_EINVAL, "T is required");
  if (!dL && dL_status_mask && !status && b->dev.n_paths > 0)
    return fail(ctx, FPT_EINVAL, "dL_status_mask needs status");
  const long long need = 9LL * s->n_obj + 3LL * (s->n_tx + s->n_rx);
  if (need > kNoAllocMaxAcc)
    return fail(ctx, FPT_EINVAL, "fpt_backward_noalloc: 9 n_obj + 3 (n_tx + n_rx) = %lld exceeds its limit %d", need,
                kNoAllocMaxAcc);
  if (b->dev.mode != BATCH_EXHAUSTIVE && !b->bucketed)
    return fail(ctx, FPT_EINVAL, "fpt_backward_noalloc: seeded/explicit batch not bucketed yet (solve it first)");
  const PathRec* lists[kMaxOrder + 1] = {nullptr};
  uint64_t counts[kMaxOrder + 1] = {0};
  for (int n = 1; n <= kMaxOrder; ++n) {
    counts[n] = order_slice(b, n, &lists[n]);
    if (counts[n] > (uint64_t)kNoAllocMaxSlice)
      return fail(ctx, FPT_EINVAL, "fpt_backward_noalloc: %llu paths of order %d exceed its limit %d",
                  (unsigned long long)counts[n], n, kNoAllocMaxSlice);
  }
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  const BackwardCfg cfg = backward_cfg(ctx, dL ? (uint8_t)0 : dL_status_mask);
  CUDA_OR_FAIL(ctx, cudaMemsetAsync(ctx->d_dropped, 0, sizeof(unsigned), ctx->stream));
  CUDA_OR_FAIL(ctx, launch_backward_noalloc(ctx->device, scene_dev(s), b->dev, cfg, lists, counts, T, status, dX, dL,
                                            g_tx, g_rx, g_vertices, ctx->stream, ctx->n_sm));
  return FPT_OK;
}

fpt_status fpt_backward_dropped(fpt_ctx* ctx, uint64_t* count) {
  if (!ctx || !count) return fail(ctx, FPT_EINVAL, "null argument");
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  unsigned h = 0;
  CUDA_OR_FAIL(ctx, cudaMemcpyAsync(&h, ctx->d_dropped, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
  CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  *count = h;
  return FPT_OK;
}

fpt_status fpt_count_status(fpt_ctx* ctx, const uint8_t* status, uint64_t n, uint8_t mask, uint64_t* count) {
  if (!ctx || !count || (!status && n > 0)) return fail(ctx, FPT_EINVAL, "null argument");
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  unsigned long long h = 0;
  CUDA_OR_FAIL(ctx, cudaMemsetAsync(ctx->d_count, 0, sizeof(unsigned long long), ctx->stream));
  CUDA_OR_FAIL(ctx, launch_count_status(status, n, mask, ctx->d_count, ctx->stream, ctx->n_sm));
  CUDA_OR_FAIL(ctx, cudaMemcpyAsync(&h, ctx->d_count, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
  CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  *count = h;
  return FPT_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// learned warm start
// ---------------------------------------------------------------------------
// Scratch for B rows of a forward pass, or of a training batch.
static fpt_status mlp_ensure_ws(fpt_ctx* ctx, fpt_mlp* m, uint64_t B, bool train) {
  const uint64_t rows = B < 128 ? 128 : B;
  const bool shared = !train && rows > m->cap && rows <= m->train_cap;  // a forward pass in the training batch's
  uint64_t& cap = train || shared ? m->train_cap : m->cap;
  const uint64_t want = rows > cap ? rows : cap;
  const size_t elems = train || shared ? want * (6 * kMlpHidden + kMlpIn) + (want + 7) / 8 * 8 * kMlpOut
                                       : want * 2 * kMlpHidden;
  const cudaError_t e = reserve(ctx, train || shared ? m->train : m->fwd, elems * sizeof(__nv_bfloat16), capturing(ctx), true);
  if (e != cudaSuccess) {
    cap = 0;
    return fail(ctx, FPT_ENOMEM, "MLP workspace for %llu rows: %s", (unsigned long long)want, cudaGetErrorString(e));
  }
  cap = want;
  return FPT_OK;
}

static GemmArgs gemm_args(int M, int N, int K, const __nv_bfloat16* A, long long sam, long long sak,
                          const __nv_bfloat16* Bm, long long sbn, long long sbk, int op, int* err) {
  GemmArgs g{};
  g.M = M;
  g.N = N;
  g.K = K;
  g.A = A;
  g.sam = sam;
  g.sak = sak;
  g.B = Bm;
  g.sbn = sbn;
  g.sbk = sbk;
  g.op = op;
  g.err = err;
  return g;
}

// forward pass of B rows of X
static fpt_status mlp_forward_impl(fpt_ctx* ctx, fpt_mlp* m, const __nv_bfloat16* X, uint64_t B, float* Y) {
  const int Bi = (int)B;
  const __nv_bfloat16* W = m->d_wb;
  const float* P = m->d_w;
  const __nv_bfloat16* in = X;
  const bool own = B <= m->cap;  // else the training batch's, which mlp_ensure_ws has found large enough
  __nv_bfloat16* const H1 = own ? static_cast<__nv_bfloat16*>(m->fwd.p) : m->H();
  __nv_bfloat16* const H2 = H1 + (own ? m->cap : m->train_cap) * kMlpHidden;
  __nv_bfloat16* H[3] = {H1, H2, H1};
  const int offW[3] = {kOffW1, kOffW2, kOffW3}, offB[3] = {kOffB1, kOffB2, kOffB3};
  for (int l = 0; l < 3; ++l) {
    const int K = l == 0 ? kMlpIn : kMlpHidden;
    GemmArgs g = gemm_args(Bi, kMlpHidden, K, in, K, 1, W + offW[l], K, 1, EPI_BIAS_GELU, ctx->d_err);
    g.bias = P + offB[l];
    g.H = H[l];
    g.shm = kMlpHidden;
    g.shn = 1;
    CUDA_OR_FAIL(ctx, launch_gemm(g, ctx->stream));
    in = H[l];
  }
  GemmArgs g = gemm_args(Bi, kMlpOut, kMlpHidden, in, kMlpHidden, 1, W + kOffW4, kMlpHidden, 1, EPI_STORE, ctx->d_err);
  g.bias = P + kOffB4;
  g.C = Y;
  g.scm = kMlpOut;
  g.scn = 1;
  CUDA_OR_FAIL(ctx, launch_gemm(g, ctx->stream));
  return FPT_OK;
}

// Loss and gradient (d_loss, d_g) of a batch.  n > 0: row i is sample perm(first + i) of n (fpt_mlp_train).  chained: the
// previous launch on the stream is this network's mlp_adam with `clear`, which left both at zero.
static fpt_status mlp_backward_impl(fpt_ctx* ctx, fpt_mlp* m, const __nv_bfloat16* X, const float* T, const float* G,
                                    uint64_t B, uint64_t n, uint64_t first, uint64_t key, bool chained) {
  fpt_status st = mlp_ensure_ws(ctx, m, B, true);
  if (st != FPT_OK) return st;
  if (!chained) CUDA_OR_FAIL(ctx, cudaMemsetAsync(m->d_g, 0, (kMlpParams + 1) * sizeof(float), ctx->stream));
  TrainArgs a{};
  a.chained = chained;
  a.X = X;
  a.T = T;
  a.G = G;
  a.B = B;
  a.n = n;
  a.first = first;
  a.key = key;
  a.wt = m->d_wt;
  a.wtT = m->d_wtT;
  a.params = m->d_w;
  a.Xb = m->Xb();
  a.H = m->H();
  a.dZ = m->dZ();
  a.dYt = m->dYt();
  a.ldY = (B + 7) / 8 * 8;
  a.grad = m->d_g;
  a.loss = m->d_loss;
  a.err = ctx->d_err;
  CUDA_OR_FAIL(ctx, launch_mlp_train(a, ctx->stream, ctx->n_sm));
  return FPT_OK;
}

// Adam step on d_g; with hist, also *hist += hist_w * the batch's loss; with clear, d_g and d_loss are zero afterwards.
static fpt_status mlp_adam(fpt_ctx* ctx, fpt_mlp* m, float lr, float* hist, float hist_w, bool clear) {
  m->step += 1;
  const float c1 = 1.f - std::pow(0.9f, (float)m->step), c2 = 1.f - std::pow(0.999f, (float)m->step);
  CUDA_OR_FAIL(ctx, launch_adam(m->d_w, m->d_m, m->d_v, m->d_g, lr, c1, c2, m->d_wb, m->d_wt, m->d_wtT, m->d_loss, hist,
                                hist_w, clear, ctx->stream));
  return FPT_OK;
}

// splitmix64 stream for the initial weights
static uint64_t sm64_next(uint64_t& state) {
  uint64_t z = (state += 0x9E3779B97F4A7C15ULL);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

extern "C" {

fpt_status fpt_mlp_create(fpt_ctx* ctx, uint64_t seed, float length_scale, fpt_mlp** out) {
  if (!ctx || !out) return fail(ctx, FPT_EINVAL, "null argument");
  *out = nullptr;
  if (!(length_scale > 0.f) || !std::isfinite(length_scale)) return fail(ctx, FPT_EINVAL, "bad length scale");
  fpt_mlp* m = new (std::nothrow) fpt_mlp();
  if (!m) return FPT_ENOMEM;
  m->ctx = ctx;
  m->scale = length_scale;
  m->seed = seed;
  cudaError_t e = cudaSetDevice(ctx->device);
  for (float** p : {&m->d_w, &m->d_m, &m->d_v, &m->d_g})
    if (e == cudaSuccess) e = cudaMalloc(p, (kMlpParams + 1) * sizeof(float));
  m->d_loss = m->d_g + kMlpParams;
  if (e == cudaSuccess) e = cudaMalloc(&m->d_wb, kMlpParams * sizeof(__nv_bfloat16));
  if (e == cudaSuccess) e = cudaMalloc(&m->d_wt, 2 * kMlpHalfBytes);
  if (e == cudaSuccess) e = cudaMalloc(&m->d_wtT, 2 * kMlpHalfTBytes);
  if (e != cudaSuccess) {
    fpt_mlp_free(m);
    return fail(ctx, FPT_ENOMEM, "MLP parameters: %s", cudaGetErrorString(e));
  }
  std::vector<float> w(kMlpParams, 0.f);
  uint64_t state = seed;
  auto fill = [&](int off, int rows, int cols, int used_rows) {
    const double bound = 1.0 / std::sqrt((double)cols);
    for (int r = 0; r < rows; ++r)
      for (int c = 0; c < cols; ++c) {
        const double u = (double)(sm64_next(state) >> 11) * (1.0 / 9007199254740992.0);
        w[off + r * cols + c] = r < used_rows ? (float)((2.0 * u - 1.0) * bound) : 0.f;
      }
  };
  fill(kOffW1, 256, 64, 256);
  fill(kOffW2, 256, 256, 256);
  fill(kOffW3, 256, 256, 256);
  fill(kOffW4, 16, 256, 8);
  fpt_status st = fpt_mlp_set_params(m, w.data());
  if (st != FPT_OK) {
    fpt_mlp_free(m);
    return st;
  }
  *out = m;
  return FPT_OK;
}

void fpt_mlp_free(fpt_mlp* m) {
  if (!m) return;
  if (m->ctx && m->ctx->init_mlp == m) m->ctx->init_mlp = nullptr;
  cudaFree(m->fwd.p);
  cudaFree(m->train.p);
  for (void* p : {(void*)m->d_w, (void*)m->d_m, (void*)m->d_v, (void*)m->d_g, (void*)m->d_wb, (void*)m->d_wt,
                  (void*)m->d_wtT, (void*)m->d_hist})
    cudaFree(p);
  delete m;
}

fpt_status fpt_mlp_get_params(const fpt_mlp* m, float* host) {
  if (!m || !host) return FPT_EINVAL;
  fpt_ctx* ctx = m->ctx;
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  CUDA_OR_FAIL(ctx, cudaMemcpy(host, m->d_w, kMlpParams * sizeof(float), cudaMemcpyDeviceToHost));
  return FPT_OK;
}

fpt_status fpt_mlp_set_params(fpt_mlp* m, const float* host) {
  if (!m || !host) return FPT_EINVAL;
  fpt_ctx* ctx = m->ctx;
  for (int i = 0; i < kMlpParams; ++i)
    if (!std::isfinite(host[i])) return fail(ctx, FPT_EINVAL, "non-finite parameter %d", i);
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  CUDA_OR_FAIL(ctx, cudaMemcpy(m->d_w, host, kMlpParams * sizeof(float), cudaMemcpyHostToDevice));
  CUDA_OR_FAIL(ctx, cudaMemset(m->d_m, 0, kMlpParams * sizeof(float)));
  CUDA_OR_FAIL(ctx, cudaMemset(m->d_v, 0, kMlpParams * sizeof(float)));
  // every layout that a kernel reads is written here and by each Adam step, so that no call (one recorded in a graph
  // among them) depends on what ran before it
  CUDA_OR_FAIL(ctx, launch_to_bf16(m->d_w, m->d_wb, kMlpParams, ctx->stream));
  CUDA_OR_FAIL(ctx, launch_mlp_tile_weights(m->d_wb, m->d_wt, m->d_wtT, ctx->stream));
  CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  m->step = 0;
  return FPT_OK;
}

static const char kMlpMagic[8] = {'F', 'P', 'T', 'M', 'L', 'P', '0', '1'};

fpt_status fpt_mlp_save(const fpt_mlp* m, const char* path) {
  if (!m || !path) return FPT_EINVAL;
  fpt_ctx* ctx = m->ctx;
  std::vector<float> buf(3 * (size_t)kMlpParams);
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  CUDA_OR_FAIL(ctx, cudaMemcpy(buf.data(), m->d_w, kMlpParams * sizeof(float), cudaMemcpyDeviceToHost));
  CUDA_OR_FAIL(ctx, cudaMemcpy(buf.data() + kMlpParams, m->d_m, kMlpParams * sizeof(float), cudaMemcpyDeviceToHost));
  CUDA_OR_FAIL(ctx, cudaMemcpy(buf.data() + 2 * kMlpParams, m->d_v, kMlpParams * sizeof(float), cudaMemcpyDeviceToHost));
  FILE* f = fopen(path, "wb");
  if (!f) return fail(ctx, FPT_EINVAL, "cannot write %s", path);
  const int32_t n = kMlpParams;
  bool ok = fwrite(kMlpMagic, 1, 8, f) == 8 && fwrite(&n, 4, 1, f) == 1 && fwrite(&m->scale, 4, 1, f) == 1 &&
            fwrite(&m->seed, 8, 1, f) == 1 && fwrite(&m->step, 8, 1, f) == 1 &&
            fwrite(buf.data(), sizeof(float), buf.size(), f) == buf.size();
  ok = (fclose(f) == 0) && ok;
  return ok ? FPT_OK : fail(ctx, FPT_EINVAL, "short write to %s", path);
}

fpt_status fpt_mlp_load(fpt_ctx* ctx, const char* path, fpt_mlp** out) {
  if (!ctx || !path || !out) return fail(ctx, FPT_EINVAL, "null argument");
  *out = nullptr;
  FILE* f = fopen(path, "rb");
  if (!f) return fail(ctx, FPT_EINVAL, "cannot read %s", path);
  char magic[8];
  int32_t n = 0;
  float scale = 0.f;
  uint64_t seed = 0;
  int64_t step = 0;
  std::vector<float> buf(3 * (size_t)kMlpParams);
  bool ok = fread(magic, 1, 8, f) == 8 && memcmp(magic, kMlpMagic, 8) == 0 && fread(&n, 4, 1, f) == 1 &&
            n == kMlpParams && fread(&scale, 4, 1, f) == 1 && fread(&seed, 8, 1, f) == 1 &&
            fread(&step, 8, 1, f) == 1 && fread(buf.data(), sizeof(float), buf.size(), f) == buf.size();
  fclose(f);
  if (!ok) return fail(ctx, FPT_EINVAL, "%s is not a network file of this version", path);
  fpt_mlp* m = nullptr;
  fpt_status st = fpt_mlp_create(ctx, seed, scale, &m);
  if (st != FPT_OK) return st;
  st = fpt_mlp_set_params(m, buf.data());
  if (st == FPT_OK) {
    cudaError_t e = cudaMemcpy(m->d_m, buf.data() + kMlpParams, kMlpParams * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
      e = cudaMemcpy(m->d_v, buf.data() + 2 * kMlpParams, kMlpParams * sizeof(float), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) st = fail(ctx, FPT_ECUDA, "%s", cudaGetErrorString(e));
  }
  if (st != FPT_OK) {
    fpt_mlp_free(m);
    return st;
  }
  m->step = step;
  *out = m;
  return FPT_OK;
}

fpt_status fpt_mlp_features(fpt_ctx* ctx, const fpt_mlp* m, const fpt_scene* s, const fpt_batch* b, void* X,
                            float* G) {
  fpt_status st = check_scene_batch(ctx, s, b);
  if (st != FPT_OK) return st;
  if (!m || !X) return fail(ctx, FPT_EINVAL, "null argument");
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  ProfScope ps(ctx, FPT_K_OTHER);
  CUDA_OR_FAIL(ctx, launch_mlp_features(scene_dev(s), b->dev, 1.f / m->scale, static_cast<__nv_bfloat16*>(X), G,
                                        ctx->stream));
  return FPT_OK;
}

fpt_status fpt_mlp_forward(fpt_ctx* ctx, fpt_mlp* m, const void* X, uint64_t B, float* Y) {
  if (!ctx || !m || !X || !Y) return fail(ctx, FPT_EINVAL, "null argument");
  if (B < 1 || B > (1ull << 30)) return fail(ctx, FPT_EINVAL, "bad batch size");
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  fpt_status st = mlp_ensure_ws(ctx, m, B, false);
  if (st != FPT_OK) return st;
  ProfScope ps(ctx, FPT_K_OTHER);
  return mlp_forward_impl(ctx, m, static_cast<const __nv_bfloat16*>(X), B, Y);
}

fpt_status fpt_mlp_loss_grad(fpt_ctx* ctx, fpt_mlp* m, const void* X, const float* T, const float* G, uint64_t B,
                             float* loss, float* grad_out) {
  if (!ctx || !m || !X || !T || !G) return fail(ctx, FPT_EINVAL, "null argument");
  if (B < 1 || B > (1ull << 30)) return fail(ctx, FPT_EINVAL, "bad batch size");
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  fpt_status st = mlp_backward_impl(ctx, m, static_cast<const __nv_bfloat16*>(X), T, G, B, 0, 0, 0, false);
  if (st != FPT_OK) return st;
  if (grad_out)
    CUDA_OR_FAIL(ctx, cudaMemcpyAsync(grad_out, m->d_g, kMlpParams * sizeof(float), cudaMemcpyDeviceToDevice, ctx->stream));
  if (loss) {
    CUDA_OR_FAIL(ctx, cudaMemcpyAsync(loss, m->d_loss, sizeof(float), cudaMemcpyDeviceToHost, ctx->stream));
    CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  }
  return FPT_OK;
}

fpt_status fpt_mlp_train_step(fpt_ctx* ctx, fpt_mlp* m, const void* X, const float* T, const float* G, uint64_t B,
                              float lr, float* loss) {
  if (!(lr > 0.f)) return fail(ctx, FPT_EINVAL, "learning rate must be positive");
  fpt_status st = fpt_mlp_loss_grad(ctx, m, X, T, G, B, nullptr, nullptr);
  if (st == FPT_OK) st = mlp_adam(ctx, m, lr, nullptr, 0.f, false);
  if (st != FPT_OK) return st;
  if (loss) {
    CUDA_OR_FAIL(ctx, cudaMemcpyAsync(loss, m->d_loss, sizeof(float), cudaMemcpyDeviceToHost, ctx->stream));
    CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  }
  return FPT_OK;
}

fpt_status fpt_mlp_train(fpt_ctx* ctx, fpt_mlp* m, const void* X, const float* T, const float* G, uint64_t n,
                         const fpt_train_params* prm, float* loss_per_epoch) {
  if (!ctx || !m || !prm) return fail(ctx, FPT_EINVAL, "null argument");
  if (m->ctx != ctx) return fail(ctx, FPT_EINVAL, "network belongs to another context");
  const fpt_train_params p = *prm;
  if (p.epochs < 1 || p.batch < 128 || !(p.lr > 0.f) || !(p.lr_decay > 0.f))
    return fail(ctx, FPT_EINVAL, "fpt_mlp_train: epochs >= 1, batch >= 128, lr > 0 and lr_decay > 0 required");
  if ((uint64_t)p.batch > n) return fail(ctx, FPT_EINVAL, "fpt_mlp_train: fewer samples (%llu) than one batch",
                                         (unsigned long long)n);
  if (!X || !T || !G) return fail(ctx, FPT_EINVAL, "fpt_mlp_train: X, T and G are required");
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  const uint64_t B = (uint64_t)p.batch;
  if ((size_t)p.epochs > m->hist_cap) {
    cudaFree(m->d_hist);
    m->d_hist = nullptr;
    m->hist_cap = 0;
    const cudaError_t e = cudaMalloc(&m->d_hist, (size_t)p.epochs * sizeof(float));
    if (e != cudaSuccess) return fail(ctx, FPT_ENOMEM, "fpt_mlp_train: losses: %s", cudaGetErrorString(e));
    m->hist_cap = (size_t)p.epochs;
  }
  CUDA_OR_FAIL(ctx, cudaMemsetAsync(m->d_hist, 0, (size_t)p.epochs * sizeof(float), ctx->stream));
  const uint64_t steps = n / B;  // the last partial batch of every epoch is left out
  const __nv_bfloat16* Xs = static_cast<const __nv_bfloat16*>(X);
  float lr = p.lr;
  for (int ep = 0; ep < p.epochs; ++ep) {
    // (lr_decay can take it to zero)
    if (!(lr > 0.f)) return fail(ctx, FPT_EINVAL, "fpt_mlp_train: learning rate not positive in epoch %d", ep);
    // a new seeded order of the samples every epoch (splitmix64 of seed and epoch)
    uint64_t s0 = p.seed + 0x9E3779B97F4A7C15ULL * (uint64_t)(ep + 1);
    const uint64_t key = sm64_next(s0);
    for (uint64_t k = 0; k < steps; ++k) {
      // the steps of one call are a chain: each starts from the gradient that the one before cleared
      fpt_status st = mlp_backward_impl(ctx, m, Xs, T, G, B, n, k * B, key, ep > 0 || k > 0);
      if (st == FPT_OK) st = mlp_adam(ctx, m, lr, m->d_hist + ep, 1.f / (float)steps, true);
      if (st != FPT_OK) return st;
    }
    lr *= p.lr_decay;
  }
  if (loss_per_epoch) {
    CUDA_OR_FAIL(ctx, cudaMemcpyAsync(loss_per_epoch, m->d_hist, (size_t)p.epochs * sizeof(float),
                                      cudaMemcpyDeviceToHost, ctx->stream));
    CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  }
  return FPT_OK;
}

fpt_status fpt_mlp_infer(fpt_ctx* ctx, fpt_mlp* m, const fpt_scene* s, const fpt_batch* bc, float* T) {
  fpt_status st = check_scene_batch(ctx, s, bc);
  if (st != FPT_OK) return st;
  if (!m) return fail(ctx, FPT_EINVAL, "null network");
  if (m->ctx != ctx) return fail(ctx, FPT_EINVAL, "network belongs to another context");
  if (!T && bc->dev.n_paths > 0) return fail(ctx, FPT_EINVAL, "T_out is required");
  fpt_batch* b = const_cast<fpt_batch*>(bc);
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  st = ensure_buckets(ctx, b, scene_dev(s));
  if (st != FPT_OK) return st;
  const SceneDev S = scene_dev(s);
  if (b->dev.n_paths == 0) return FPT_OK;
  // Records carry their order, and a batch's lists follow the orders: one launch takes all orders whose records
  // hold the ids, one the longer sequences.  The kernel also clears the slots past a path's order.
  const PathRec* first = nullptr;
  uint64_t run = 0;
  for (int n = 1; n <= kMaxOrder; ++n) {
    const PathRec* list;
    const uint64_t cnt = order_slice(b, n, &list);
    if (cnt && !run) first = list;
    run += cnt;
    const bool last = n == kMaxOrder || n == kMaxBfgsOrder || b->dev.mode == BATCH_EXHAUSTIVE;
    if (!run || !last) continue;
    ProfScope ps(ctx, FPT_K_MLP);
    CUDA_OR_FAIL(ctx, launch_mlp_infer(S, b->dev, n, first, run, 1.f / m->scale, m->d_wt, m->d_w, T, b->dev.n_max,
                                       ctx->d_err, ctx->stream, ctx->n_sm));
    run = 0;
  }
  return FPT_OK;
}

fpt_status fpt_set_init_mlp(fpt_ctx* ctx, fpt_mlp* m) {
  if (!ctx) return FPT_EINVAL;
  if (m && m->ctx != ctx) return fail(ctx, FPT_EINVAL, "network belongs to another context");
  ctx->init_mlp = m;
  return FPT_OK;
}

fpt_status fpt_tc_gemm_bf16(fpt_ctx* ctx, int32_t M, int32_t N, int32_t K, const void* A, const void* W,
                            const float* bias, float* C) {
  if (!ctx || !A || !W || !C) return fail(ctx, FPT_EINVAL, "null argument");
  if (M < 1 || K < 1 || N < 1 || N > 256) return fail(ctx, FPT_EINVAL, "bad GEMM shape %d x %d x %d", M, N, K);
  GemmArgs g{};
  g.M = M;
  g.N = N;
  g.K = K;
  g.A = static_cast<const __nv_bfloat16*>(A);
  g.sam = K;
  g.sak = 1;
  g.B = static_cast<const __nv_bfloat16*>(W);
  g.sbn = K;
  g.sbk = 1;
  g.op = EPI_STORE;
  g.bias = bias;
  g.C = C;
  g.scm = N;
  g.scn = 1;
  g.err = ctx->d_err;
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  ProfScope ps(ctx, FPT_K_OTHER);
  CUDA_OR_FAIL(ctx, launch_gemm(g, ctx->stream));
  return FPT_OK;
}

fpt_status fpt_check_bounded_wait(fpt_ctx* ctx, uint32_t limit_us, int arrive, uint64_t* elapsed_ns) {
  if (!ctx) return FPT_EINVAL;
  if (limit_us < 1 || limit_us > 1000000u) return fail(ctx, FPT_EINVAL, "limit %u us outside [1, 10^6]", limit_us);
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  unsigned long long* d_ns = nullptr;
  if (elapsed_ns) CUDA_OR_FAIL(ctx, cudaMalloc(&d_ns, sizeof(unsigned long long)));
  cudaError_t e;
  {
    ProfScope ps(ctx, FPT_K_OTHER);
    e = launch_bounded_wait_check(limit_us * 1000u, arrive, ctx->d_err, d_ns, ctx->stream);
  }
  unsigned long long h = 0;
  if (e == cudaSuccess && elapsed_ns) {
    e = cudaMemcpyAsync(&h, d_ns, sizeof h, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  }
  if (d_ns) cudaFree(d_ns);
  CUDA_OR_FAIL(ctx, e);
  if (elapsed_ns) *elapsed_ns = h;
  return FPT_OK;
}

fpt_status fpt_profile_enable(fpt_ctx* ctx, int on) {
  if (!ctx) return FPT_EINVAL;
  ctx->prof = on != 0;
  return FPT_OK;
}

fpt_status fpt_profile_read(fpt_ctx* ctx, double* ms, uint64_t* launches, int reset) {
  if (!ctx) return FPT_EINVAL;
  CUDA_OR_FAIL(ctx, cudaSetDevice(ctx->device));
  CUDA_OR_FAIL(ctx, cudaStreamSynchronize(ctx->stream));
  for (auto& p : ctx->ev_pending) {
    float t = 0.f;
    if (cudaEventElapsedTime(&t, p.second.first, p.second.second) == cudaSuccess) ctx->prof_ms[p.first] += t;
    ctx->ev_pool.push_back(p.second.first);
    ctx->ev_pool.push_back(p.second.second);
  }
  ctx->ev_pending.clear();
  for (int k = 0; k < FPT_K_COUNT; ++k) {
    if (ms) ms[k] = ctx->prof_ms[k];
    if (launches) launches[k] = ctx->prof_kernels[k];
    if (reset) {
      ctx->prof_ms[k] = 0;
      ctx->prof_kernels[k] = 0;
    }
  }
  return FPT_OK;
}

}  // extern "C"
