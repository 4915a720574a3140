// Host side of the library: argument checks, workspace layout, TMA descriptors, and the
// sequence of launches of the Root Newton-Schulz step (Section 3.4).  Everything here
// only enqueues work on the caller's stream.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>
#include <stdlib.h>
#include <type_traits>
#include <unordered_map>
#include <vector>

#include <cudaTypedefs.h>

#include "fp4_gemm_common.cuh"

namespace fp4 {

namespace {
std::atomic<uint64_t> g_launches{0};
std::atomic<int> g_prof_on{0};
struct ProfRec { int cls; cudaEvent_t e0, e1; };
std::vector<ProfRec> g_prof;
std::mutex g_prof_mu;
}  // namespace

void count_launches(int n) { g_launches.fetch_add((uint64_t)n, std::memory_order_relaxed); }

// Programmatic dependent launch hides a launch behind the kernel before, but a successor's blocks take the SMs as they drain: where
// launches fill the machine for long, the CTA pairs of the next one then lie less favourably.  So each part of a call decides
// (run_group).
namespace {
thread_local bool t_pdl_group = false;
}
bool pdl_enabled() {
  static const bool allowed = getenv("FP4ROOT_NO_PDL") == nullptr;
  return allowed && t_pdl_group;
}
void pdl_select(bool on) { t_pdl_group = on; }

ProfScope::ProfScope(int cls_, cudaStream_t st_) : cls(cls_), st(st_), e0(nullptr), on(g_prof_on.load() != 0) {
  if (on) {
    if (cudaEventCreate(&e0) != cudaSuccess) { on = false; return; }
    cudaEventRecord(e0, st);
  }
}
ProfScope::~ProfScope() {
  if (!on) return;
  cudaEvent_t e1;
  if (cudaEventCreate(&e1) != cudaSuccess) { cudaEventDestroy(e0); return; }
  cudaEventRecord(e1, st);
  std::lock_guard<std::mutex> lock(g_prof_mu);
  g_prof.push_back({cls, e0, e1});
}

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct DeviceInfo {
  bool ready = false;
  fp4_status status = FP4_OK;
  int sms = 0;
  EncodeTiledFn encode = nullptr;
  // of drivers that know them (12.5): the context behind a stream, and what of the device it may use
  PFN_cuStreamGetCtx_v12050 stream_context = nullptr;
  PFN_cuCtxGetDevResource_v12040 context_resource = nullptr;
  PFN_cuGreenCtxGetDevResource_v12040 green_resource = nullptr;
};
DeviceInfo g_dev[64];
std::mutex g_mu;

// Per-device set-up on first use: architecture check, driver entry point, kernel attributes.
const DeviceInfo* device_info() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lock(g_mu);
  DeviceInfo& d = g_dev[dev];
  if (d.ready) return &d;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) { d.status = FP4_ERR_CUDA; d.ready = true; return &d; }
  if (prop.major != 10) { d.status = FP4_ERR_ARCH; d.ready = true; return &d; }
  d.sms = prop.multiProcessorCount;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
      qres != cudaDriverEntryPointSuccess || fn == nullptr) {
    d.status = FP4_ERR_CUDA; d.ready = true; return &d;
  }
  d.encode = reinterpret_cast<EncodeTiledFn>(fn);
  auto optional = [&](const char* name, unsigned version, auto& entry) {
    if (cudaGetDriverEntryPointByVersion(name, &fn, version, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess && fn != nullptr)
      entry = reinterpret_cast<std::decay_t<decltype(entry)>>(fn);
    else
      cudaGetLastError();
  };
  optional("cuStreamGetCtx", 12050, d.stream_context);
  optional("cuCtxGetDevResource", 12040, d.context_resource);
  optional("cuGreenCtxGetDevResource", 12040, d.green_resource);
  if (gemm_pair_set_attributes() != cudaSuccess ||
      chain_set_attributes() != cudaSuccess ||
      prologue_set_attributes() != cudaSuccess || quantize_set_attributes() != cudaSuccess)
    d.status = FP4_ERR_CUDA;
  d.ready = true;
  return &d;
}

// SMs that kernels on this stream can occupy: fewer than the device has where the stream belongs to a green context or to a
// context with a limit of its own.  The cooperative launches need all their blocks resident there.
int stream_sms(const DeviceInfo* d, cudaStream_t st) {
  if (!d->stream_context || !d->context_resource || !d->green_resource) return d->sms;
  CUcontext ctx = nullptr;
  CUgreenCtx green = nullptr;
  CUdevResource r;
  if (d->stream_context(st, &ctx, &green) != CUDA_SUCCESS) return d->sms;
  const CUresult e = green ? d->green_resource(green, &r, CU_DEV_RESOURCE_TYPE_SM) : d->context_resource(ctx, &r, CU_DEV_RESOURCE_TYPE_SM);
  return e == CUDA_SUCCESS && r.sm.smCount > 0 && (int)r.sm.smCount < d->sms ? (int)r.sm.smCount : d->sms;
}

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }
inline bool shape_ok(int64_t v) { return v >= 128 && v % 128 == 0 && v <= (1 << 20); }
// The Newton-Schulz entry points pad internally: any positive multiple of the block length.
inline bool ns_shape_ok(int64_t v) { return v >= 16 && v % 16 == 0 && v <= (1 << 20); }
inline int64_t pad128(int64_t v) { return (v + 127) / 128 * 128; }
// flag bits the Newton-Schulz entry points know
constexpr uint32_t kNsFlags =
    FP4_FLAG_KEEP_OPERANDS | FP4_FLAG_RHT | FP4_FLAG_FOUR_SIX | FP4_FLAG_STORE_BF16 | FP4_FLAG_NO_OUT |
    FP4_FLAG_OVERLAP_GROUPS;

// 2-D map over a row-major byte matrix (NVFP4 codes): box = one operand stage of `stage_k` elements of K
// (64 or 128 bytes x box_rows rows), swizzled over the box width.
bool make_codes_map(const DeviceInfo* d, CUtensorMap* tm, const void* base, int64_t rows, int64_t row_bytes, int stage_k,
                    int box_rows = 128) {
  const cuuint32_t bw = (cuuint32_t)(stage_k / 2);
  cuuint64_t dims[2] = {(cuuint64_t)row_bytes, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)row_bytes};
  cuuint32_t box[2] = {bw, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return d->encode(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, bw == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// 2-D map over a row-major FP32 matrix: box = 16 columns x 32 rows, one epilogue warp's block, 64-byte swizzle.
bool make_f32_map(const DeviceInfo* d, CUtensorMap* tm, const void* base, int64_t rows, int64_t cols) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 4};
  cuuint32_t box[2] = {16, 32};
  cuuint32_t estr[2] = {1, 1};
  return d->encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A contiguous FP32 tensor as rows of 16 elements (one block each): box = 128 blocks, 64-byte swizzle.
bool make_blocks_map(const DeviceInfo* d, CUtensorMap* tm, const void* base, int64_t blocks) {
  cuuint64_t dims[2] = {16, (cuuint64_t)blocks};
  cuuint64_t strides[1] = {64};
  cuuint32_t box[2] = {16, 128};
  cuuint32_t estr[2] = {1, 1};
  return d->encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D map over a row-major FP32 matrix for the operand preparation: box = 32 columns x 128 rows (a quarter
// of a 128 x 128 tile), 128-byte swizzle.
bool make_f32_tile_map(const DeviceInfo* d, CUtensorMap* tm, const void* base, int64_t rows, int64_t cols) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 4};
  cuuint32_t box[2] = {32, 128};
  cuuint32_t estr[2] = {1, 1};
  return d->encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D map over a row-major FP32 matrix whose transpose the CTA-pair kernel works on: box = 32 columns x 16 rows
// (one epilogue warp's 32 x 16 block, transposed), no swizzle.
bool make_f32_tr_map(const DeviceInfo* d, CUtensorMap* tm, const void* base, int64_t rows, int64_t cols) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 4};
  cuuint32_t box[2] = {32, 16};
  cuuint32_t estr[2] = {1, 1};
  return d->encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D map over a row-major BF16 matrix: box = 16 columns x 32 rows (32-byte rows), no swizzle: the block of
// one epilogue warp of the CTA-pair kernel.
bool make_bf16_map(const DeviceInfo* d, CUtensorMap* tm, const void* base, int64_t rows, int64_t cols) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {16, 32};
  cuuint32_t estr[2] = {1, 1};
  return d->encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D map over a row-major byte matrix (NVFP4 codes) for the stores of the CTA-pair kernel's epilogue
// warps: box = box_bytes x box_rows, no swizzle.
bool make_code_store_map(const DeviceInfo* d, CUtensorMap* tm, const void* base, int64_t rows, int64_t row_bytes,
                         int box_bytes, int box_rows, CUtensorMapSwizzle swizzle) {
  cuuint64_t dims[2] = {(cuuint64_t)row_bytes, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)row_bytes};
  cuuint32_t box[2] = {(cuuint32_t)box_bytes, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return d->encode(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

constexpr int kDefaultMaxGroup = kPackMax;

// 2-D map over the scale atoms of a rows x K operand: one map row per 128-row block, 64-bit
// elements, box = the atoms of one operand stage (`stage_k` elements of 8 bytes: 1 or 2 KB), no swizzle.
bool make_sf_map(const DeviceInfo* d, CUtensorMap* tm, const void* base, int64_t rows, int64_t K, int stage_k) {
  cuuint64_t dims[2] = {(cuuint64_t)(K / 64) * 64, (cuuint64_t)(rows / 128)};
  cuuint64_t strides[1] = {(cuuint64_t)(K / 64) * 512};
  cuuint32_t box[2] = {(cuuint32_t)stage_k, 1};
  cuuint32_t estr[2] = {1, 1};
  return d->encode(tm, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

void default_params(fp4_ns_params* p) {
  p->a = p->b = p->c = NAN;
  p->clip_quantile = 0.99f;
  p->eps = 1e-7f;
  p->flags = 0;
  p->max_group = 0;
  p->seed = 0;
  p->top_hist = nullptr;
  p->weights = nullptr;
  p->lr = p->weight_decay = 0.0f;
  p->update_scale = 1.0f;
}

// Quantiser options of the j-th product of a call.
QuantOpts quant_opts(const fp4_ns_params* p, uint64_t j) {
  QuantOpts q;
  q.rht = (p->flags & FP4_FLAG_RHT) ? 1u : 0u;
  q.four_six = (p->flags & FP4_FLAG_FOUR_SIX) ? 1u : 0u;
  q.mask = q.rht ? rht_signs(p->seed, j) : 0u;
  q.widen = q.rht ? 4.0f : 1.0f;
  q.minus_one = -1.0f;
  set_signs(q);
  return q;
}

int64_t quantile_rank(int64_t n, float q) {
  // resolved to parts per million so that 0.99f means 99/100
  int64_t ppm = (int64_t)llround((double)q * 1e6);
  int64_t k = (ppm * n + 999999) / 1000000;
  if (k < 1) k = 1;
  if (k > n) k = n;
  return k;
}

void coeffs(int64_t m, int64_t n, float abc[3]) {
  // quintic with p(1) = 1, p'(1) = 0: b = 2.5 - 2a, c = a - 1.5; a from the aspect ratio
  double s = (double)(m < n ? m : n), l = (double)(m < n ? n : m);
  double delta = (std::sqrt(7.0 / 3.0) - 1.0) / 2.0;
  double rr = 1.0 + delta * (1.0 + std::sqrt(s / l));
  double R = rr * rr;
  double a = (1.5 * R - 1.0) / (R - 1.0);
  abc[0] = (float)a;
  abc[1] = (float)(2.5 - 2.0 * a);
  abc[2] = (float)(a - 1.5);
}

// Workspace layout of one matrix.
fp4_status make_plan(int64_t m, int64_t n, int steps, const fp4_ns_params* p, int sms, NsPlan* pl) {
  if (!ns_shape_ok(m) || !ns_shape_ok(n)) return FP4_ERR_SHAPE;
  if (steps < 0 || steps > kMaxSteps) return FP4_ERR_INVALID_ARG;
  memset(pl, 0, sizeof(*pl));
  pl->m = m; pl->n = n;
  pl->tall = m > n;
  pl->s0 = m < n ? m : n;
  pl->l0 = m < n ? n : m;
  // Zero rows and columns stay zero through the iteration and add nothing to any product or
  // maximum; since the dimensions are multiples of 16 no block mixes data and padding.
  pl->s = pad128(pl->s0);
  pl->l = pad128(pl->l0);
  pl->bf16 = (p->flags & FP4_FLAG_STORE_BF16) != 0;
  const int64_t s = pl->s, l = pl->l;
  pl->clip = p->clip_quantile > 0.0f && p->clip_quantile < 1.0f;
  pl->clip_rank = pl->clip ? quantile_rank(m * n, p->clip_quantile) : 0;
  pl->eps = p->eps;
  pl->sms = sms;
  int64_t blocks = (m * n / 4 + 1023) / 1024;
  pl->stat_blocks = (int)(blocks < 1024 ? blocks : 1024);

  NsScalarIdx& ix = pl->ix;
  ix.tau = 0; ix.nu = 1; ix.inv = 2;
  const int span = kMaxSteps + 2;
  ix.amax_X0 = 8; ix.amax_A0 = 8 + span; ix.sg_X0 = 8 + 2 * span; ix.sg_A0 = 8 + 3 * span; ix.sg_B0 = 8 + 4 * span;
  const size_t scalar_bytes = align_up((size_t)(8 + 5 * span) * 4, 1024);

  fp4_ws_layout& L = pl->lay;
  size_t off = 0;
  L.header = off; off += 1024;
  L.scalars = off; off += scalar_bytes;
  pl->off_hist = off; off += 8192 * 4;
  pl->zero_bytes = off;
  pl->off_partial = off; off += 1024 * 8;
  off = align_up(off, 1024);
  L.X = off; if (pl->tall) off += align_up((size_t)s * l * 4, 1024);
  L.A = off; off += align_up((size_t)s * s * 4, 1024);
  L.qX_codes = off; off += align_up((size_t)s * l / 2, 1024);
  L.qX_scales = off; off += align_up((size_t)s * l / 16, 1024);
  for (int i = 0; i < 2; ++i) {
    L.qXt_codes[i] = off; off += align_up((size_t)s * l / 2, 1024);
    L.qXt_scales[i] = off; off += align_up((size_t)s * l / 16, 1024);
  }
  L.qA_codes = off; off += align_up((size_t)s * s / 2, 1024);
  L.qA_scales = off; off += align_up((size_t)s * s / 16, 1024);
  L.qB_codes = off; off += align_up((size_t)s * s / 2, 1024);
  L.qB_scales = off; off += align_up((size_t)s * s / 16, 1024);
  L.Xh = 0;
  if (pl->bf16) { pl->off_Xh = off; L.Xh = off; off += align_up((size_t)s * l * 2, 1024); }
  L.idx_tau = ix.tau; L.idx_nu = ix.nu; L.idx_inv = ix.inv;
  L.idx_amax_X0 = ix.amax_X0; L.idx_amax_A0 = ix.amax_A0;
  L.idx_sg_X0 = ix.sg_X0; L.idx_sg_A0 = ix.sg_A0; L.idx_sg_B0 = ix.sg_B0;
  L.total = off;
  return FP4_OK;
}

// Everything the launches need to know about one matrix of a call.
struct MatrixCtx {
  NsPlan pl;
  const float* G;
  float* out;
  float* X;        // FP32 X in the work orientation: `out` itself, or the workspace when tall
  uint8_t* ws;     // this matrix's workspace
  GemmProblem g1, g2, g3[2];  // g3[cur]: reads qXt[cur], writes qXt[cur ^ 1]
  GemmProblem g3_first;       // iteration 0: as g3[0], but a wide input's FP32 tile is G itself (no X0 copy)
  bool store_x0;              // the prologue writes X0 in FP32
  int64_t x_rows, x_cols;     // extent (and row pitch) of X
  uint32_t* hist_top;         // the caller's first-pass histogram of G, or null
  uint16_t* W;                // the BF16 parameter that takes Root's update in this call, or null
  CUtensorMap tm_G;           // the caller's matrix for the operand preparation (tiles of 128 x 128)
  CUtensorMap tm_outT;        // tall: the caller's result through transposing boxes
  ChainProblem chain;         // for a run of all iterations in one launch
};

// Estimated times in us of the CTA-pair kernel's launches (see chain_iteration_us): a launch and, per round of 256 x 256
// tiles over the SM pairs, an epilogue or a main loop; a partly filled last round costs half of what it lacks.
struct PairUs {
  double g1, g2, g3;
  PairUs(const WorkShape* w, int count, bool opts, int sms) {
    const double pairs = (double)(sms / 2);
    auto rounds = [](double r) { return (std::ceil(r) + (r > 1.0 ? r : 1.0)) / 2; };
    const double epi = 3.95 * (opts ? 1.5 : 1.0), kb = 0.22;
    double sym = 0.0, full = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;   // tiles, and their times in all
    for (int j = 0; j < count; ++j) {
      const double ts = (double)((w[j].s + 255) / 256), tl = (double)((w[j].l + 255) / 256);
      const double k1 = kb * tl, k2 = kb * ts, n = ts * (ts + 1) / 2;
      sym += n;
      full += ts * tl;
      t1 += n * (epi > k1 ? epi : k1);
      t2 += n * (epi > k2 ? epi : k2);
      t3 += ts * tl * (epi > k2 ? epi : k2);
    }
    const double rs = rounds(sym / pairs), rf = rounds(full / pairs);
    g1 = 6.25 + rs * (t1 / sym);
    g2 = 6.25 + rs * (t2 / sym);
    g3 = 6.25 + rf * (t3 / full);
  }
};

// How a group runs its iterations: all of them in one launch (fp4_chain.cu), three launches of the CTA-pair kernel per
// iteration, or two - G1 and G2 as one launch with a 128 x 128 tile per SM where their 256 x 256 tiles would leave half of
// the SM pairs idle, and the pairs' G3.  What is estimated to be fastest.  Measured, 5 iterations, one launch (width of its tiles) / two /
// three per iteration: 1024 x 1024 102 (64) / 159 / 178 us, 1280 x 8192 304 (64) / 324 / 358, 1280 x 10240 353 (64) / 347 / 380,
// 1536 x 4096 241 (128) / 232 / 254, 2048 x 2048 196 (128) / 200 / 223, 2048 x 8192 502 (128) / 422 / 450, 2304 x 2304 277 (64) / - / 262
// (with the quantiser options 332 / - / 370), 12 x 896 x 896 308 (64) / - / 373, 7 x 1040 x 1040 326 (64) / - / 377, 2 x 1792 x 1792
// 242 (64) / - / 273, 8 x 1280 x 1280 415 (64) / - / 413.  (Not for inspection of BF16-stored intermediates: in single launches A and
// X stay FP32 tensors with rounded values.  Nor, without the options, for long sides beyond 32768, where one launch would be the
// faster, 458 (64) / 559 / 545 at 128 x 56784: these keep the route that they have been tested on.)
constexpr int64_t kChainLong = 32768;
enum Route { kOneLaunch, kTwoLaunches, kThreeLaunches };
struct Plan { Route route; double iteration_us; };
Plan plan_of(const WorkShape* w, int count, const fp4_ns_params* p, int sms) {
  const bool opts = (p->flags & (FP4_FLAG_RHT | FP4_FLAG_FOUR_SIX)) != 0;
  const PairUs pair(w, count, opts, sms);
  Plan plan{kThreeLaunches, pair.g1 + pair.g2 + pair.g3};
  int64_t longest = 0;
  for (int j = 0; j < count; ++j) longest = w[j].l > longest ? w[j].l : longest;
  if (count > kChainMax || (longest > kChainLong && !opts) ||
      ((p->flags & FP4_FLAG_STORE_BF16) && (p->flags & FP4_FLAG_KEEP_OPERANDS)))
    return plan;
  const double sym = chain_symmetric_us(w, count, opts, sms);
  if (sym > 0.0 && sym + pair.g3 < plan.iteration_us) plan = {kTwoLaunches, sym + pair.g3};
  const double one = chain_iteration_us(w, count, opts, sms);
  if (one > 0.0 && one <= plan.iteration_us) plan = {kOneLaunch, one};
  return plan;
}

fp4_status build_matrix(const DeviceInfo* d, const float* G, float* out, int64_t m, int64_t n, int steps,
                        const fp4_ns_params* p, uint8_t* ws, MatrixCtx* c) {
  fp4_status rc = make_plan(m, n, steps, p, d->sms, &c->pl);
  if (rc != FP4_OK) return rc;
  const fp4_ws_layout& L = c->pl.lay;
  const int64_t s = c->pl.s, l = c->pl.l;
  c->G = G; c->out = out; c->ws = ws;
  c->hist_top = nullptr;
  c->W = nullptr;
  c->X = c->pl.tall ? reinterpret_cast<float*>(ws + L.X) : out;
  // extent of X: the padded work shape in the workspace, the caller's shape in `out` (TMA fills what
  // lies outside with zeros on loads and drops it on stores)
  const int64_t xr = c->pl.tall ? s : c->pl.s0, xc = c->pl.tall ? l : c->pl.l0;
  c->x_rows = xr; c->x_cols = xc;
  c->store_x0 = steps == 0;   // else the first G3 stage reads the caller's matrix
  if (!make_f32_tile_map(d, &c->tm_G, G, m, n)) return FP4_ERR_CUDA;
  if (steps == 0) return FP4_OK;
  float abc[3] = {p->a, p->b, p->c};
  if (std::isnan(p->a)) coeffs(m, n, abc);
  CUtensorMap tm_qX, tm_qXt[2], tm_qA, tm_qB, tm_A, tm_X;
  CUtensorMap sf_qX, sf_qXt[2], sf_qA, sf_qB;
  // every operand is read by exactly one stage: its descriptors take that stage's depth in K
  const int k1 = gemm_pair_stage_k(kG1), k2 = gemm_pair_stage_k(kG2), k3 = gemm_pair_stage_k(kG3);
  bool ok = make_sf_map(d, &sf_qX, ws + L.qX_scales, s, l, k1) && make_sf_map(d, &sf_qXt[0], ws + L.qXt_scales[0], l, s, k3) &&
            make_sf_map(d, &sf_qXt[1], ws + L.qXt_scales[1], l, s, k3) && make_sf_map(d, &sf_qA, ws + L.qA_scales, s, s, k2) &&
            make_sf_map(d, &sf_qB, ws + L.qB_scales, s, s, k3) &&
            make_codes_map(d, &tm_qX, ws + L.qX_codes, s, l / 2, k1) &&
            make_codes_map(d, &tm_qXt[0], ws + L.qXt_codes[0], l, s / 2, k3) &&
            make_codes_map(d, &tm_qXt[1], ws + L.qXt_codes[1], l, s / 2, k3) &&
            make_codes_map(d, &tm_qA, ws + L.qA_codes, s, s / 2, k2) &&
            make_codes_map(d, &tm_qB, ws + L.qB_codes, s, s / 2, k3) &&
            make_f32_map(d, &tm_A, ws + L.A, s, s) && make_f32_map(d, &tm_X, c->X, xr, xc);
  if (!ok) return FP4_ERR_CUDA;
  // stores of the quantised outputs by the CTA-pair kernel's epilogue warps
  CUtensorMap st_qA_r, st_qA_c, st_qB_r, st_qB_c, st_qX_r, st_qXt_c[2];
  ok = make_code_store_map(d, &st_qA_r, ws + L.qA_codes, s, s / 2, 32, 32, CU_TENSOR_MAP_SWIZZLE_32B) &&
       make_code_store_map(d, &st_qA_c, ws + L.qA_codes, s, s / 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_64B) &&
       make_code_store_map(d, &st_qB_r, ws + L.qB_codes, s, s / 2, 32, 32, CU_TENSOR_MAP_SWIZZLE_32B) &&
       make_code_store_map(d, &st_qB_c, ws + L.qB_codes, s, s / 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_64B) &&
       make_code_store_map(d, &st_qX_r, ws + L.qX_codes, s, l / 2, 32, 32, CU_TENSOR_MAP_SWIZZLE_32B) &&
       make_code_store_map(d, &st_qXt_c[0], ws + L.qXt_codes[0], l, s / 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_64B) &&
       make_code_store_map(d, &st_qXt_c[1], ws + L.qXt_codes[1], l, s / 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_64B);
  if (!ok) return FP4_ERR_CUDA;
  GemmProblem base;
  memset(&base, 0, sizeof(base));
  base.scalars = reinterpret_cast<float*>(ws + L.scalars);
  base.ca = abc[0]; base.cb = abc[1]; base.cc = abc[2];
  base.out_rows = (int)s; base.out_cols = (int)s;
  base.K = (int)s;
  base.blocks_m = base.blocks_n = (int)(s / 128);
  base.l_cols = (float)l;
  const bool bf16 = c->pl.bf16 != 0;
  CUtensorMap tm_Ah, tm_Xh;
  uint8_t* Xh = bf16 ? ws + c->pl.off_Xh : nullptr;
  if (bf16 && (!make_bf16_map(d, &tm_Ah, ws + L.A, s, s) || !make_bf16_map(d, &tm_Xh, Xh, s, l))) return FP4_ERR_CUDA;
  // G1: A = qX qX^T (upper-triangle tiles), qA in both triangles
  c->g1 = base;
  c->g1.K = (int)l;
  c->g1.tmA = c->g1.tmB = tm_qX; c->g1.tmAux = c->g1.tmOut = tm_A;
  c->g1.tmRq = st_qA_r; c->g1.tmCq = st_qA_c;
  c->g1.tmSfa = c->g1.tmSfb = sf_qX;
  c->g1.rq_sf = c->g1.cq_sf = ws + L.qA_scales;
  if (bf16) c->g1.tmH = tm_Ah;                                           // A as a BF16 tensor
  // G2: B = bA + c qA qA^T, qB in both triangles
  c->g2 = base;
  c->g2.tmA = c->g2.tmB = tm_qA; c->g2.tmAux = c->g2.tmOut = tm_A;
  c->g2.tmRq = st_qB_r; c->g2.tmCq = st_qB_c;
  c->g2.tmSfa = c->g2.tmSfb = sf_qA;
  if (bf16) c->g2.tmH = tm_Ah;
  c->g2.rq_sf = c->g2.cq_sf = ws + L.qB_scales;
  // G3: X+ = aX + qB qXt^T in place on X; new operand copies
  for (int cur = 0; cur < 2; ++cur) {
    GemmProblem& g = c->g3[cur];
    g = base;
    g.blocks_n = (int)(l / 128);
    g.tmA = tm_qB; g.tmB = tm_qXt[cur]; g.tmAux = g.tmOut = tm_X;
    g.out_rows = (int)xr; g.out_cols = (int)xc;
    if (bf16) g.tmH = tm_Xh;
    g.tmSfa = sf_qB; g.tmSfb = sf_qXt[cur];
    g.rq_sf = ws + L.qX_scales;
    g.cq_sf = ws + L.qXt_scales[cur ^ 1];
    g.tmRq = st_qX_r; g.tmCq = st_qXt_c[cur ^ 1];
  }
  {
    ChainProblem& h = c->chain;
    memset(&h, 0, sizeof(h));
    const bool tall = c->pl.tall;
    auto load = [&](CUtensorMap* m, size_t off, int64_t rows, int64_t k) { return make_codes_map(d, m, ws + off, rows, k / 2, 256, 64); };
    auto rows32 = [&](CUtensorMap* m, size_t off, int64_t k) { return make_code_store_map(d, m, ws + off, s, k / 2, 32, 128, CU_TENSOR_MAP_SWIZZLE_32B); };
    auto cols64 = [&](CUtensorMap* m, size_t off, int64_t rows) { return make_code_store_map(d, m, ws + off, rows, s / 2, 64, 64, CU_TENSOR_MAP_SWIZZLE_64B); };
    if (!load(&h.tm_qX, L.qX_codes, s, l) || !load(&h.tm_qXt[0], L.qXt_codes[0], l, s) || !load(&h.tm_qXt[1], L.qXt_codes[1], l, s) ||
        !load(&h.tm_qA, L.qA_codes, s, s) || !load(&h.tm_qB, L.qB_codes, s, s) ||
        !rows32(&h.st_qX, L.qX_codes, l) || !rows32(&h.st_qA, L.qA_codes, s) || !rows32(&h.st_qB, L.qB_codes, s) ||
        !cols64(&h.st_qXt[0], L.qXt_codes[0], l) || !cols64(&h.st_qXt[1], L.qXt_codes[1], l) ||
        !cols64(&h.st_qAc, L.qA_codes, s) || !cols64(&h.st_qBc, L.qB_codes, s) ||
        !make_f32_map(d, &h.tm_A, ws + L.A, s, s) || !make_f32_map(d, &h.tm_X, c->X, xr, xc) ||
        !(tall ? make_f32_tr_map(d, &h.tm_G, G, c->pl.l0, c->pl.s0) && make_f32_tr_map(d, &h.tm_outT, out, c->pl.l0, c->pl.s0)
               : make_f32_map(d, &h.tm_G, G, c->pl.s0, c->pl.l0)))
      return FP4_ERR_CUDA;
    h.scalars = base.scalars;
    h.done = &reinterpret_cast<NsHeader*>(ws + L.header)->tiles_done;
    h.qx_sf = ws + L.qX_scales;
    for (int i = 0; i < 2; ++i) h.qt_sf[i] = ws + L.qXt_scales[i];
    h.qa_sf = ws + L.qA_scales; h.qb_sf = ws + L.qB_scales;
    h.ca = abc[0]; h.cb = abc[1]; h.cc = abc[2];
    h.tall = tall;
    h.s = (int)s; h.l = (int)l; h.s0 = (int)c->pl.s0; h.l0 = (int)c->pl.l0;
    h.l_cols = (float)l;
  }
  c->g3_first = c->g3[0];
  if (c->pl.tall) {
    // the caller's matrices are l0 x s0
    CUtensorMap tm_Gt;
    if (!make_f32_tr_map(d, &tm_Gt, G, c->pl.l0, c->pl.s0) || !make_f32_tr_map(d, &c->tm_outT, out, c->pl.l0, c->pl.s0))
      return FP4_ERR_CUDA;
    c->g3_first.tmAux = tm_Gt;
    c->g3_first.aux_raw = 1;
    c->g3_first.aux_tr = 1;
  } else {
    CUtensorMap tm_G;
    if (!make_f32_map(d, &tm_G, G, c->pl.s0, c->pl.l0)) return FP4_ERR_CUDA;
    c->g3_first.tmAux = tm_G;
    c->g3_first.aux_raw = 1;
  }
  return FP4_OK;
}

// Everything build_matrix derives (workspace plan, some forty TMA descriptors, the problem
// descriptions) depends only on the pointers, the shape and a few parameters: an optimiser calls with
// the same buffers every step, so the results are kept, keyed by exactly those inputs.  The library
// keeps no other state between calls; a hit costs one hash lookup instead of some forty driver calls.
struct CtxKey {
  int dev; int steps; uint32_t flags;
  const void* G; const void* out; const void* ws;
  int64_t m, n;
  uint32_t a, b, c, q, eps;   // bit patterns of the float parameters
  bool operator==(const CtxKey& o) const {
    return dev == o.dev && steps == o.steps && flags == o.flags && G == o.G && out == o.out && ws == o.ws && m == o.m &&
           n == o.n && a == o.a && b == o.b && c == o.c && q == o.q && eps == o.eps;
  }
};
struct CtxKeyHash {
  size_t operator()(const CtxKey& k) const {
    uint64_t h = 1469598103934665603ull;
    auto mix = [&](uint64_t v) { h = (h ^ v) * 1099511628211ull; };
    mix((uint64_t)k.dev); mix((uint64_t)k.steps); mix(k.flags);
    mix((uint64_t)(uintptr_t)k.G); mix((uint64_t)(uintptr_t)k.out); mix((uint64_t)(uintptr_t)k.ws);
    mix((uint64_t)k.m); mix((uint64_t)k.n); mix(k.a); mix(k.b); mix(k.c); mix(k.q); mix(k.eps);
    return (size_t)h;
  }
};
std::unordered_map<CtxKey, MatrixCtx, CtxKeyHash> g_ctx_cache;
std::mutex g_ctx_mu;
constexpr size_t kCtxCacheMax = 1024;   // entries (about 8 KB each); the cache is emptied when it is full

inline uint32_t fbits(float v) { uint32_t u; memcpy(&u, &v, 4); return u; }

fp4_status prepare_matrix(const DeviceInfo* d, const float* G, float* out, int64_t m, int64_t n, int steps,
                          const fp4_ns_params* p, uint8_t* ws, MatrixCtx* c) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return FP4_ERR_CUDA;
  // NO_OUT only matters to the launch sequence, not to what is prepared here
  const CtxKey key{dev, steps, p->flags & ~FP4_FLAG_NO_OUT, G, out, ws, m, n,
                   fbits(p->a), fbits(p->b), fbits(p->c), fbits(p->clip_quantile), fbits(p->eps)};
  {
    std::lock_guard<std::mutex> lock(g_ctx_mu);
    auto it = g_ctx_cache.find(key);
    if (it != g_ctx_cache.end()) { *c = it->second; return FP4_OK; }
  }
  fp4_status rc = build_matrix(d, G, out, m, n, steps, p, ws, c);
  if (rc != FP4_OK) return rc;
  std::lock_guard<std::mutex> lock(g_ctx_mu);
  if (g_ctx_cache.size() >= kCtxCacheMax) g_ctx_cache.clear();
  g_ctx_cache.emplace(key, *c);
  return FP4_OK;
}

// Enqueue the whole step for a group of matrices: the prologue, then every Newton-Schulz stage as one launch over all
// matrices of the group.
// count <= kPackMax: the problems of a launch travel as its parameter.
fp4_status run_group(const DeviceInfo* d, MatrixCtx* mats, int count, int steps, const fp4_ns_params* p,
                     uint32_t* status, bool clear_status, bool two_streams, cudaStream_t st) {
  if (count < 1 || count > kPackMax) return FP4_ERR_INVALID_ARG;
  const bool keep = (p->flags & FP4_FLAG_KEEP_OPERANDS) != 0;
  ParamUpdate upd;
  upd.W = nullptr;
  {
    // every operation rounded to FP32 on its own (volatile keeps the host compiler from fusing them)
    volatile float t = p->lr * p->weight_decay;
    volatile float dec = 1.0f - t;
    volatile float stp = p->lr * p->update_scale;
    upd.decay = dec;
    upd.step = stp;
  }
  upd.no_out = (p->flags & FP4_FLAG_NO_OUT) ? 1 : 0;
  bool any_update = false;
  for (int i = 0; i < count; ++i) any_update = any_update || mats[i].W != nullptr;
  std::vector<char> fused_update((size_t)count, 0);
  // a tall input's result leaves the last G3 stage transposed (no transpose pass) unless that stage also has to
  // write operand copies
  std::vector<char> direct_out((size_t)count, 0);
  bool any_direct = false;
  for (int i = 0; i < count; ++i)
    if (steps > 0 && mats[i].pl.tall && !keep) { direct_out[(size_t)i] = 1; any_direct = true; }
  const NsPlan& pl0 = mats[0].pl;   // for what does not depend on the shape
  WorkShape shapes[kPackMax];
  int64_t elements = 0;
  for (int i = 0; i < count; ++i) {
    shapes[i] = {mats[i].pl.s, mats[i].pl.l};
    elements += mats[i].pl.s * mats[i].pl.l;
  }
  // A cooperative launch that needs more than half of the SMs keeps the other stream's group waiting: the two take half each, and
  // what does not fit is left to the plain launches, which share the SMs as they become free.
  // Measured, 5 iterations, one stream / two with whole-device launches / with halves: six groups of one matrix (1536 x 1536 ..
  // 2816) 1177 / 1160 / 834 us, eight of one (640 x 640 .. 1536) 885 / 680 / 490, six of two (1280 x 1280 .. 2560)
  // 1197 / 1184 / 996, eight tiny ones 780 / 405 / 407; four groups of four with the quantiser options lose (1323 / 1447).
  const int sms = stream_sms(d, st), coop_sms = two_streams && sms > 1 ? sms / 2 : sms;
  const Route route = steps > 0 ? plan_of(shapes, count, p, coop_sms).route : kThreeLaunches;
  {
    std::vector<PrologueItem> items((size_t)count);
    for (int i = 0; i < count; ++i) {
      MatrixCtx& c = mats[i];
      items[(size_t)i] = PrologueItem{c.G, c.X, c.ws, &c.pl, clear_status && reinterpret_cast<uint32_t*>(c.ws + c.pl.lay.header) == status, c.store_x0, c.x_rows, c.x_cols,
                                      c.hist_top, &c.tm_G};
    }
    // Up to 64 M elements the launches of the prologue are short: 8192 x 2048 413 -> 406 us, 1536 x 8192 345 -> 334, a decoder block
    // 2048 wide (44 M) 1009 -> 995; the 28 matrices of four blocks 3072 wide 10.22 -> 10.24 ms.
    pdl_select(elements <= (int64_t)64 << 20);
    if (launch_prologue_group(items.data(), count, steps > 0 || keep, quant_opts(p, 0), status, coop_sms, sms, st) != cudaSuccess)
      return FP4_ERR_CUDA;
  }
  // The stages: always where two short launches make an iteration (2048 x 8192, chained / plain, 396 / 406 us, with options 548 / 560,
  // 2048 x 16384 681 / 690, 1024 x 30720 720 / 729); with three up to some 13 M elements (2304 x 4096 312 / 324, 3072 x 3072 373 / 391,
  // 3072 x 4096 444 / 454, 3584 x 3584 466 / 475, 2560 x 5120 394 / 394; but 2304 x 6144 408 / 389, 2560 x 8192 545 / 526, 4096 x 4096
  // 610 / 600, one decoder block 1536 wide 581 / 566), with the quantiser options 8 M (2560 x 3200 438 / 438, 3072 x 4096
  // 654 / 622, 4096 x 4096 814 / 738).
  const bool opts = (p->flags & (FP4_FLAG_RHT | FP4_FLAG_FOUR_SIX)) != 0;
  pdl_select(route != kThreeLaunches || elements <= (opts ? (int64_t)8 << 20 : (int64_t)25 << 19));
  ChainPack pack;
  ChainLaunch a;
  if (route != kThreeLaunches) {
    for (int j = 0; j < kChainMax; ++j) {
      pack.p[j] = mats[j < count ? j : 0].chain;
      pack.p[j].W = mats[j < count ? j : 0].W;
    }
    memset(&a, 0, sizeof(a));
    a.count = count; a.steps = steps;
    a.clip = pl0.clip; a.keep = keep; a.bf16 = pl0.bf16;
    for (int j = 0; j < count; ++j) a.tall |= mats[j].pl.tall;
    a.update = any_update && !keep; a.no_out = upd.no_out; a.upd_decay = upd.decay; a.upd_step = upd.step;
    a.q = quant_opts(p, 0);
    a.seed = p->seed;
    a.ix = pl0.ix;
    a.status = status;
  }
  if (route == kOneLaunch) {
    for (int j = 0; j < count; ++j) {
      // the parameter updates are written there, too, unless operand copies are kept
      if (!keep) fused_update[(size_t)j] = 1;
    }
    ProfScope ps(FP4_PROF_G3, st);
    if (launch_chain(pack, a, coop_sms, sms == d->sms, st) != cudaSuccess) return FP4_ERR_CUDA;
  } else if (steps > 0) {
    // the problems of the five kinds of launches: G1, G2, G3 reading qXt[0] / qXt[1], the first G3
    std::vector<ProblemPack> packs(5);
    for (int kind = 0; kind < 5; ++kind) {
      for (int j = 0; j < kPackMax; ++j) {
        const MatrixCtx& c = mats[j < count ? j : 0];
        packs[(size_t)kind].p[j] = kind == 0 ? c.g1 : kind == 1 ? c.g2 : kind == 4 ? c.g3_first : c.g3[kind - 2];
      }
    }
    // Root's parameter update: fused into the last G3 stage when no operand copies are wanted from that stage; else into the final
    // transpose for a tall matrix, and a separate elementwise pass otherwise (below).
    if (!keep) {
      for (int kind = 2; kind < 5; ++kind)
        for (int j = 0; j < count; ++j)
          if (mats[j].W) {
            packs[(size_t)kind].p[j].W = mats[j].W;
            packs[(size_t)kind].p[j].W_ld = mats[j].pl.n;
            fused_update[(size_t)j] = 1;
          }
    }
    GemmLaunch base;
    memset(&base, 0, sizeof(base));
    base.num_problems = count;
    base.ix = pl0.ix;
    base.status = status;
    base.clip = pl0.clip;
    const int bf16 = pl0.bf16;
    for (int k = 0; k < steps; ++k) {
      const int cur = k & 1;
      const bool last = (k == steps - 1);
      GemmLaunch L1 = base;
      L1.iter = k; L1.symmetric = 1; L1.write_q = 1;
      L1.q = quant_opts(p, 2 * (uint64_t)k + 1);  // qA_k
      L1.out_h = bf16;
      if (route == kTwoLaunches) {
        ProfScope ps(FP4_PROF_G1, st);
        if (launch_chain_symmetric(pack, a, k, coop_sms, sms == d->sms, st) != cudaSuccess) return FP4_ERR_CUDA;
      } else {
        ProfScope ps(FP4_PROF_G1, st);
        if (launch_gemm_pair(kG1, packs[0], L1, sms, st) != cudaSuccess)
          return FP4_ERR_CUDA;
      }
      GemmLaunch L2 = L1;
      L2.q = quant_opts(p, 2 * (uint64_t)k);      // qB_k meets qX_k^{16x1}
      L2.out_h = 0; L2.aux_h = bf16;
      if (route == kThreeLaunches) {
        ProfScope ps(FP4_PROF_G2, st);
        if (launch_gemm_pair(kG2, packs[1], L2, sms, st) != cudaSuccess)
          return FP4_ERR_CUDA;
      }
      GemmLaunch L3 = base;
      L3.iter = k; L3.symmetric = 0;
      L3.write_q = (!last || keep) ? 1 : 0;
      L3.q = quant_opts(p, 2 * (uint64_t)k + 2);  // both copies of X_{k+1}
      L3.aux_h = k > 0 ? bf16 : 0;   // X_0 is FP32 (or the raw input)
      L3.out_h = last ? 0 : bf16;                 // the result itself is FP32
      if (last && !keep && any_update) {
        L3.update = 1;
        L3.upd_decay = upd.decay; L3.upd_step = upd.step;
        L3.no_out = upd.no_out;
      }
      ProblemPack* pk = &packs[k == 0 ? 4 : 2 + cur];
      ProblemPack last_pack;
      if (last && any_direct) {
        // tall inputs whose result goes straight to the caller's matrix, transposed on the way out
        last_pack = *pk;
        for (int j = 0; j < count; ++j)
          if (direct_out[(size_t)j]) {
            GemmProblem& g = last_pack.p[j];
            g.tmOut = mats[j].tm_outT;
            g.out_tr = 1;
            g.out_rows = (int)mats[j].pl.s0; g.out_cols = (int)mats[j].pl.l0;
          }
        pk = &last_pack;
      }
      {
        ProfScope ps(FP4_PROF_G3, st);
        if (launch_gemm_pair(kG3, *pk, L3, sms, st) != cudaSuccess)
          return FP4_ERR_CUDA;
      }
    }
  }
  for (int i = 0; i < count; ++i) {
    ParamUpdate u = upd;
    u.W = mats[i].W;
    if (direct_out[(size_t)i]) continue;
    if (mats[i].pl.tall) {
      ProfScope ps(FP4_PROF_TRANSPOSE, st);
      if (launch_transpose_out(mats[i].X, mats[i].pl.s, mats[i].pl.l, mats[i].out, mats[i].pl.s0, mats[i].pl.l0, u, st) != cudaSuccess) return FP4_ERR_CUDA;
    } else if (u.W && !fused_update[(size_t)i]) {
      ProfScope ps(FP4_PROF_TRANSPOSE, st);
      if (launch_param_update(mats[i].out, mats[i].pl.m * mats[i].pl.n, u, sms, st) != cudaSuccess) return FP4_ERR_CUDA;
    }
  }
  return FP4_OK;
}

// Matrices of one shape form a group whose stages run as single launches over all of them (many tiles per launch: no idle SMs
// in a last partial wave, the two CTAs of an SM fall out of step so that main loops and epilogues overlap).  A group has at most
// `cap` matrices, which bounds the working set competing for L2.
std::vector<std::vector<MatrixCtx>> group_by_shape(const std::vector<MatrixCtx>& ctx, int cap) {
  const size_t count = ctx.size();
  std::vector<char> done(count, 0);
  std::vector<std::vector<MatrixCtx>> groups;
  for (size_t i = 0; i < count; ++i) {
    if (done[i]) continue;
    groups.emplace_back();
    std::vector<MatrixCtx>& group = groups.back();
    for (size_t j = i; j < count && (int)group.size() < cap; ++j) {
      if (!done[j] && ctx[j].pl.s0 == ctx[i].pl.s0 && ctx[j].pl.l0 == ctx[i].pl.l0) {
        group.push_back(ctx[j]);
        done[j] = 1;
      }
    }
  }
  return groups;
}

// Groups of different shapes run together where one set of launches over all their tiles is estimated to be the faster: a launch
// has a start, a last partial wave and, in a prologue, passes of one block that all matrices share.  The groups are ordered by their
// short side, then the long one, descending (the longest main loops first in a launch's tile list), and neighbours
// merge, the best pair first.  Measured, the groups one after the other / together: the 14 matrices of two decoder blocks 512 wide (four each of
// 512 x 512 and 128 x 512, six of 512 x 1536) 310 / 172 us, of one 1024 wide (1024, 256, 2816) 470 / 323, of two 1600 wide (400,
// 4304) 1425 / 1220, of one 4096 wide (1024, 11008) with the quantiser options 5600 / 5420, the optimiser step around one
// 3072 wide (8192) 3240 / 3095.  (Single matrices only join a group, they do not form one, although they
// would gain, too: six of 1536 x 1536 .. 2816 take 1177 us, with FP4_FLAG_OVERLAP_GROUPS 823, together 540; 192 x 176 and 256 x 272 with BF16
// storage 146, together 83.  A test of that option takes a call of single matrices as the case that it makes faster.)  The group of the call's first matrix, whose prologue clears the status word, comes first.
void merge_groups(std::vector<std::vector<MatrixCtx>>& groups, int cap, int steps, const fp4_ns_params* p, int device_sms, int sms) {
  if (groups.size() < 2) return;
  const uint8_t* first = groups[0][0].ws;
  std::vector<std::vector<WorkShape>> shapes;
  auto estimate = [&](const std::vector<WorkShape>& w) {
    const double prologue = prologue_us(w.data(), (int)w.size(), device_sms, sms);
    return steps > 0 ? prologue + steps * plan_of(w.data(), (int)w.size(), p, sms).iteration_us : prologue;
  };
  std::sort(groups.begin(), groups.end(), [](const std::vector<MatrixCtx>& a, const std::vector<MatrixCtx>& b) {
    return a[0].pl.s != b[0].pl.s ? a[0].pl.s > b[0].pl.s : a[0].pl.l > b[0].pl.l;
  });
  std::vector<double> alone, together;   // of every group; of it and the next one
  for (const auto& g : groups) {
    shapes.emplace_back();
    for (const MatrixCtx& c : g) shapes.back().push_back({c.pl.s, c.pl.l});
    alone.push_back(estimate(shapes.back()));
  }
  auto pair_us = [&](size_t i) {
    if (shapes[i].size() + shapes[i + 1].size() > (size_t)cap || (shapes[i].size() == 1 && shapes[i + 1].size() == 1)) return 1e30;
    std::vector<WorkShape> w = shapes[i];
    w.insert(w.end(), shapes[i + 1].begin(), shapes[i + 1].end());
    return estimate(w);
  };
  for (size_t i = 0; i + 1 < groups.size(); ++i) together.push_back(pair_us(i));
  for (;;) {
    size_t best = 0;
    double gain = 0.0;
    for (size_t i = 0; i + 1 < groups.size(); ++i) {
      const double saved = alone[i] + alone[i + 1] - together[i];
      if (saved > gain) { gain = saved; best = i; }
    }
    if (gain <= 0.0) break;
    groups[best].insert(groups[best].end(), groups[best + 1].begin(), groups[best + 1].end());
    shapes[best].insert(shapes[best].end(), shapes[best + 1].begin(), shapes[best + 1].end());
    alone[best] = together[best];
    groups.erase(groups.begin() + best + 1);
    shapes.erase(shapes.begin() + best + 1);
    alone.erase(alone.begin() + best + 1);
    together.erase(together.begin() + best);
    if (best > 0) together[best - 1] = pair_us(best - 1);
    if (best + 1 < groups.size()) together[best] = pair_us(best);
  }
  for (size_t i = 1; i < groups.size(); ++i)
    for (const MatrixCtx& c : groups[i])
      if (c.ws == first) { std::swap(groups[0], groups[i]); return; }
}

// Enqueue the whole step for one matrix.
fp4_status run_one(const DeviceInfo* d, const float* G, float* out, int64_t m, int64_t n, int steps,
                   const fp4_ns_params* p, uint8_t* ws, bool clear_status, cudaStream_t st) {
  MatrixCtx c;
  fp4_status rc = prepare_matrix(d, G, out, m, n, steps, p, ws, &c);
  if (rc != FP4_OK) return rc;
  if (p->top_hist) c.hist_top = p->top_hist[0];
  if (p->weights) c.W = p->weights[0];
  return run_group(d, &c, 1, steps, p, reinterpret_cast<uint32_t*>(ws + c.pl.lay.header), clear_status, false, st);
}

fp4_status check_common(const DeviceInfo** d) {
  *d = device_info();
  if (*d == nullptr) return FP4_ERR_CUDA;
  return (*d)->status;
}

}  // namespace
}  // namespace fp4

using namespace fp4;

extern "C" {

const char* fp4_status_string(fp4_status s) {
  switch (s) {
    case FP4_OK: return "ok";
    case FP4_ERR_INVALID_ARG: return "invalid argument";
    case FP4_ERR_SHAPE: return "unsupported shape (Newton-Schulz entry points: positive multiples of 16; fp4_quantize, fp4_gemm_nt: of 128)";
    case FP4_ERR_ALIGNMENT: return "misaligned pointer";
    case FP4_ERR_WORKSPACE: return "workspace too small";
    case FP4_ERR_ARCH: return "device is not compute capability 10.x (sm_100a kernels only, no fallback)";
    case FP4_ERR_CUDA: return "CUDA runtime or driver call failed";
    case FP4_ERR_DEVICE_TIMEOUT: return "a kernel gave up on a bounded wait";
    case FP4_ERR_UNIMPLEMENTED: return "not implemented";
    case FP4_ERR_STATIC_LIMIT: return "problem needs more scratch than the library's built-in static array holds";
  }
  return "unknown status";
}

size_t fp4_scale_bytes(int64_t rows, int64_t cols) {
  if (rows <= 0 || cols <= 0) return 0;
  return (size_t)((rows + 127) / 128) * (size_t)((cols + 63) / 64) * 512;
}

fp4_status fp4_quantize(const float* x, int64_t rows, int64_t cols, uint8_t* codes, uint8_t* scales,
                        float* tensor_scale, uint32_t flags, cudaStream_t stream) {
  if (!x || !codes || !scales || !tensor_scale) return FP4_ERR_INVALID_ARG;
  if (flags & 0xFFFFu & ~(FP4_FLAG_RHT | FP4_FLAG_FOUR_SIX)) return FP4_ERR_INVALID_ARG;
  if (!(flags & FP4_FLAG_RHT) && (flags >> 16)) return FP4_ERR_INVALID_ARG;
  QuantOpts q;
  q.rht = (flags & FP4_FLAG_RHT) ? 1u : 0u;
  q.four_six = (flags & FP4_FLAG_FOUR_SIX) ? 1u : 0u;
  q.mask = flags >> 16;
  q.widen = q.rht ? 4.0f : 1.0f;
  q.minus_one = -1.0f;
  set_signs(q);
  if (!shape_ok(rows) || !shape_ok(cols)) return FP4_ERR_SHAPE;
  if (!aligned(x, 16) || !aligned(codes, 16) || !aligned(scales, 16) || !aligned(tensor_scale, 4))
    return FP4_ERR_ALIGNMENT;
  const DeviceInfo* d;
  fp4_status rc = check_common(&d);
  if (rc != FP4_OK) return rc;
  CUtensorMap tm;
  const int sms = stream_sms(d, stream);
  const bool small = quantize_fits_smem(rows * cols, sms);
  if (small && !make_blocks_map(d, &tm, x, rows * cols / 16)) return FP4_ERR_CUDA;
  ProfScope ps(FP4_PROF_QUANTIZE, stream);
  return launch_quantize(small ? &tm : nullptr, x, rows, cols, codes, scales, tensor_scale, q, sms, stream) == cudaSuccess
             ? FP4_OK
             : FP4_ERR_CUDA;
}

fp4_status fp4_selftest_quantize_wait(const float* x, int64_t rows, int64_t cols, uint8_t* codes, uint8_t* scales,
                                      float* tensor_scale, uint32_t limit_us, cudaStream_t stream) {
  if (!x || !codes || !scales || !tensor_scale || limit_us < 1 || limit_us > 100000) return FP4_ERR_INVALID_ARG;
  if (!shape_ok(rows) || !shape_ok(cols)) return FP4_ERR_SHAPE;
  if (!aligned(x, 16) || !aligned(codes, 16) || !aligned(scales, 16) || !aligned(tensor_scale, 4)) return FP4_ERR_ALIGNMENT;
  const DeviceInfo* d;
  fp4_status rc = check_common(&d);
  if (rc != FP4_OK) return rc;
  const int sms = stream_sms(d, stream);
  if (!quantize_fits_smem(rows * cols, sms)) return FP4_ERR_SHAPE;
  QuantOpts q;
  memset(&q, 0, sizeof(q));
  q.widen = 1.0f;
  CUtensorMap tm;
  if (!make_blocks_map(d, &tm, x, rows * cols / 16)) return FP4_ERR_CUDA;
  return launch_quantize(&tm, x, rows, cols, codes, scales, tensor_scale, q, sms, stream, (uint64_t)limit_us * 1000ull) ==
                 cudaSuccess
             ? FP4_OK
             : FP4_ERR_CUDA;
}

fp4_status fp4_momentum_update(const float* G, int64_t rows, int64_t cols, uint8_t* codes, uint16_t* scales,
                               float* M_out, uint32_t* hist, const fp4_momentum_params* params,
                               cudaStream_t stream) {
  if (!G || !codes || !scales || !params) return FP4_ERR_INVALID_ARG;
  if (params->flags & ~FP4_MOM_FLAG_SR) return FP4_ERR_INVALID_ARG;
  if (rows <= 0 || cols <= 0 || (cols & 15)) return FP4_ERR_SHAPE;
  if (!aligned(G, 32) || !aligned(codes, 16) || !aligned(scales, 16) || (M_out && !aligned(M_out, 32)) ||
      (hist && !aligned(hist, 4)))
    return FP4_ERR_ALIGNMENT;
  const DeviceInfo* d;
  fp4_status rc = check_common(&d);
  if (rc != FP4_OK) return rc;
  ProfScope ps(FP4_PROF_MOMENTUM, stream);
  return launch_momentum_update(G, rows, cols, params->mu, params->g_scale, (params->flags & FP4_MOM_FLAG_SR) != 0,
                                params->seed, codes, scales, M_out, hist, d->sms, stream) == cudaSuccess
             ? FP4_OK
             : FP4_ERR_CUDA;
}

fp4_status fp4_adamw_update(uint16_t* W, const uint16_t* G, int64_t n, uint8_t* m_codes, uint16_t* m_scales,
                            uint8_t* v_codes, uint16_t* v_scales, uint16_t* v_means,
                            const fp4_adamw_params* params, cudaStream_t stream) {
  if (!W || !G || !m_codes || !m_scales || !v_codes || !v_scales || !v_means || !params) return FP4_ERR_INVALID_ARG;
  if ((params->flags & ~FP4_MOM_FLAG_SR) || params->step < 1) return FP4_ERR_INVALID_ARG;
  if (n <= 0 || (n & 255)) return FP4_ERR_SHAPE;
  if (!aligned(W, 32) || !aligned(G, 32) || !aligned(m_codes, 16) || !aligned(m_scales, 16) ||
      !aligned(v_codes, 16) || !aligned(v_scales, 16) || !aligned(v_means, 16))
    return FP4_ERR_ALIGNMENT;
  const DeviceInfo* d;
  fp4_status rc = check_common(&d);
  if (rc != FP4_OK) return rc;
  ProfScope ps(FP4_PROF_ADAMW, stream);
  const AdamwConsts k = adamw_consts(params->lr, params->beta1, params->beta2, params->eps, params->weight_decay,
                                     params->step, params->seed);
  return launch_adamw_update(W, G, n, k, (params->flags & FP4_MOM_FLAG_SR) != 0, m_codes, m_scales, v_codes, v_scales,
                             v_means, stream) == cudaSuccess
             ? FP4_OK
             : FP4_ERR_CUDA;
}

fp4_status fp4_momentum_decode(const uint8_t* codes, const uint16_t* scales, int64_t rows, int64_t cols,
                               float* M_out, cudaStream_t stream) {
  if (!codes || !scales || !M_out) return FP4_ERR_INVALID_ARG;
  if (rows <= 0 || cols <= 0 || (cols & 15)) return FP4_ERR_SHAPE;
  if (!aligned(codes, 16) || !aligned(scales, 16) || !aligned(M_out, 32)) return FP4_ERR_ALIGNMENT;
  const DeviceInfo* d;
  fp4_status rc = check_common(&d);
  if (rc != FP4_OK) return rc;
  return launch_momentum_decode(codes, scales, rows, cols, M_out, d->sms, stream) == cudaSuccess ? FP4_OK
                                                                                                 : FP4_ERR_CUDA;
}

fp4_status fp4_root_coeffs(int64_t m, int64_t n, int steps, float abc[3]) {
  if (m <= 0 || n <= 0 || steps < 0 || !abc) return FP4_ERR_INVALID_ARG;
  coeffs(m, n, abc);
  return FP4_OK;
}

fp4_status fp4_root_ns_workspace_layout(int64_t m, int64_t n, int steps, uint32_t flags, fp4_ws_layout* layout) {
  if (!layout || (flags & ~kNsFlags)) return FP4_ERR_INVALID_ARG;
  fp4_ns_params p;
  default_params(&p);
  p.flags = flags;
  NsPlan pl;
  fp4_status rc = make_plan(m, n, steps, &p, 1, &pl);
  if (rc != FP4_OK) return rc;
  *layout = pl.lay;
  return FP4_OK;
}

size_t fp4_root_ns_workspace_bytes(int64_t m, int64_t n, int steps, uint32_t flags) {
  fp4_ws_layout L;
  if (fp4_root_ns_workspace_layout(m, n, steps, flags, &L) != FP4_OK) return 0;
  return L.total;
}

fp4_status fp4_root_ns(const float* G, float* out, int64_t m, int64_t n, int steps, const fp4_ns_params* p,
                       void* ws, size_t ws_bytes, cudaStream_t stream) {
  fp4_ns_params dp;
  if (!p) { default_params(&dp); p = &dp; }
  if (!G || !out || !ws || (p->flags & ~kNsFlags)) return FP4_ERR_INVALID_ARG;
  if (!ns_shape_ok(m) || !ns_shape_ok(n)) return FP4_ERR_SHAPE;
  if (steps < 0 || steps > kMaxSteps) return FP4_ERR_INVALID_ARG;
  if (!aligned(G, 16) || !aligned(out, 16) || !aligned(ws, 256)) return FP4_ERR_ALIGNMENT;
  const size_t need = fp4_root_ns_workspace_bytes(m, n, steps, p->flags);
  if (need == 0 || ws_bytes < need) return FP4_ERR_WORKSPACE;
  const DeviceInfo* d;
  fp4_status rc = check_common(&d);
  if (rc != FP4_OK) return rc;
  return run_one(d, G, out, m, n, steps, p, static_cast<uint8_t*>(ws), true, stream);
}

// The second stream of a batched call with FP4_FLAG_OVERLAP_GROUPS, one per host thread and device,
// created on first use.
struct SideStream {
  int dev = -1;
  cudaStream_t stream = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
};
SideStream* side_stream(int dev) {
  thread_local SideStream t;
  if (t.stream && t.dev == dev) return &t;
  if (t.stream) {   // the thread moved to another device
    cudaEventDestroy(t.fork); cudaEventDestroy(t.join); cudaStreamDestroy(t.stream);
    t = SideStream();
  }
  if (cudaStreamCreateWithFlags(&t.stream, cudaStreamNonBlocking) != cudaSuccess) { t = SideStream(); return nullptr; }
  if (cudaEventCreateWithFlags(&t.fork, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&t.join, cudaEventDisableTiming) != cudaSuccess) {
    cudaStreamDestroy(t.stream);
    t = SideStream();
    return nullptr;
  }
  t.dev = dev;
  return &t;
}

// Batched workspace: one workspace per matrix (the stages of equal-shape matrices run in
// lockstep, so none can be shared).
size_t fp4_root_ns_batched_workspace_bytes(int count, const int64_t* m, const int64_t* n, int steps,
                                           uint32_t flags) {
  if (count <= 0 || !m || !n) return 0;
  size_t need = 0;
  for (int i = 0; i < count; ++i) {
    size_t b = fp4_root_ns_workspace_bytes(m[i], n[i], steps, flags);
    if (b == 0) return 0;
    need += align_up(b, 1024);
  }
  return need;
}

fp4_status fp4_root_ns_batched(int count, const float* const* G, float* const* out, const int64_t* m,
                               const int64_t* n, int steps, const fp4_ns_params* p, void* ws, size_t ws_bytes,
                               cudaStream_t stream) {
  fp4_ns_params dp;
  if (!p) { default_params(&dp); p = &dp; }
  if (count < 0 || (count > 0 && (!G || !out || !m || !n)) || !ws || (p->flags & ~kNsFlags)) return FP4_ERR_INVALID_ARG;
  if (steps < 0 || steps > kMaxSteps) return FP4_ERR_INVALID_ARG;
  if (!aligned(ws, 256)) return FP4_ERR_ALIGNMENT;
  for (int i = 0; i < count; ++i) {
    if (!G[i] || !out[i]) return FP4_ERR_INVALID_ARG;
    if (!ns_shape_ok(m[i]) || !ns_shape_ok(n[i])) return FP4_ERR_SHAPE;
    if (!aligned(G[i], 16) || !aligned(out[i], 16)) return FP4_ERR_ALIGNMENT;
  }
  if (count == 0) return FP4_OK;
  const size_t need = fp4_root_ns_batched_workspace_bytes(count, m, n, steps, p->flags);
  if (need == 0 || ws_bytes < need) return FP4_ERR_WORKSPACE;
  const DeviceInfo* d;
  fp4_status rc = check_common(&d);
  if (rc != FP4_OK) return rc;

  uint8_t* base = static_cast<uint8_t*>(ws);
  std::vector<MatrixCtx> ctx((size_t)count);
  size_t off = 0;
  for (int i = 0; i < count; ++i) {
    rc = prepare_matrix(d, G[i], out[i], m[i], n[i], steps, p, base + off, &ctx[(size_t)i]);
    if (rc != FP4_OK) return rc;
    if (p->top_hist) ctx[(size_t)i].hist_top = p->top_hist[i];
    if (p->weights) ctx[(size_t)i].W = p->weights[i];
    off += align_up(ctx[(size_t)i].pl.lay.total, 1024);
  }
  uint32_t* status = reinterpret_cast<uint32_t*>(base);  // header of the first matrix

  const int cap = p->max_group > 0 && (int)p->max_group < kPackMax ? (int)p->max_group : kDefaultMaxGroup;
  std::vector<std::vector<MatrixCtx>> groups = group_by_shape(ctx, cap);
  // Groups do not depend on one another.  On request (FP4_FLAG_OVERLAP_GROUPS) they alternate between the
  // caller's stream and a second one that forks from it and joins it again before the call returns: every
  // launch is a persistent grid that ends in a partial wave of tiles, and the next launch of the same
  // group cannot start before it has drained - a launch of another group can.  (Not while stage times
  // are being collected: the event pairs of the two streams would overlap.)
  SideStream* side = (p->flags & FP4_FLAG_OVERLAP_GROUPS) && groups.size() >= 2 && g_prof_on.load() == 0
                         ? side_stream((int)(d - g_dev)) : nullptr;
  if (!side) merge_groups(groups, cap, steps, p, d->sms, stream_sms(d, stream));
  if (side) {
    // the status word is cleared once, before the fork (a group's own clearing kernel could wipe what
    // a kernel of the other group has just reported)
    if (cudaMemsetAsync(status, 0, 4, stream) != cudaSuccess || cudaEventRecord(side->fork, stream) != cudaSuccess ||
        cudaStreamWaitEvent(side->stream, side->fork, 0) != cudaSuccess)
      return FP4_ERR_CUDA;
  }
  for (size_t gi = 0; gi < groups.size(); ++gi) {
    cudaStream_t st = (side && (gi & 1)) ? side->stream : stream;
    rc = run_group(d, groups[gi].data(), (int)groups[gi].size(), steps, p, status, !side, side != nullptr, st);
    if (rc != FP4_OK) break;
  }
  if (side) {
    if (cudaEventRecord(side->join, side->stream) != cudaSuccess || cudaStreamWaitEvent(stream, side->join, 0) != cudaSuccess)
      return FP4_ERR_CUDA;
  }
  return rc;
}

fp4_status fp4_last_device_status(const void* ws, cudaStream_t stream) {
  if (!ws) return FP4_ERR_INVALID_ARG;
  uint32_t word = 0;
  if (cudaMemcpyAsync(&word, ws, 4, cudaMemcpyDeviceToHost, stream) != cudaSuccess) return FP4_ERR_CUDA;
  if (cudaStreamSynchronize(stream) != cudaSuccess) return FP4_ERR_CUDA;
  return word == 0 ? FP4_OK : (fp4_status)word;
}

static fp4_status gemm_nt_impl(int dry, const uint8_t* a_codes, const uint8_t* a_scales, float a_tensor_scale,
                       const uint8_t* b_codes, const uint8_t* b_scales, float b_tensor_scale, int64_t M, int64_t N,
                       int64_t K, float* D, uint32_t* device_status, cudaStream_t stream) {
  pdl_select(false);  // a single product: plain launch
  if (!a_codes || !a_scales || !b_codes || !b_scales || !D) return FP4_ERR_INVALID_ARG;
  if (!shape_ok(M) || !shape_ok(N) || !shape_ok(K)) return FP4_ERR_SHAPE;
  if (!aligned(a_codes, 16) || !aligned(a_scales, 16) || !aligned(b_codes, 16) || !aligned(b_scales, 16) ||
      !aligned(D, 16))
    return FP4_ERR_ALIGNMENT;
  const DeviceInfo* d;
  fp4_status rc = check_common(&d);
  if (rc != FP4_OK) return rc;
  ProblemPack pack;
  memset(&pack, 0, sizeof(pack));
  GemmProblem& pr = pack.p[0];
  const int sk = gemm_pair_stage_k(kPlain);
  if (!make_codes_map(d, &pr.tmA, a_codes, M, K / 2, sk) || !make_codes_map(d, &pr.tmB, b_codes, N, K / 2, sk) ||
      !make_f32_map(d, &pr.tmOut, D, M, N) || !make_sf_map(d, &pr.tmSfa, a_scales, M, K, sk) ||
      !make_sf_map(d, &pr.tmSfb, b_scales, N, K, sk))
    return FP4_ERR_CUDA;
  pr.tmAux = pr.tmOut;
  pr.sg_a = a_tensor_scale; pr.sg_b = b_tensor_scale;
  pr.out_rows = (int)M; pr.out_cols = (int)N;
  pr.K = (int)K;
  pr.blocks_m = (int)(M / 128); pr.blocks_n = (int)(N / 128);
  GemmLaunch L;
  memset(&L, 0, sizeof(L));
  L.num_problems = 1;
  L.status = device_status;
  L.dry_operands = dry;
  if (dry && (M % 256 || N % 256 || K % 256)) return FP4_ERR_SHAPE;
  return launch_gemm_pair(kPlain, pack, L, stream_sms(d, stream), stream) == cudaSuccess ? FP4_OK : FP4_ERR_CUDA;
}

fp4_status fp4_gemm_nt(const uint8_t* a_codes, const uint8_t* a_scales, float a_tensor_scale,
                       const uint8_t* b_codes, const uint8_t* b_scales, float b_tensor_scale, int64_t M, int64_t N,
                       int64_t K, float* D, uint32_t* device_status, cudaStream_t stream) {
  return gemm_nt_impl(0, a_codes, a_scales, a_tensor_scale, b_codes, b_scales, b_tensor_scale, M, N, K, D, device_status,
                      stream);
}

fp4_status fp4_gemm_nt_resident(const uint8_t* a_codes, const uint8_t* a_scales, float a_tensor_scale,
                                const uint8_t* b_codes, const uint8_t* b_scales, float b_tensor_scale, int64_t M,
                                int64_t N, int64_t K, float* D, uint32_t* device_status, cudaStream_t stream) {
  return gemm_nt_impl(1, a_codes, a_scales, a_tensor_scale, b_codes, b_scales, b_tensor_scale, M, N, K, D, device_status,
                      stream);
}

}  // extern "C"

// ---- fp4_selftest_bounded_wait ----------------------------------------------------------------
namespace fp4 {
static __global__ void __launch_bounds__(32) k_selftest_wait(uint32_t* status, uint64_t limit_ns) {
  __shared__ uint64_t bar_seen, bar_never;
  __shared__ uint32_t abort_flag;
  if (threadIdx.x == 0) {
    fp4::mbar_init(&bar_seen, 1);
    fp4::mbar_init(&bar_never, 1);
    abort_flag = 0;
    fp4::mbar_fence_init();
  }
  __syncwarp();
  if (threadIdx.x == 1) fp4::mbar_arrive(&bar_seen);
  if (threadIdx.x == 0) {
    fp4::wait_or_abort(&bar_seen, 0, &abort_flag);                                  // lane 1 arrives: must succeed
    const bool first = *(volatile uint32_t*)&abort_flag == 0;
    fp4::wait_limited_abort(fp4::smem_u32(&bar_never), 0, &abort_flag, limit_ns);   // nobody arrives: must give up
    *status = (first && abort_flag == 1) ? (uint32_t)FP4_ERR_DEVICE_TIMEOUT : (uint32_t)FP4_ERR_INVALID_ARG;
  }
}
}  // namespace fp4

extern "C" fp4_status fp4_selftest_bounded_wait(uint32_t* device_status, uint32_t limit_us, cudaStream_t stream) {
  if (!device_status || limit_us < 1 || limit_us > 100000) return FP4_ERR_INVALID_ARG;
  const fp4::DeviceInfo* d;
  fp4_status rc = fp4::check_common(&d);
  if (rc != FP4_OK) return rc;
  fp4::count_launches(1);
  fp4::k_selftest_wait<<<1, 32, 0, stream>>>(device_status, (uint64_t)limit_us * 1000ull);
  return cudaGetLastError() == cudaSuccess ? FP4_OK : FP4_ERR_CUDA;
}

extern "C" fp4_status fp4_selftest_rounding(uint32_t* counts, cudaStream_t stream) {
  if (!counts) return FP4_ERR_INVALID_ARG;
  if (!fp4::aligned(counts, 4)) return FP4_ERR_ALIGNMENT;
  const fp4::DeviceInfo* d;
  fp4_status rc = fp4::check_common(&d);
  if (rc != FP4_OK) return rc;
  return fp4::launch_selftest_rounding(counts, d->sms, stream) == cudaSuccess ? FP4_OK : FP4_ERR_CUDA;
}

// ---- fp4_root_ns_static: the step with the workspace in a static device array ------------
// For callers that cannot allocate device memory (no cudaMalloc allowed where they run, or
// no pool to take a workspace from).  The array is part of the module image: every device
// that loads the library holds these 16 MiB until the process ends.  In host code the
// array's name stands for the symbol, it is not a device address; the address is looked up
// with cudaGetSymbolAddress, with the caller's device current, and handed to the kernels like
// any workspace.
namespace {
static __device__ __align__(256) unsigned char g_static_scratch[FP4_STATIC_SCRATCH_BYTES];

// Device address of the static array on the current device.  Looked up on every call: the lookup is a
// table read once the module is loaded, allocates nothing, and stays right if the context was torn
// down and rebuilt in between (a cached address would not).
fp4_status static_scratch_address(void** ptr) {
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || p == nullptr) return FP4_ERR_CUDA;
  *ptr = p;
  return FP4_OK;
}
}  // namespace

extern "C" {

fp4_status fp4_root_ns_static(const float* G, float* out, int64_t m, int64_t n, int steps, const fp4_ns_params* p,
                              uint32_t* device_status, cudaStream_t stream) {
  fp4_ns_params dp;
  if (!p) { default_params(&dp); p = &dp; }
  if (!G || !out || (p->flags & ~kNsFlags)) return FP4_ERR_INVALID_ARG;
  if (!ns_shape_ok(m) || !ns_shape_ok(n)) return FP4_ERR_SHAPE;
  if (steps < 0 || steps > kMaxSteps) return FP4_ERR_INVALID_ARG;
  if (!aligned(G, 16) || !aligned(out, 16) || (device_status && !aligned(device_status, 4))) return FP4_ERR_ALIGNMENT;
  const size_t need = fp4_root_ns_workspace_bytes(m, n, steps, p->flags);
  if (need == 0) return FP4_ERR_SHAPE;
  if (need > FP4_STATIC_SCRATCH_BYTES) return FP4_ERR_STATIC_LIMIT;
  const DeviceInfo* d;
  fp4_status rc = check_common(&d);
  if (rc != FP4_OK) return rc;
  void* scratch = nullptr;
  rc = static_scratch_address(&scratch);
  if (rc != FP4_OK) return rc;
  // run_one clears the header, the scalars and the histogram of the shared array itself
  rc = run_one(d, G, out, m, n, steps, p, static_cast<uint8_t*>(scratch), true, stream);
  if (rc != FP4_OK) return rc;
  if (device_status &&
      cudaMemcpyAsync(device_status, scratch, 4, cudaMemcpyDeviceToDevice, stream) != cudaSuccess)
    return FP4_ERR_CUDA;
  return FP4_OK;
}

void fp4_profile_enable(int on) { g_prof_on.store(on ? 1 : 0); }

fp4_status fp4_profile_collect(float* ms, int* groups) {
  if (!ms || !groups) return FP4_ERR_INVALID_ARG;
  for (int i = 0; i < FP4_PROF_CLASSES; ++i) { ms[i] = 0.0f; groups[i] = 0; }
  std::lock_guard<std::mutex> lock(g_prof_mu);
  fp4_status rc = FP4_OK;
  for (const ProfRec& r : g_prof) {
    float t = 0.0f;
    if (cudaEventSynchronize(r.e1) != cudaSuccess || cudaEventElapsedTime(&t, r.e0, r.e1) != cudaSuccess)
      rc = FP4_ERR_CUDA;
    if (r.cls >= 0 && r.cls < FP4_PROF_CLASSES) { ms[r.cls] += t; groups[r.cls] += 1; }
    cudaEventDestroy(r.e0);
    cudaEventDestroy(r.e1);
  }
  g_prof.clear();
  return rc;
}

uint64_t fp4_kernel_launches(void) { return g_launches.load(); }

}  // extern "C"
