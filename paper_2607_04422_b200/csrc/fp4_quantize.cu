// fp4_quantize: standalone NVFP4 block quantiser (Section 2, "NVFP4 format"), and the
// transposing copy that returns the result of a tall input.
#include "fp4_gemm_common.cuh"
#include "fp4_state.cuh"

namespace fp4 {

// ----------------------------------------------------------------------------------
// amax over a tensor: 128-bit loads (four independent ones in flight per thread), warp
// shuffle reduction, one atomicMax per block on the bit pattern (non-negative floats order
// like unsigned integers).
// ----------------------------------------------------------------------------------
__device__ __forceinline__ float amax4(float4 v) {
  return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
}

__global__ void __launch_bounds__(256) k_amax(const float4* x, int64_t n4, uint32_t* amax_bits) {
  pdl_launch_dependents();
  pdl_wait();
  float m = 0.0f;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (; i + 3 * stride < n4; i += 4 * stride) {
    const float4 a = ld_f32x4(x + i), b = ld_f32x4(x + i + stride), c = ld_f32x4(x + i + 2 * stride),
                 d = ld_f32x4(x + i + 3 * stride);
    m = fmaxf(m, fmaxf(fmaxf(amax4(a), amax4(b)), fmaxf(amax4(c), amax4(d))));
  }
  for (; i < n4; i += stride) m = fmaxf(m, amax4(ld_f32x4(x + i)));
#pragma unroll
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ float wm[8];
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) m = fmaxf(m, wm[w]);
    atomicMax(amax_bits, __float_as_uint(m));
  }
}

// 8 values by one 256-bit load where the tensor lies on a 32-byte boundary, else by two 128-bit ones
__device__ __forceinline__ void load8(const float* p, bool wide, float* v) {
  if (wide) {
    ld_f32x8(p, v);
  } else {
    const float4 s = ld_f32x4(reinterpret_cast<const float4*>(p)), t = ld_f32x4(reinterpret_cast<const float4*>(p) + 1);
    v[0] = s.x; v[1] = s.y; v[2] = s.z; v[3] = s.w;
    v[4] = t.x; v[5] = t.y; v[6] = t.z; v[7] = t.w;
  }
}
__device__ __forceinline__ void load_block16(const float* p, bool wide, float (&v)[16]) {
  load8(p, wide, v);
  load8(p + 8, wide, v + 8);
}

// ----------------------------------------------------------------------------------
// Row quantiser: one thread per block of 16 (64 contiguous bytes, a warp covers 512 consecutive elements of a row); 8-byte code
// store and 1-byte scale store per thread.  Thread blocks walk the tensor from its end, since the amax pass has just read it front to
// back.  grid: (strips of 4096 columns, 128, rows / 128), all three counted down, so that the pieces of a row stay together without a
// division.  amax_bits holds the tensor amax on entry (bit pattern).
//
// Bounds: HBM with reads and writes mixed, 6 TB/s of it.  The pass finds 36 MB of 8192 x 8192 and of 4096 x 16384 (268 MB) in the L2, the
// amax pass of a repeated call 50 (dram__bytes_read, caches as they are); strip after strip it found 31 and 21, and whole calls took
// 8192 x 8192 85.9 us (now 84.5), 4096 x 16384 93.0 (84.3), 5120 x 14464 100.4 (94.7), 11776 x 14592 218 (212).  With 256-bit
// loads (every sector looked up once), no 64-bit division for the place and none of the two IEEE divisions per block, whole calls, before /
// after: 8192 x 8192 86.6 / 84.5, 16384 x 8192 168 / 167, 4096 x 4096 23.1 / 22.8, 2048 x 4352 16.6 / 15.2, 8192 x 8192 with the
// options 106.8 / 100.5.  (One cooperative launch in which every block walks the same units in both passes is slower: 93.3 us at 8192 x
// 8192 where the two passes took 91.4, prefetched a unit ahead or not.)
// ----------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t row_of_block() { return (gridDim.z - 1 - blockIdx.z) * 128 + (127 - blockIdx.y); }
__global__ void __launch_bounds__(256) k_quantize_rows(const float* x, int64_t cols,
                                                       uint8_t* __restrict__ codes, uint8_t* __restrict__ scales,
                                                       const uint32_t* amax_bits, const bool wide) {
  pdl_launch_dependents();
  pdl_wait();
  const float sg = scale_exact(__uint_as_float(ld_u32(amax_bits)));
  const float six_sg = __fmul_rn(6.0f, sg), rcp_six_sg = __frcp_rn(six_sg);
  const uint32_t r = row_of_block(), kblocks = (uint32_t)cols >> 4;
  const uint32_t kb = (gridDim.x - 1 - blockIdx.x) * 256 + threadIdx.x;
  if (kb >= kblocks) return;
  const uint64_t b = (uint64_t)r * kblocks + kb;   // block of the tensor
  float v[16];
  load_block16(x + b * 16, wide, v);
  uint32_t lo, hi;
  const uint32_t sb = quantize_block16_fast(v, sg, six_sg, rcp_six_sg, lo, hi);
  *reinterpret_cast<uint2*>(codes + b * 8) = make_uint2(lo, hi);
  scales[sf_offset(r, kb, kblocks)] = (uint8_t)sb;
}

__global__ void k_finish_tensor_scale(float* ts, float widen) {
  pdl_wait();
  *ts = scale_exact(__fmul_rn(widen, *ts));  // amax (bit pattern of a float) -> s_g
}

// Row quantiser with the paper-faithful options (Section 3.4): one thread per block of 16
// (the transform and the two candidate encodings are local to a block), a warp covers 512
// consecutive elements of a row.  grid: as k_quantize_rows.
__global__ void __launch_bounds__(256) k_quantize_rows_opts(const float* x, int64_t cols,
                                                            uint8_t* __restrict__ codes, uint8_t* __restrict__ scales,
                                                            const uint32_t* amax_bits, const bool wide,
                                                            const QuantOpts q) {
  pdl_launch_dependents();
  pdl_wait();
  const float sg = scale_exact(__fmul_rn(q.widen, __uint_as_float(ld_u32(amax_bits))));
  const uint32_t r = row_of_block(), kblocks = (uint32_t)cols >> 4;
  const uint32_t kb = (gridDim.x - 1 - blockIdx.x) * 256 + threadIdx.x;
  if (kb >= kblocks) return;
  const uint64_t b = (uint64_t)r * kblocks + kb;   // block of the tensor
  float v[16];
  load_block16(x + b * 16, wide, v);
  uint32_t lo, hi;
  const uint32_t sb = quantize_block16_opts(v, q, sg, lo, hi);
  *reinterpret_cast<uint2*>(codes + b * 8) = make_uint2(lo, hi);
  scales[sf_offset(r, kb, kblocks)] = (uint8_t)sb;
}

// ----------------------------------------------------------------------------------
// fp4_quantize of a tensor that fits the shared memories of all SMs, in one cooperative launch: every element is read
// once - the largest magnitude, a barrier over all blocks, then the blocks of 16 from where they lie.
//
// A tensor is cut into units of 2048 elements (128 blocks of 16; rows and columns are multiples of 128, so
// units are whole).  Four groups of 128 threads per SM hold up to six units each; TMA brings a unit as 128 rows of 64
// bytes with the 64-byte swizzle, so that a thread reads its block without bank conflicts.
//
// Bounds: launch latency (three kernels and a memset before).  1152 x 2688: 16.1 -> 12.4 us, 16384 x 384: 27.3 -> 14.5,
// 512 x 512 15.8 -> 10.  (A ring that streams larger tensors through the same kernel was slower than the two
// passes below, 185 against 178 us at 16384 x 8192: a quarter of their threads hides less latency.)
//
// The blocks' maxima lie in the scale buffer (at least 1 KB), which is written only after a second barrier: all have
// read them by then.  The barriers' counter, cleared by the host, is the word of the tensor scale, which takes the place of
// the count while slower blocks may still poll it: as an unsigned number a normal FP32 value is larger than any count, so it
// releases them, too.  A tensor scale so small that its bits are not (below 512 2^-149) is stored by the last
// of the blocks to count themselves out.  (Counting out always: 13.6 us at 1152 x 2688 instead of 13.2.)
// There is no workspace to report in: a block that gave up on a wait turns the word into a NaN, which no tensor has as its scale.
// The bits it sets stay set: a count does not reach them, and the tensor scale takes the count's place as the larger number.
// (An exchange there, whose answer the block waits for: 13.4 us.)
// ----------------------------------------------------------------------------------
constexpr int kQUnit = 2048;
constexpr int kQUnitBytes = kQUnit * 4;
constexpr int kQMaxBlocks = 256;      // maxima in words 0 .. 255 of the scale buffer
constexpr uint32_t kQGaveUp = 0xFFC00000u;
constexpr int kQGroups = 4, kQHold = 6, kQThreads = kQGroups * 128;
struct QuantShared {
  uint64_t full[kQGroups][kQHold];
  float wmax[kQThreads / 32];
  uint32_t abort_flag;
};
constexpr int kQSmem = kQGroups * kQHold * kQUnitBytes + (int)sizeof(QuantShared) + 1024;

template <bool PF>
__global__ void __launch_bounds__(kQThreads, 1)
k_quantize_small(const __grid_constant__ CUtensorMap tm, int units, int64_t cols, uint8_t* __restrict__ codes, uint8_t* scales,
                 float* tensor_scale, const QuantOpts q, const uint32_t blocks, const uint64_t limit_ns) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  QuantShared* sh = reinterpret_cast<QuantShared*>(smem + kQGroups * kQHold * kQUnitBytes);
  volatile uint32_t* abort_flag = &sh->abort_flag;
  const int group = threadIdx.x >> 7, row = threadIdx.x & 127;
  // this group's units: blockIdx.x + (group + 4 i) gridDim.x - a small tensor spreads over the SMs first
  const int first = (int)blockIdx.x + group * (int)gridDim.x, step = kQGroups * (int)gridDim.x;
  const int m = units > first ? (units - first + step - 1) / step : 0;   // at most kQHold
  if (threadIdx.x == 0) {
    for (int i = 0; i < kQGroups * kQHold; ++i) mbar_init(&sh->full[0][0] + i, 1);
    sh->abort_flag = 0;
    mbar_fence_init();
  }
  __syncthreads();
  if (row == 0)
    for (int i = 0; i < m; ++i) {
      mbar_expect_tx(&sh->full[group][i], kQUnitBytes);
      tma_load_2d(smem + (group * kQHold + i) * kQUnitBytes, &tm, 0, (first + i * step) * 128, &sh->full[group][i]);
    }
  const uint32_t sw = (uint32_t)(row >> 1 & 3) << 4;
  auto read = [&](int i, float (&v)[16]) {
    const uint32_t at = smem_u32(smem + (group * kQHold + i) * kQUnitBytes) + row * 64;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(v[4 * j]), "=f"(v[4 * j + 1]), "=f"(v[4 * j + 2]), "=f"(v[4 * j + 3])
                   : "r"(at + ((uint32_t)(j << 4) ^ sw))
                   : "memory");
  };
  float mx = 0.0f;
  for (int i = 0; i < m; ++i) {
    float v[16];
    wait_or_abort(&sh->full[group][i], 0, abort_flag);
    read(i, v);
    mx = fmaxf(mx, amax16(v));
  }
  mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
  if ((threadIdx.x & 31) == 0) sh->wmax[threadIdx.x >> 5] = mx;
  __syncthreads();
  uint32_t* scratch = reinterpret_cast<uint32_t*>(scales);
  if (threadIdx.x == 0) {
    for (int w = 0; w < kQThreads / 32; ++w) mx = fmaxf(mx, sh->wmax[w]);
    scratch[blockIdx.x] = __float_as_uint(mx);
  }
  uint32_t* counter = reinterpret_cast<uint32_t*>(tensor_scale);
  grid_barrier(counter, blocks, abort_flag, limit_ns);
  uint32_t bits = 0;
  for (int i = threadIdx.x & 31; i < (int)gridDim.x; i += 32) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(scratch + i) : "memory");
    bits = max(bits, v);
  }
  bits = __reduce_max_sync(0xffffffffu, bits);
  const float sg = scale_exact(__fmul_rn(q.widen, __uint_as_float(bits)));
  const float six_sg = __fmul_rn(6.0f, sg), rcp_six_sg = __frcp_rn(six_sg);
  grid_barrier(counter, 2 * blocks, abort_flag, limit_ns);   // everyone has read the maxima: scales may be written
  const uint32_t kblocks = (uint32_t)(cols >> 4);
  for (int i = 0; i < m; ++i) {
    float v[16];
    read(i, v);
    const uint32_t b = (uint32_t)(first + i * step) * 128 + row;   // block of the tensor
    uint32_t lo, hi, sb;
    if (PF) sb = quantize_block16_opts(v, q, sg, lo, hi);
    else sb = quantize_block16_fast(v, sg, six_sg, rcp_six_sg, lo, hi);
    *reinterpret_cast<uint2*>(codes + (int64_t)b * 8) = make_uint2(lo, hi);
    const uint32_t r = b / kblocks;
    scales[sf_offset(r, b - r * kblocks, kblocks)] = (uint8_t)sb;
  }
  if (threadIdx.x == 0) {
    const uint32_t sg_bits = __float_as_uint(sg);
    if (sh->abort_flag) atomicOr(counter, kQGaveUp);
    else if (sg_bits >= 2 * blocks) { if (blockIdx.x == 0) atomicMax(counter, sg_bits); }
    else if (atomicAdd(counter, 1u) == 3 * blocks - 1) atomicCAS(counter, 3 * blocks, sg_bits);
  }
}

// out (l0 x s0) = the leading s0 x l0 part of X^T, X being s x l (row pitch l): 64 x 64 tiles through
// shared memory, 128-bit loads along the rows of X and 128-bit stores along the rows of out
// (s0 and l0 are multiples of 16, so a 16-byte piece is all inside or all outside).
__global__ void __launch_bounds__(256) k_transpose_out(const float* X, int64_t l, float* __restrict__ out,
                                                       int64_t s0, int64_t l0, const ParamUpdate upd) {
  __shared__ float t[64][65];
  pdl_launch_dependents();
  pdl_wait();
  const int64_t r0 = (int64_t)blockIdx.y * 64, c0 = (int64_t)blockIdx.x * 64;  // tile origin in X
  const int q = threadIdx.x & 15, row = threadIdx.x >> 4;                      // 16 pieces per row, 16 rows per sweep
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int r = row + 16 * j;
    const float4 v = ld_f32x4(reinterpret_cast<const float4*>(X + (r0 + r) * l + c0) + q);  // inside the padded work matrix
    t[r][4 * q] = v.x; t[r][4 * q + 1] = v.y; t[r][4 * q + 2] = v.z; t[r][4 * q + 3] = v.w;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = row + 16 * j;  // column of X = row of out
    if (c0 + c < l0 && r0 + 4 * q < s0) {
      const int64_t at = (c0 + c) * s0 + r0 + 4 * q;
      const float4 o = make_float4(t[4 * q][c], t[4 * q + 1][c], t[4 * q + 2][c], t[4 * q + 3][c]);
      if (!(upd.W && upd.no_out)) *reinterpret_cast<float4*>(out + at) = o;
      if (upd.W) {
        // Root's parameter update from the values on their way out (the parameter has the caller's
        // orientation, like `out`)
        uint2* wp = reinterpret_cast<uint2*>(upd.W + at);
        const uint2 w = *wp;
        *wp = make_uint2(cvt_bf16x2(param_update_value(bf16_lo(w.x), o.x, upd.decay, upd.step),
                                    param_update_value(bf16_hi(w.x), o.y, upd.decay, upd.step)),
                         cvt_bf16x2(param_update_value(bf16_lo(w.y), o.z, upd.decay, upd.step),
                                    param_update_value(bf16_hi(w.y), o.w, upd.decay, upd.step)));
      }
    }
  }
}

// W <- update(W, O) elementwise, 8 elements per thread
__global__ void __launch_bounds__(256) k_param_update(const float* O, int64_t n8, const ParamUpdate upd) {
  pdl_launch_dependents();
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n8; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 a = ld_f32x4(reinterpret_cast<const float4*>(O) + 2 * i), b = ld_f32x4(reinterpret_cast<const float4*>(O) + 2 * i + 1);
    uint4* wp = reinterpret_cast<uint4*>(upd.W) + i;
    const uint4 w = *wp;
    *wp = make_uint4(cvt_bf16x2(param_update_value(bf16_lo(w.x), a.x, upd.decay, upd.step),
                                param_update_value(bf16_hi(w.x), a.y, upd.decay, upd.step)),
                     cvt_bf16x2(param_update_value(bf16_lo(w.y), a.z, upd.decay, upd.step),
                                param_update_value(bf16_hi(w.y), a.w, upd.decay, upd.step)),
                     cvt_bf16x2(param_update_value(bf16_lo(w.z), b.x, upd.decay, upd.step),
                                param_update_value(bf16_hi(w.z), b.y, upd.decay, upd.step)),
                     cvt_bf16x2(param_update_value(bf16_lo(w.w), b.z, upd.decay, upd.step),
                                param_update_value(bf16_hi(w.w), b.w, upd.decay, upd.step)));
  }
}

// ----------------------------------------------------------------------------------
// host launchers
// ----------------------------------------------------------------------------------
static int grid_for(int64_t n4, int threads, int sms) {
  int64_t blocks = (n4 + threads - 1) / threads;
  int64_t cap = (int64_t)sms * 8;
  return (int)(blocks < cap ? (blocks < 1 ? 1 : blocks) : cap);
}

cudaError_t quantize_set_attributes() {
  cudaError_t e = cudaFuncSetAttribute(k_quantize_small<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kQSmem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_quantize_small<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kQSmem);
}

// tm: x as rows of 16 floats, box = 128 rows, 64-byte swizzle (tensors small enough for one launch).  give_up_ns: not 0 in the
// self-test, whose barriers expect a block that is not launched.
cudaError_t launch_quantize(const CUtensorMap* tm, const float* x, int64_t rows, int64_t cols, uint8_t* codes, uint8_t* scales,
                            float* tensor_scale, const QuantOpts& q, int sms, cudaStream_t st, uint64_t give_up_ns) {
  const bool pf = q.rht || q.four_six;
  if (tm) {
    const int units = (int)(rows * cols / kQUnit);
    cudaError_t e = cudaMemsetAsync(tensor_scale, 0, 4, st);
    if (e != cudaSuccess) return e;
    int grid = sms < kQMaxBlocks ? sms : kQMaxBlocks;
    if (units < grid) grid = units;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kQThreads); cfg.dynamicSmemBytes = kQSmem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    count_launches(1);
    return cudaLaunchKernelEx(&cfg, pf ? k_quantize_small<true> : k_quantize_small<false>, *tm, units, cols, codes, scales,
                              tensor_scale, q, (uint32_t)grid + (give_up_ns ? 1u : 0u), give_up_ns ? give_up_ns : kWaitLimitNs);
  }
  const int64_t n4 = rows * cols / 4;
  const bool wide = (reinterpret_cast<uintptr_t>(x) & 31) == 0;
  cudaError_t e = cudaMemsetAsync(tensor_scale, 0, 4, st);
  if (e != cudaSuccess) return e;
  // chained: a kernel's blocks become resident while the one before drains (8192 x 8192: 96 -> 92.5 us)
  pdl_select(true);
  uint32_t* amax = reinterpret_cast<uint32_t*>(tensor_scale);
  launch_chained(k_amax, dim3(grid_for(n4, 256 * 8, sms)), dim3(256), 0, st, reinterpret_cast<const float4*>(x), n4, amax);
  const dim3 qgrid((unsigned)((cols / 16 + 255) / 256), 128, (unsigned)(rows / 128));   // rows: a multiple of 128, at most 2^20
  if (pf) launch_chained(k_quantize_rows_opts, qgrid, dim3(256), 0, st, x, cols, codes, scales, amax, wide, q);
  else launch_chained(k_quantize_rows, qgrid, dim3(256), 0, st, x, cols, codes, scales, amax, wide);
  launch_chained(k_finish_tensor_scale, dim3(1), dim3(1), 0, st, tensor_scale, q.widen);
  count_launches(3);
  return cudaGetLastError();
}

// Whether a tensor of `elements` fits the shared memories of all SMs (one launch that reads it once).
bool quantize_fits_smem(int64_t elements, int sms) {
  const int grid = sms < kQMaxBlocks ? sms : kQMaxBlocks;
  return elements / kQUnit <= (int64_t)grid * kQGroups * kQHold;
}

cudaError_t launch_transpose_out(const float* X, int64_t s, int64_t l, float* out, int64_t s0, int64_t l0,
                                 const ParamUpdate& upd, cudaStream_t st) {
  dim3 grid((unsigned)((l0 + 63) / 64), (unsigned)((s0 + 63) / 64));
  (void)s;
  count_launches(1);
  launch_chained(k_transpose_out, grid, dim3(256), 0, st, X, l, out, s0, l0, upd);
  return cudaGetLastError();
}

// n is a multiple of 256 (both dimensions are multiples of 16)
cudaError_t launch_param_update(const float* O, int64_t n, const ParamUpdate& upd, int sms, cudaStream_t st) {
  if (!upd.W) return cudaSuccess;
  count_launches(1);
  launch_chained(k_param_update, dim3(grid_for(n / 8, 256, sms)), dim3(256), 0, st, O, n / 8, upd);
  return cudaGetLastError();
}

}  // namespace fp4
