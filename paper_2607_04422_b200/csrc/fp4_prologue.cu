// Prologue of the Root step for a group of matrices (Section 3.4: "p99 outlier
// clipping"; normalisation; the first operand copies qX = Q_1x16(X), qX^{16x1} = Q_16x1(X)).
// Every kernel covers the whole group (gridDim.y = matrix, or a tile list over all matrices), so a
// group needs six launches instead of six per matrix; a group that fits the shared memories of all SMs
// needs one (kp_resident, at the end).
//
// Clip threshold tau = nearest-rank quantile of |g|, found exactly with two passes over the data:
//   pass 1  histogram of the top 13 magnitude bits (exponent + 5 mantissa bits);
//   pick    the bin that holds the wanted rank;
//   pass 2  elements of that bin are appended to a candidate list (they are about 1 % of a
//           continuous distribution) and counted by their next 9 bits; in the same pass the squares of all
//           elements below the bin are summed in FP64 (they are certainly not clipped);
//   finish  the candidates are gone through once more, for their last 9 bits: tau, the candidates' squares
//           exactly (they share an exponent, so their squares add as integers) and tau^2 for every clipped
//           element give nu, 1/(nu+eps), amax(X0) and the tensor scale of X0.
// If the bin holds more candidates than the list can take (many equal values, e.g. a
// constant matrix) one finishing block continues the radix select with two more passes
// over the matrix and a statistics pass (slow, rare, no extra launch).
#include <stddef.h>

#include "fp4_gemm_common.cuh"
#include "fp4_kernels.h"

namespace fp4 {

namespace {

constexpr int kMaxPack = 16;

struct PrepMatrix {
  const float* G;
  float* X;
  NsHeader* hdr;
  float* scalars;
  uint32_t* hist;      // 8192 counters
  uint32_t* hist_top;  // the caller's counters of the first radix pass (then pass 1 is skipped), or null
  double* partial;     // one FP64 partial per statistics block
  uint32_t* cand;      // candidate list (workspace that is unused until the first product)
  uint8_t* qx_codes; uint8_t* qx_sf;
  uint8_t* qt_codes; uint8_t* qt_sf;
  int tall;
  int clear_status;
  int store_x;
  int x_rows, x_cols;  // extent and row pitch of X
  int s, l;            // work shape (multiples of 128)
  int s0, l0;          // the caller's short and long side; the rest of the work shape is zero padding
  int64_t n4;          // elements of the caller's matrix / 4
  uint32_t clip_rank;
  uint32_t cand_cap;
  int tiles, first_tile;   // 128 x 128 tiles, place in the launch's tile list
  int tiled;           // the sum of squares is taken tile by tile (see kp_compact_stats)
  int hist_blocks, stat_blocks, select_blocks;   // thread blocks of the passes
};

struct PrepGroup {
  PrepMatrix mat[kMaxPack];
  int count;
  int tiles;           // of all matrices
  int clip;
  float eps;
  int write_q;
  int zero_words;      // 32-bit words of header + scalars + histogram to clear
  QuantOpts q;         // quantiser options of X0's operand copies
  NsScalarIdx ix;
  uint32_t* status;    // the call's status word
  CUtensorMap tmG[kMaxPack];  // the callers' matrices as FP32 tensors, box = 32 columns x 128 rows, 128-byte swizzle
};

__device__ __forceinline__ uint32_t mag_bits(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }

// ---- init: clear header (keeping the status word of all but the first matrix of a call),
// scalars and histogram; arm the select
__global__ void __launch_bounds__(256) kp_init(const __grid_constant__ PrepGroup g) {
  pdl_launch_dependents();
  pdl_wait();
  const PrepMatrix& m = g.mat[blockIdx.y];
  uint32_t* w = reinterpret_cast<uint32_t*>(m.hdr);
  const int first = m.clear_status ? 0 : 4;
  // the select starts with an empty prefix and the wanted rank (written instead of the zero)
  const int rank_word = (int)(offsetof(NsHeader, sel_rank) / 4);
  for (int i = first + blockIdx.x * blockDim.x + threadIdx.x; i < g.zero_words; i += gridDim.x * blockDim.x)
    w[i] = (i == rank_word) ? m.clip_rank : 0u;
}

constexpr int kTopBits = 13;                 // bits of the first radix pass
constexpr int kTopShift = 31 - kTopBits;     // 18
constexpr int kTopBins = 1 << kTopBits;      // 8192

// True in every thread of the last of `blocks` thread blocks that get here: it sees what the others wrote before.
__device__ __forceinline__ bool last_block(uint32_t* ticket, uint32_t blocks) {
  __shared__ uint32_t s_ticket;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_ticket = atomicAdd(ticket, 1u);
    __threadfence();
  }
  __syncthreads();
  return s_ticket == blocks - 1;
}

// The bin of the 8192 counters that holds rank hdr->sel_rank: becomes the prefix; the rank is reduced to one within
// the bin and the counters are cleared.  For 512 threads.
__device__ __forceinline__ void pick_top_bin(NsHeader* hdr, uint32_t* hist) {
  constexpr int PER = kTopBins / 512;
  __shared__ uint32_t wtot[16];
  uint32_t local[PER];
  uint32_t sum = 0;
  if ((reinterpret_cast<uintptr_t>(hist) & 15) == 0) {
#pragma unroll
    for (int j = 0; j < PER; j += 4) {
      const uint4 v = ld_cg(reinterpret_cast<const uint4*>(hist + threadIdx.x * PER + j));
      local[j] = v.x; local[j + 1] = v.y; local[j + 2] = v.z; local[j + 3] = v.w;
    }
  } else {   // a caller's histogram need only be 4-byte aligned
#pragma unroll
    for (int j = 0; j < PER; ++j) local[j] = ld_cg(hist + threadIdx.x * PER + j);
  }
#pragma unroll
  for (int j = 0; j < PER; ++j) sum += local[j];
  // exclusive prefix of the chunk sums: scan inside each warp, then add the totals of the warps before
  uint32_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if ((int)(threadIdx.x & 31) >= o) incl += t;
  }
  if ((threadIdx.x & 31) == 31) wtot[threadIdx.x >> 5] = incl;
  const uint32_t rank = hdr->sel_rank;
  __syncthreads();
  uint32_t before = incl - sum;
  for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) before += wtot[w];
  if (rank > before && rank <= before + sum) {
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      if (rank > before && rank <= before + local[j]) {
        hdr->sel_prefix = (uint32_t)(threadIdx.x * PER + j) << kTopShift;
        hdr->sel_rank = rank - before;
        hdr->bin_count = local[j];
        hdr->count_below = before;
      }
      before += local[j];
    }
  }
#pragma unroll
  for (int j = 0; j < PER; ++j) hist[threadIdx.x * PER + j] = 0;
}

// (The last block of the histogram could do this, too: then every block waits for its counts to arrive before it takes its
// ticket, and the histogram of sixteen 3072 x 3072 took 144 us instead of 116 + 10.)
__global__ void __launch_bounds__(512) kp_pick_top(const __grid_constant__ PrepGroup g) {
  pdl_launch_dependents();
  pdl_wait();
  const PrepMatrix& m = g.mat[blockIdx.y];
  pick_top_bin(m.hdr, m.hist_top ? m.hist_top : m.hist);
}

// ---- pass 1: histogram of the top 13 magnitude bits
__global__ void __launch_bounds__(512) kp_hist_top(const __grid_constant__ PrepGroup g) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ uint32_t sh[kTopBins];
  const PrepMatrix& m = g.mat[blockIdx.y];
  if (m.hist_top || (int)blockIdx.x >= m.hist_blocks) return;  // the caller counted this matrix already; a smaller matrix
  for (int i = threadIdx.x; i < kTopBins; i += blockDim.x) sh[i] = 0;
  __syncthreads();
  const float4* src = reinterpret_cast<const float4*>(m.G);
  const int64_t stride = (int64_t)m.hist_blocks * blockDim.x;
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (; i + stride < m.n4; i += 2 * stride) {
    const float4 v = ld_f32x4(src + i), w = ld_f32x4(src + i + stride);
    atomicAdd(&sh[mag_bits(v.x) >> kTopShift], 1u);
    atomicAdd(&sh[mag_bits(v.y) >> kTopShift], 1u);
    atomicAdd(&sh[mag_bits(v.z) >> kTopShift], 1u);
    atomicAdd(&sh[mag_bits(v.w) >> kTopShift], 1u);
    atomicAdd(&sh[mag_bits(w.x) >> kTopShift], 1u);
    atomicAdd(&sh[mag_bits(w.y) >> kTopShift], 1u);
    atomicAdd(&sh[mag_bits(w.z) >> kTopShift], 1u);
    atomicAdd(&sh[mag_bits(w.w) >> kTopShift], 1u);
  }
  for (; i < m.n4; i += stride) {
    const float4 v = ld_f32x4(src + i);
    atomicAdd(&sh[mag_bits(v.x) >> kTopShift], 1u);
    atomicAdd(&sh[mag_bits(v.y) >> kTopShift], 1u);
    atomicAdd(&sh[mag_bits(v.z) >> kTopShift], 1u);
    atomicAdd(&sh[mag_bits(v.w) >> kTopShift], 1u);
  }
  __syncthreads();
  for (int j = threadIdx.x; j < kTopBins; j += blockDim.x)
    if (sh[j]) atomicAdd(&m.hist[j], sh[j]);
}

// Sum of a warp's values, the same in every lane: pairs 16 lanes apart first.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

constexpr int kSubBins = 512;                 // counters of bits 17..9 and of bits 8..0 of the candidates

// ---- pass 2: candidates of the picked bin, FP64 sum of squares below the bin, max |g|.
// Candidates are rare: they are collected in a shared-memory buffer per block and copied to
// the global list with one reservation per block (or directly when the buffer is full); on the way there the next 9
// bits of each are counted, in the counters the first pass has left cleared.
//
// The sum of squares must not depend on how many matrices a call has, so it is the same sum in kp_resident: a matrix small
// enough to be resident is summed tile by tile (a lane 4 columns of 4 rows, a warp its lanes, then the 32 row sums), larger
// ones as their elements lie in memory.
//
// Eight blocks per SM: the 1024 blocks of a matrix are resident at once.  (With 40 registers and six blocks an eighth of them
// ran as a second wave: 16384 x 16384 248 us against 178, 6.0 TB/s; 4096 x 8192 36 against 27.5.)
template <bool TILED>
__global__ void __launch_bounds__(256, 8) kp_compact_stats(const __grid_constant__ PrepGroup g) {
  pdl_launch_dependents();
  pdl_wait();
  constexpr uint32_t kBuf = 2048;
  __shared__ uint32_t s_buf[kBuf];
  __shared__ uint32_t s_sub[kSubBins];
  __shared__ uint32_t s_cnt, s_base;
  const PrepMatrix& m = g.mat[blockIdx.y];
  if ((m.tiled != 0) != TILED || (int)blockIdx.x >= m.stat_blocks) return;
  const uint32_t bin = g.clip ? (m.hdr->sel_prefix >> kTopShift) : 0xFFFFFFFFu;
  const float4* src = reinterpret_cast<const float4*>(m.G);
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) s_cnt = 0;
  for (int j = threadIdx.x; j < kSubBins; j += blockDim.x) s_sub[j] = 0;
  __syncthreads();
  double acc = 0.0;
  float mx = 0.0f;
  auto visit = [&](float x) {
    const uint32_t k = mag_bits(x);
    const uint32_t kb = k >> kTopShift;
    if (kb < bin) {
      acc += (double)x * (double)x;
      mx = fmaxf(mx, __uint_as_float(k));
    } else if (kb == bin) {
      const uint32_t pos = atomicAdd(&s_cnt, 1u);
      if (pos < kBuf) {
        s_buf[pos] = k;
      } else {
        const uint32_t gpos = atomicAdd(&m.hdr->cand_count, 1u);
        if (gpos < m.cand_cap) m.cand[gpos] = k;
        atomicAdd(&s_sub[(k >> 9) & (kSubBins - 1)], 1u);   // (in global memory: 14.1 ms for an all-zero 4096 x 4096)
      }
    }
  };
  __shared__ double wa[32];
  __shared__ float wm[8];
  const int warp = threadIdx.x >> 5;
  if (TILED) {
    const int rows = (m.tall ? m.l0 : m.s0), cols = (m.tall ? m.s0 : m.l0);
    const int tiles_x = (m.tall ? m.s : m.l) >> 7, ty = (int)blockIdx.x / tiles_x;
    const int row0 = ty * 128, col = ((int)blockIdx.x - ty * tiles_x) * 128 + lane * 4;
#pragma unroll 1
    for (int r = warp; r < 32; r += 8) {
      acc = 0.0;
      if (col < cols) {
#pragma unroll 1
        for (int k = 0; k < 128; k += 64) {
          const int ra = row0 + r + k, rb = ra + 32;
          const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          const float4 v = ra < rows ? ld_f32x4(src + ((int64_t)ra * cols + col) / 4) : zero;
          const float4 w = rb < rows ? ld_f32x4(src + ((int64_t)rb * cols + col) / 4) : zero;
          if (ra < rows) { visit(v.x); visit(v.y); visit(v.z); visit(v.w); }
          if (rb < rows) { visit(w.x); visit(w.y); visit(w.z); visit(w.w); }
        }
      }
      acc = warp_sum(acc);
      if (lane == 0) wa[r] = acc;
    }
  } else {
    const int64_t stride = (int64_t)m.stat_blocks * blockDim.x;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (; i + stride < m.n4; i += 2 * stride) {
      const float4 v = ld_f32x4(src + i), w = ld_f32x4(src + i + stride);
      visit(v.x); visit(v.y); visit(v.z); visit(v.w);
      visit(w.x); visit(w.y); visit(w.z); visit(w.w);
    }
    for (; i < m.n4; i += stride) {
      const float4 v = ld_f32x4(src + i);
      visit(v.x); visit(v.y); visit(v.z); visit(v.w);
    }
    acc = warp_sum(acc);
    if (lane < 4) wa[warp + 8 * lane] = lane == 0 ? acc : 0.0;
  }
  mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
  if (lane == 0) wm[warp] = mx;
  __syncthreads();
  if (warp == 0) acc = warp_sum(wa[lane]);
  const uint32_t nbuf = s_cnt < kBuf ? s_cnt : kBuf;
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) mx = fmaxf(mx, wm[w]);
    m.partial[blockIdx.x] = acc;
    atomicMax(&m.hdr->maxabs_bits, __float_as_uint(mx));
    s_base = nbuf ? atomicAdd(&m.hdr->cand_count, nbuf) : 0u;
  }
  __syncthreads();
  for (uint32_t j = threadIdx.x; j < nbuf; j += blockDim.x) {
    const uint32_t gpos = s_base + j;
    if (gpos < m.cand_cap) m.cand[gpos] = s_buf[j];
  }
  if (nbuf <= kSubBins) {
    for (uint32_t j = threadIdx.x; j < nbuf; j += blockDim.x) atomicAdd(&m.hist[(s_buf[j] >> 9) & (kSubBins - 1)], 1u);
  } else {   // fewer global atomics by way of shared counters
    for (uint32_t j = threadIdx.x; j < nbuf; j += blockDim.x) atomicAdd(&s_sub[(s_buf[j] >> 9) & (kSubBins - 1)], 1u);
    __syncthreads();
    for (int j = threadIdx.x; j < kSubBins; j += blockDim.x)
      if (s_sub[j]) atomicAdd(&m.hist[j], s_sub[j]);
  }
}

// Fixed-order sum of at most 1024 partials by a block of 1024 threads, returned in warp 0; `wsum`: 32 words.
__device__ __forceinline__ double sum_partials(const double* partial, int nparts, double* wsum) {
  const int tid = threadIdx.x;
  const double v = warp_sum(tid < nparts ? ld_cg(partial + tid) : 0.0);
  if ((tid & 31) == 0) wsum[tid >> 5] = v;
  __syncthreads();
  return tid < 32 ? warp_sum(wsum[tid]) : 0.0;
}
// The clipped matrix's sum of squares: `below` the clip's bin, the candidates' lo + hi 2^24 in units of the square of their last
// place, and tau^2 for each of the n_clipped elements above it.
__device__ __forceinline__ double clipped_squares(double below, unsigned long long lo, unsigned long long hi, uint32_t efield,
                                                  double n_clipped, float tau) {
  const int e2 = 2 * ((int)(efield ? efield : 1u) - 150);
  const double cand = ldexp(__fma_rn((double)hi, 16777216.0, (double)lo), e2);
  return __fma_rn(__dmul_rn(n_clipped, (double)tau), (double)tau, __dadd_rn(below, cand));
}

struct NormScalars { float nu, inv, amax0, sg; };
__device__ __forceinline__ NormScalars norm_scalars(double sumsq, float maxabs, float eps, float widen) {
  NormScalars n;
  n.nu = (float)sqrt(sumsq);
  n.inv = __fdiv_rn(1.0f, __fadd_rn(n.nu, eps));
  n.amax0 = __fmul_rn(maxabs, n.inv);
  n.sg = scale_exact(__fmul_rn(widen, n.amax0));
  return n;
}
__device__ __forceinline__ void write_norm_scalars(float* scalars, const NsScalarIdx& ix, const NormScalars& n) {
  scalars[ix.nu] = n.nu;
  scalars[ix.inv] = n.inv;
  scalars[ix.amax_X0] = n.amax0;
  scalars[ix.sg_X0] = n.sg;
}

// ---- fallback when the candidate list overflowed (so many equal magnitudes that the picked bin holds more
// than the list takes: constant matrices and the like).  One block finishes the job alone: two more
// radix rounds over the whole matrix (bits 17..7, then 6..0) and the clamped sum of squares.  Slow
// (three passes by 1024 threads) but rare, and it costs no launch when it is not needed.  Bound by the latency of its loads and the
// counters: all-zero 2560 x 2560, 2 iterations, 1606 us with one load in flight per thread, 1280 with four.
// hist: 2048 counters; shd: 1024 doubles.
__device__ __forceinline__ void fallback_select_and_stats(const PrepGroup& g, const PrepMatrix& m, uint32_t* hist, double* shd) {
  __shared__ uint32_t s_fb_prefix, s_fb_rank;
  NsHeader* hdr = m.hdr;
  const float4* src = reinterpret_cast<const float4*>(m.G);
  auto each = [&](auto&& visit) {   // four loads in flight
    const int64_t step = blockDim.x;
    int64_t i = threadIdx.x;
    for (; i + 3 * step < m.n4; i += 4 * step) {
      const float4 v0 = ld_f32x4(src + i), v1 = ld_f32x4(src + i + step), v2 = ld_f32x4(src + i + 2 * step), v3 = ld_f32x4(src + i + 3 * step);
      visit(v0); visit(v1); visit(v2); visit(v3);
    }
    for (; i < m.n4; i += step) visit(ld_f32x4(src + i));
  };
  if (threadIdx.x == 0) { s_fb_prefix = hdr->sel_prefix; s_fb_rank = hdr->sel_rank; }
  __syncthreads();
  for (int round = 0; round < 2; ++round) {
    const int shift = round == 0 ? 7 : 0, nbits = round == 0 ? 11 : 7;
    const uint32_t nb = 1u << nbits;
    const uint32_t high_mask = (0x7FFFFFFFu >> (shift + nbits)) << (shift + nbits);
    for (uint32_t i = threadIdx.x; i < nb; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    const uint32_t prefix = s_fb_prefix;
    each([&](const float4& v) {
      const uint32_t k[4] = {mag_bits(v.x), mag_bits(v.y), mag_bits(v.z), mag_bits(v.w)};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if ((k[j] & high_mask) == prefix) atomicAdd(&hist[(k[j] >> shift) & (nb - 1)], 1u);
    });
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t run = 0;
      const uint32_t rank = s_fb_rank;
      for (uint32_t b = 0; b < nb; ++b) {
        if (rank <= run + hist[b]) { s_fb_prefix = prefix | (b << shift); s_fb_rank = rank - run; break; }
        run += hist[b];
      }
    }
    __syncthreads();
  }
  const float tau = __uint_as_float(s_fb_prefix);
  double acc = 0.0;
  each([&](const float4& v) {
    const float c[4] = {fminf(fabsf(v.x), tau), fminf(fabsf(v.y), tau), fminf(fabsf(v.z), tau), fminf(fabsf(v.w), tau)};
#pragma unroll
    for (int j = 0; j < 4; ++j) acc += (double)c[j] * (double)c[j];
  });
  shd[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o; o >>= 1) {
    if ((int)threadIdx.x < o) shd[threadIdx.x] += shd[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    hdr->sel_prefix = s_fb_prefix;
    m.scalars[g.ix.tau] = tau;
    write_norm_scalars(m.scalars, g.ix, norm_scalars(shd[0], tau, g.eps, g.q.widen));
  }
}

// What the select's blocks of a matrix add up (in the matrix's counters behind the 512 of bits 17..9).
struct SelectSums {
  uint32_t low[kSubBins];          // candidates of the picked sub-bin by their last 9 bits
  unsigned long long lo, hi;       // exact squares of the candidates below the sub-bin, in two parts
  uint32_t above;                  // candidates above it
};

// Exclusive prefix of one value per thread over a block of 1024 threads; `wtot`: 32 words.
__device__ __forceinline__ uint32_t block_prefix(uint32_t v, uint32_t* wtot) {
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if ((int)(threadIdx.x & 31) >= o) incl += t;
  }
  if ((threadIdx.x & 31) == 31) wtot[threadIdx.x >> 5] = incl;
  __syncthreads();
  uint32_t w = wtot[threadIdx.x & 31], s = w;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, s, o);
    if ((int)(threadIdx.x & 31) >= o) s += t;
  }
  const uint32_t before = __shfl_sync(0xffffffffu, s - w, (int)(threadIdx.x >> 5));
  __syncthreads();
  return before + incl - v;
}

// ---- finish: select tau among the candidates and derive the normalisation scalars.
// The candidates share their top 13 bits.  Every block finds the sub-bin of bits 17..9 from the counters of the second
// pass and goes through its share of the list: members of the sub-bin are counted by their last 9 bits, and the
// squares of those below it (certainly not clipped) are summed as exact integers -- all candidates share the
// exponent field, so x = mant * 2^(e-150) with a 24-bit integer mant.  The last block picks tau.
// (One block alone, counting both halves of the bits itself, took 135 us for the candidates of 16384 x 16384 and 26 us for
// those of 4096 x 8192; now 12 us each.)
__global__ void __launch_bounds__(1024) kp_finalize(const __grid_constant__ PrepGroup g) {
  pdl_launch_dependents();
  pdl_wait();
  const PrepMatrix& m = g.mat[blockIdx.y];
  if ((int)blockIdx.x >= m.select_blocks) return;
  __shared__ double shd[1024];
  __shared__ uint32_t hist[kSubBins];
  __shared__ uint32_t wtot[32];
  __shared__ uint32_t s_prefix, s_rank;
  __shared__ unsigned long long s_lo, s_hi;
  __shared__ uint32_t s_above;
  NsHeader* hdr = m.hdr;
  const int tid = threadIdx.x;
  if (!g.clip) {
    if (blockIdx.x) return;
    const double total = sum_partials(m.partial, m.stat_blocks, shd);
    if (tid == 0)
      write_norm_scalars(m.scalars, g.ix, norm_scalars(total, __uint_as_float(hdr->maxabs_bits), g.eps, g.q.widen));
    return;
  }
  const uint32_t count = hdr->cand_count;
  if (count > m.cand_cap) {
    if (blockIdx.x) return;
    if (tid == 0) hdr->overflow = 1;
    __shared__ uint32_t fb_hist[2048];
    fallback_select_and_stats(g, m, fb_hist, shd);
    return;
  }
  SelectSums* sums = reinterpret_cast<SelectSums*>(m.hist + kSubBins);
  const uint32_t top = hdr->sel_prefix, top_rank = hdr->sel_rank;
  const uint32_t efield = top >> 23;
  const uint32_t implicit = efield ? 0x800000u : 0u;
  if (tid == 0) { s_lo = 0; s_hi = 0; s_above = 0; }
  if (tid < kSubBins) hist[tid] = 0;
  {
    const uint32_t c = tid < kSubBins ? m.hist[tid] : 0u;
    const uint32_t before = block_prefix(c, wtot);
    if (c && top_rank > before && top_rank <= before + c) {
      s_prefix = top | ((uint32_t)tid << 9);
      s_rank = top_rank - before;
    }
  }
  __syncthreads();
  const uint32_t prefix = s_prefix, rank = s_rank;
  unsigned long long lo = 0, hi = 0;
  uint32_t above = 0;
  const uint32_t stride = m.select_blocks * blockDim.x;
  for (uint32_t i0 = blockIdx.x * blockDim.x + tid; i0 < count; i0 += 8 * stride) {
    uint32_t k[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) k[u] = i0 + u * (uint64_t)stride < count ? m.cand[i0 + u * stride] : 0xFFFFFFFFu;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (k[u] == 0xFFFFFFFFu) continue;
      if ((k[u] & ~511u) == prefix) {
        atomicAdd(&hist[k[u] & 511u], 1u);
      } else if (k[u] < prefix) {
        const unsigned long long mant = (k[u] & 0x7FFFFFu) | implicit;
        const unsigned long long sq = mant * mant;
        lo += sq & 0xFFFFFFull;
        hi += sq >> 24;
      } else {
        above += 1;
      }
    }
  }
  // one shared atomic per warp (64-bit shared atomics from all 1024 threads serialise badly)
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    lo += __shfl_xor_sync(0xffffffffu, lo, o);
    hi += __shfl_xor_sync(0xffffffffu, hi, o);
    above += __shfl_xor_sync(0xffffffffu, above, o);
  }
  if ((tid & 31) == 0) {
    atomicAdd(&s_lo, lo);
    atomicAdd(&s_hi, hi);
    atomicAdd(&s_above, above);
  }
  __syncthreads();
  if (m.select_blocks > 1) {
    if (tid < kSubBins && hist[tid]) atomicAdd(&sums->low[tid], hist[tid]);
    if (tid == 0) {
      atomicAdd(&sums->lo, s_lo);
      atomicAdd(&sums->hi, s_hi);
      atomicAdd(&sums->above, s_above);
    }
    if (!last_block(&hdr->ticket, m.select_blocks)) return;
    if (tid < kSubBins) hist[tid] = ld_cg(&sums->low[tid]);
    if (tid == 0) { s_lo = ld_cg(&sums->lo); s_hi = ld_cg(&sums->hi); s_above = ld_cg(&sums->above); }
    __syncthreads();
  }
  const uint32_t cnt = tid < kSubBins ? hist[tid] : 0u;
  {
    const uint32_t before = block_prefix(cnt, wtot);
    if (cnt && rank > before && rank <= before + cnt) s_prefix = prefix | (uint32_t)tid;
  }
  __syncthreads();
  const uint32_t tau_bits = s_prefix;
  // a counter stands for one exact magnitude (all 31 bits known), so its members' squares are count * mant^2
  lo = 0; hi = 0; above = 0;
  if (cnt) {
    const uint32_t kk = prefix | (uint32_t)tid;
    if (kk <= tau_bits) {
      const unsigned long long mant = (kk & 0x7FFFFFu) | implicit;
      const unsigned long long sq = mant * mant;
      lo = (unsigned long long)cnt * (sq & 0xFFFFFFull);
      hi = (unsigned long long)cnt * (sq >> 24);
    } else {
      above = cnt;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    lo += __shfl_xor_sync(0xffffffffu, lo, o);
    hi += __shfl_xor_sync(0xffffffffu, hi, o);
    above += __shfl_xor_sync(0xffffffffu, above, o);
  }
  if (tid < kSubBins && (tid & 31) == 0) {
    atomicAdd(&s_lo, lo);
    atomicAdd(&s_hi, hi);
    atomicAdd(&s_above, above);
  }
  __syncthreads();
  const double below = sum_partials(m.partial, m.stat_blocks, shd);
  if (tid == 0) {
    const float tau = __uint_as_float(tau_bits);
    // clamped to tau: everything in the bins above the picked one, and the candidates above tau
    const double n_total = (double)m.n4 * 4.0;
    const double n_clipped = n_total - (double)hdr->count_below - (double)hdr->bin_count + (double)s_above;
    const double total = clipped_squares(below, s_lo, s_hi, efield, n_clipped, tau);
    m.scalars[g.ix.tau] = tau;
    write_norm_scalars(m.scalars, g.ix, norm_scalars(total, tau, g.eps, g.q.widen));
    hdr->overflow = 0;
  }
}

// ---- X0 = clamp(G) * inv in the work orientation (s x l; transposed when G is tall), its FP32
// copy (unless the first G3 stage will form X0 from G itself), and both NVFP4 operand copies.
//
// A persistent block per SM walks 128 x 128 tiles of G.  Three tiles are kept in flight with TMA
// (64 KB each, four 32-column boxes with the 128-byte swizzle; what lies outside the caller's
// matrix arrives as zeros, which is the padding of the work shape).  Thirty-two warps quantise the
// tiles as they land: sixteen along the rows (a warp takes 8 rows, a thread one 32-column box of a
// row), sixteen along the columns (a warp takes a band of 16 rows and 64 columns, a thread two
// columns).  The tile is never transposed: for a tall G the two passes simply swap destinations
// (blocks along the rows of G are blocks along the columns of X = G^T).  The row pass writes its
// codes itself (the four lanes of a row fill 64 contiguous bytes); the column pass's codes (8 bytes
// per column) and both kinds of scale bytes are staged in shared memory and leave as 64-byte rows
// and whole 512-byte atoms.
// One block-wide barrier per tile: after it the tile's buffer is refilled and the staged bytes go out.
// Tile buffers and staging areas form rings of three.
constexpr int kPrepBufs = 3;
constexpr int kPrepTile = 128 * 128 * 4;       // bytes of a tile
constexpr int kPrepBox = 32 * 128 * 4;         // bytes of one 32-column box
constexpr int kQtSlot = 1024 + 16;             // staged column codes: [band][column][8 B], padded bands
constexpr int kPrepStage = 8 * kQtSlot + 2 * 1024;  // + two scale atoms per pass
constexpr int kPrepWarps = 32;
constexpr int kPrepThreads = kPrepWarps * 32;

struct PrepTileInfo {
  int mi, gr0, gc0, index;   // matrix, origin of the tile in G, its index in the matrix
  uint32_t row_k, col_k;     // contraction lengths of what is quantised along the rows and along the columns of G (for a wide G
                             // qX and qX^T, for a tall one qX^T and qX)
};
// Tile t of the launch; mi: a matrix at or before its own.
__device__ __forceinline__ PrepTileInfo place_tile(const PrepGroup& g, int t, int mi) {
  PrepTileInfo ti;
  ti.mi = mi;
  while (ti.mi + 1 < g.count && t >= g.mat[ti.mi + 1].first_tile) ++ti.mi;
  const PrepMatrix& m = g.mat[ti.mi];
  ti.index = t - m.first_tile;
  ti.row_k = (uint32_t)(m.tall ? m.s : m.l);
  ti.col_k = (uint32_t)(m.tall ? m.l : m.s);
  const int tiles_x = (int)(ti.row_k >> 7);  // tiles along a row of G
  const int ty = ti.index / tiles_x;
  ti.gr0 = ty * 128;
  ti.gc0 = (ti.index - ty * tiles_x) * 128;
  return ti;
}
struct PrepShared {
  uint64_t full[kPrepBufs];
  uint32_t abort_flag;
  PrepTileInfo info[4];           // tiles it .. it + 3 of this block (ring)
  float rcp_tab[kMaxPack][8];     // per matrix: fl(1 / fl((8 + j) sg))
};
constexpr int kPrepSmem = kPrepBufs * (kPrepTile + kPrepStage) + (int)sizeof(PrepShared) + 1024;
static_assert(kPrepSmem <= 232448, "at most 227 KB of dynamic shared memory");

// address of the 16-byte piece c4 (0..31) of row r in a tile of four swizzled boxes
__device__ __forceinline__ uint32_t prep_piece(uint32_t tile, int r, int c4) {
  return tile + (uint32_t)((c4 >> 3) * kPrepBox + r * 128 + (((c4 & 7) ^ (r & 7)) << 4));
}
__device__ __forceinline__ float4 lds128f(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ float lds32f(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}
// ---- block quantisers of the operand preparation.
// They quantise x0 = clamp(g, +-tau) * inv (quantize_block16 applied to x0) with fewer instructions,
// bit for bit the same result; whatever the short cuts do not cover goes to quantize_block16 itself.
//  * No clamp per element.  With y = fl(g * inv) and tinv = fl(tau * inv), rounding is monotonic, so
//    x0 = clamp(y, +-tinv) exactly and the block's amax is min(max |y|, tinv).  An element beyond the clip
//    level would be quantised from fl(tinv * rcp), which lies near 6 (the block's scale maps its amax = tinv
//    there); every larger product saturates to the same code 6.  Checked per matrix: fl(tinv * rcp) > 5
//    for the scale byte of a block whose amax is tinv.
//  * The scale byte is E4M3(fl(amax / 6sg)).  q = amax * fl(1 / 6sg) with one correction step
//    (r = amax - q * 6sg exactly by FMA, q += r * fl(1 / 6sg)) is within one ulp of the correctly rounded
//    quotient, so both convert to the same byte unless q lies within two ulps of a rounding boundary of
//    E4M3 (mantissa bits 19..0 = 0x80000 in the normal range); those blocks, and scale bytes <= 8
//    (subnormal E4M3, where the boundaries lie elsewhere), take the exact path.
//  * The reciprocal of the decoded scale d = fl(s * sg), s = (8 + m) 2^(E - 10): for sg far from the ends
//    of the exponent range d = fl((8 + m) sg) 2^(E - 10) exactly, so fl(1 / d) is one of eight values per
//    matrix with the exponent shifted; the eight values fl(1 / fl((8 + j) sg)) lie in shared memory.
struct PrepScalars {
  float tau, inv, tinv, six_sg, rcp_six_sg, sg;
  uint32_t rcp_tab;     // shared-memory address of the matrix's eight reciprocals
  uint32_t near_limit;  // 4 when the short cuts hold for this matrix (sg in [2^-60, 2^60], and the clip level
                        // itself is quantised to 6: fl(tinv * rcp) > 5 for the scale of a clipped block), else all ones
};

__device__ __noinline__ uint32_t prep_quant_exact(const float (&gv)[16], float tau, float inv, float six_sg, float sg,
                                                  uint32_t& lo, uint32_t& hi) {
  float v[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __fmul_rn(fminf(fmaxf(gv[i], -tau), tau), inv);
  return quantize_block16(v, six_sg, sg, lo, hi);
}

// amax (of |y|, not yet limited to tinv) -> scale byte and fl(1 / d); `rare` is set when the block must take
// the exact path.
__device__ __forceinline__ uint32_t prep_scale(const PrepScalars& ps, float amax_y, float& rcp, bool& rare) {
  const float amax = fminf(amax_y, ps.tinv);
  float q = __fmul_rn(amax, ps.rcp_six_sg);
  const float r = __fmaf_rn(-q, ps.six_sg, amax);
  q = __fmaf_rn(r, ps.rcp_six_sg, q);
  const uint32_t sb = cvt_ue4m3(q);
  uint32_t tab;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tab) : "r"(ps.rcp_tab + ((sb & 7u) << 2)));
  rcp = __uint_as_float(tab - (((sb >> 3) - 10u) << 23));
  const uint32_t near = (__float_as_uint(q) + 2u - 0x80000u) & 0xFFFFFu;
  // q < 1.0625 * 2^-6: scale bytes <= 8 (and the boundary to 9)
  rare = near <= ps.near_limit || q < 0.0166015625f;
  return sb;
}

// One block of 16 consecutive elements, given as four 16-byte pieces of two packed pairs each.
// `rare`: the caller must redo the block with prep_quant_exact.
__device__ __forceinline__ uint32_t prep_quant_row(uint64_t (&y2)[8], const PrepScalars& ps, uint32_t& lo,
                                                   uint32_t& hi, bool& rare) {
  const uint64_t inv2 = pack2(ps.inv, ps.inv);
  float m8[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float a, b;
    y2[i] = mul2(y2[i], inv2);
    unpack2(y2[i], a, b);
    m8[i] = fmaxf(fabsf(a), fabsf(b));
  }
  const float amax_y = fmaxf(fmaxf(fmaxf(m8[0], m8[1]), fmaxf(m8[2], m8[3])),
                             fmaxf(fmaxf(m8[4], m8[5]), fmaxf(m8[6], m8[7])));
  float rcp;
  const uint32_t sb = prep_scale(ps, amax_y, rcp, rare);
  const uint64_t rcp2 = pack2(rcp, rcp);
  float z[16];
#pragma unroll
  for (int i = 0; i < 8; ++i) unpack2(mul2(y2[i], rcp2), z[2 * i], z[2 * i + 1]);
  lo = cvt_e2m1x8(z[0], z[1], z[2], z[3], z[4], z[5], z[6], z[7]);
  hi = cvt_e2m1x8(z[8], z[9], z[10], z[11], z[12], z[13], z[14], z[15]);
  return sb;
}

// Two blocks side by side: g2[i] = the elements of row i in two neighbouring columns; block j runs down
// column j.  The pairs stay together through both multiplications.  Returns the two scale bytes.
__device__ __forceinline__ void prep_quant_col2(uint64_t (&y2)[16], const PrepScalars& ps, uint32_t (&cw)[4],
                                                uint32_t& sb0, uint32_t& sb1, bool& rare) {
  const uint64_t inv2 = pack2(ps.inv, ps.inv);
  float ax = 0.0f, ay = 0.0f;
#pragma unroll
  for (int i = 0; i < 16; i += 2) {
    float a, b, c, d;
    y2[i] = mul2(y2[i], inv2);
    y2[i + 1] = mul2(y2[i + 1], inv2);
    unpack2(y2[i], a, b);
    unpack2(y2[i + 1], c, d);
    ax = fmaxf(ax, fmaxf(fabsf(a), fabsf(c)));
    ay = fmaxf(ay, fmaxf(fabsf(b), fabsf(d)));
  }
  float r0, r1;
  bool rare0, rare1;
  sb0 = prep_scale(ps, ax, r0, rare0);
  sb1 = prep_scale(ps, ay, r1, rare1);
  const uint64_t rcp2 = pack2(r0, r1);
  float zx[16], zy[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) unpack2(mul2(y2[i], rcp2), zx[i], zy[i]);
  cw[0] = cvt_e2m1x8(zx[0], zx[1], zx[2], zx[3], zx[4], zx[5], zx[6], zx[7]);
  cw[1] = cvt_e2m1x8(zx[8], zx[9], zx[10], zx[11], zx[12], zx[13], zx[14], zx[15]);
  cw[2] = cvt_e2m1x8(zy[0], zy[1], zy[2], zy[3], zy[4], zy[5], zy[6], zy[7]);
  cw[3] = cvt_e2m1x8(zy[8], zy[9], zy[10], zy[11], zy[12], zy[13], zy[14], zy[15]);
  rare = rare0 || rare1;
}

// Lane-dependent parts of the shared-memory addresses of a thread's blocks, fixed for a whole kernel.
struct PrepLane {
  bool row_warp;
  int rr, box;         // row pass: a warp takes 8 rows, a thread one 32-column box of a row (two blocks)
  int band, cp;        // column pass: a warp takes a band of 16 rows and 64 columns, a thread two columns (pair cp)
  uint32_t base_off, sw;
};
__device__ __forceinline__ PrepLane prep_lane() {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cwp = warp & 15;
  PrepLane p;
  p.row_warp = warp < kPrepWarps / 2;
  p.rr = cwp * 8 + (lane & 7); p.box = lane >> 3;
  p.band = cwp >> 1; p.cp = (cwp & 1) * 32 + lane;
  if (p.row_warp) { p.base_off = (uint32_t)(p.box * kPrepBox + p.rr * 128); p.sw = (uint32_t)(p.rr & 7) << 4; }
  else { p.base_off = (uint32_t)((p.cp >> 4) * kPrepBox + p.band * 16 * 128 + (p.cp & 1) * 8); p.sw = (uint32_t)((p.cp >> 1) & 7) << 4; }
  return p;
}
// Scalars of a matrix; sg = its tensor scale, rcp_tab = the shared-memory address of its eight reciprocals.
__device__ __forceinline__ PrepScalars prep_scalars(float tau, float inv, float sg, uint32_t rcp_tab) {
  PrepScalars ps;
  ps.tau = tau;
  ps.inv = inv;
  ps.tinv = __fmul_rn(ps.tau, ps.inv);
  ps.sg = sg;
  ps.six_sg = __fmul_rn(6.0f, ps.sg);
  ps.rcp_six_sg = __frcp_rn(ps.six_sg);
  ps.rcp_tab = rcp_tab;
  const uint32_t esg = (__float_as_uint(ps.sg) >> 23) & 0xFFu;
  bool ok = esg >= 67u && esg <= 187u;   // 2^-60 .. 2^60
  if (ps.tinv < __int_as_float(0x7f800000)) {
    // a block with clipped elements has amax = tinv: is the clip level quantised to 6 there?
    const float dc = __fmul_rn(ue4m3_to_float(cvt_ue4m3(__fdiv_rn(ps.tinv, ps.six_sg))), ps.sg);
    ok = ok && dc != 0.0f && __fmul_rn(ps.tinv, __frcp_rn(dc)) > 5.0f;
  }
  ps.near_limit = ok ? 4u : 0xFFFFFFFFu;
  return ps;
}
// One tile: its origin in G is (gr0, gc0), its elements lie at `tile`.  Row codes (and X0 where it is wanted) are stored,
// column codes and scale bytes are staged.
template <bool PF>
__device__ __forceinline__ void prep_tile(const PrepGroup& g, const PrepMatrix& m, const PrepScalars& ps, const PrepLane& pl,
                                          uint32_t tile, uint8_t* stage, const PrepTileInfo& at) {
  const int gr0 = at.gr0, gc0 = at.gc0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool row_warp = pl.row_warp;
  const int rr = pl.rr, box = pl.box, band = pl.band, cp = pl.cp;
  const uint32_t base_off = pl.base_off, sw = pl.sw;
  auto x0 = [&](float gval) { return __fmul_rn(fminf(fmaxf(gval, -ps.tau), ps.tau), ps.inv); };
  const int tall = m.tall;

  if (m.store_x) {
    if (!tall) {
      // X = G: rows of the tile are rows of X
#pragma unroll 4
      for (int r = warp; r < 128; r += kPrepWarps) {
        const float4 v = lds128f(prep_piece(tile, r, lane));
        if ((gr0 + r) < m.x_rows && (gc0 + lane * 4) < m.x_cols)
          *reinterpret_cast<float4*>(m.X + (int64_t)(gr0 + r) * m.x_cols + gc0 + lane * 4) =
              make_float4(x0(v.x), x0(v.y), x0(v.z), x0(v.w));
      }
    } else {
      // X = G^T: a lane group of 8 consecutive tile rows writes one 32-byte sector of a row of X;
      // the 8 rows x 4 columns a warp reads at once lie in 32 different banks
      const int r8 = lane & 7, cq = lane >> 3;
#pragma unroll 4
      for (int k = 0; k < 512 / kPrepWarps; ++k) {
        const int p = warp * (512 / kPrepWarps) + k;
        const int row = (p & 15) * 8 + r8, col = (p >> 4) * 4 + cq;
        const float v = lds32f(prep_piece(tile, row, col >> 2) + (uint32_t)(col & 3) * 4u);
        if ((gc0 + col) < m.x_rows && (gr0 + row) < m.x_cols) m.X[(int64_t)(gc0 + col) * m.x_cols + gr0 + row] = x0(v);
      }
    }
  }

  if (g.write_q) {
    uint8_t* sf_stage = stage + 8 * kQtSlot;
    const uint32_t tb = tile + base_off;
    const uint64_t inv2 = pack2(ps.inv, ps.inv);
    if (row_warp) {
      uint32_t code[4];
      uint32_t sfw = 0;
      bool redo = false;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint64_t g2[8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];"
                       : "=l"(g2[2 * i]), "=l"(g2[2 * i + 1])
                       : "r"(tb + (((uint32_t)(q * 4 + i) << 4) ^ sw)));
        uint32_t sb;
        if (PF) {
          float v[16];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float a, b2;
            unpack2(mul2(g2[i], inv2), a, b2);
            v[2 * i] = fminf(fmaxf(a, -ps.tinv), ps.tinv); v[2 * i + 1] = fminf(fmaxf(b2, -ps.tinv), ps.tinv);
          }
          sb = quantize_block16_opts(v, g.q, ps.sg, code[2 * q], code[2 * q + 1]);
        } else {
          bool rare;
          sb = prep_quant_row(g2, ps, code[2 * q], code[2 * q + 1], rare);
          redo = redo || rare;
        }
        sfw |= sb << (8 * q);
      }
      if (!PF && redo) {   // rare: both blocks again from the tile, with the plain quantiser
        sfw = 0;
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
          float gv[16];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 f = lds128f(tb + (((uint32_t)(q * 4 + i) << 4) ^ sw));
            gv[4 * i] = f.x; gv[4 * i + 1] = f.y; gv[4 * i + 2] = f.z; gv[4 * i + 3] = f.w;
          }
          sfw |= prep_quant_exact(gv, ps.tau, ps.inv, ps.six_sg, ps.sg, code[2 * q], code[2 * q + 1]) << (8 * q);
        }
      }
      // the four lanes of a row write 64 contiguous bytes
      uint8_t* rp_codes = tall ? m.qt_codes : m.qx_codes;
      *reinterpret_cast<uint4*>(rp_codes + (uint64_t)(uint32_t)(gr0 + rr) * (at.row_k / 2) + gc0 / 2 + box * 16) =
          make_uint4(code[0], code[1], code[2], code[3]);
      *reinterpret_cast<uint16_t*>(sf_stage + (box >> 1) * 512 + (rr & 31) * 16 + (rr >> 5) * 4 + (box & 1) * 2) =
          (uint16_t)sfw;
    } else {
      uint64_t g2[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        // row band * 16 + i of the tile: its low three bits are those of i
        const uint32_t a = tb + (uint32_t)(i * 128) + (sw ^ ((uint32_t)(i & 7) << 4));
        asm volatile("ld.shared.b64 %0, [%1];" : "=l"(g2[i]) : "r"(a));
      }
      uint32_t cw[4], sb0 = 0, sb1 = 0;
      if (PF) {
#pragma unroll
        for (int i = 0; i < 16; ++i) g2[i] = mul2(g2[i], inv2);   // clamped to tinv below: fl(clamp(g, tau) inv)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          float v[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            float a, b2;
            unpack2(g2[i], a, b2);
            v[i] = fminf(fmaxf(j == 0 ? a : b2, -ps.tinv), ps.tinv);
          }
          const uint32_t sb = quantize_block16_opts(v, g.q, ps.sg, cw[2 * j], cw[2 * j + 1]);
          if (j == 0) sb0 = sb; else sb1 = sb;
        }
      } else {
        bool rare;
        prep_quant_col2(g2, ps, cw, sb0, sb1, rare);
        if (rare) {   // redo both blocks from the tile with the plain quantiser
#pragma unroll 1
          for (int j = 0; j < 2; ++j) {
            float gv[16];
#pragma unroll
            for (int i = 0; i < 16; ++i)
              gv[i] = lds32f(tb + (uint32_t)(i * 128 + j * 4) + (sw ^ ((uint32_t)(i & 7) << 4)));
            const uint32_t sb = prep_quant_exact(gv, ps.tau, ps.inv, ps.six_sg, ps.sg, cw[2 * j], cw[2 * j + 1]);
            if (j == 0) sb0 = sb; else sb1 = sb;
          }
        }
      }
      uint8_t* sfc = sf_stage + 1024 + (band >> 2) * 512 + (band & 3);
      const int c = cp * 2;
      sfc[(c & 31) * 16 + (c >> 5) * 4] = (uint8_t)sb0;
      sfc[((c + 1) & 31) * 16 + ((c + 1) >> 5) * 4] = (uint8_t)sb1;
      *reinterpret_cast<uint4*>(stage + band * kQtSlot + cp * 16) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
    }
  }

}
// The staged bytes of a tile go out (after a block-wide barrier).
__device__ __forceinline__ void prep_copy_out(const PrepGroup& g, const PrepMatrix& m, const uint8_t* stage, const PrepTileInfo& at) {
  const int gr0 = at.gr0, gc0 = at.gc0;
  const int tall = m.tall;
  if (g.write_q) {
    const int tid = threadIdx.x;
    if (tid < 512) {
      // column-pass codes: row (gc0 + c) of the destination, 64 bytes from byte gr0 / 2; four lanes per row
      uint8_t* cp_codes = tall ? m.qx_codes : m.qt_codes;
      const int c = tid >> 2, h = tid & 3;
      const uint8_t* src = stage + c * 8;
      const uint2 a = *reinterpret_cast<const uint2*>(src + (2 * h) * kQtSlot);
      const uint2 d = *reinterpret_cast<const uint2*>(src + (2 * h + 1) * kQtSlot);
      *reinterpret_cast<uint4*>(cp_codes + (uint64_t)(uint32_t)(gc0 + c) * (at.col_k / 2) + gr0 / 2 + h * 16) = make_uint4(a.x, a.y, d.x, d.y);
    } else if (tid < 640) {
      // scale atoms: two adjacent 512-byte atoms per pass
      const bool rowpass = tid < 576;
      uint8_t* sf_base = rowpass ? (tall ? m.qt_sf : m.qx_sf) : (tall ? m.qx_sf : m.qt_sf);
      const int64_t row0 = rowpass ? gr0 : gc0, k0 = rowpass ? gc0 : gr0, kk = rowpass ? at.row_k : at.col_k;
      const int j = tid & 63;
      const uint4 w = *reinterpret_cast<const uint4*>(stage + 8 * kQtSlot + (rowpass ? 0 : 1024) + j * 16);
      *reinterpret_cast<uint4*>(sf_base + sf_offset(row0, k0 / 16, kk / 16) + j * 16) = w;
    }
  }
}

template <bool PF>
__global__ void __launch_bounds__(kPrepThreads, 1) kp_prep_operands(const __grid_constant__ PrepGroup g) {
  extern __shared__ uint8_t prep_smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(prep_smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* stage_base = smem + kPrepBufs * kPrepTile;
  PrepShared* sh = reinterpret_cast<PrepShared*>(stage_base + kPrepBufs * kPrepStage);
  volatile uint32_t* abort_flag = &sh->abort_flag;
  const int my_tiles = (g.tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;  // tiles of this block
  pdl_launch_dependents();

  // Tile `it` of this block: work out where it lies, publish that in the ring and start its copy.  Called by
  // one thread, a block-wide barrier before the tile's turn.
  auto fetch = [&](int it_) {
    if (it_ >= my_tiles) return;
    const int t_ = (int)blockIdx.x + it_ * (int)gridDim.x;
    const int b_ = it_ % kPrepBufs;
    const PrepTileInfo ti = place_tile(g, t_, it_ > 0 ? sh->info[(it_ - 1) & 3].mi : 0);
    sh->info[it_ & 3] = ti;
    mbar_expect_tx(&sh->full[b_], kPrepTile);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      tma_load_2d(smem + b_ * kPrepTile + q * kPrepBox, &g.tmG[ti.mi], ti.gc0 + 32 * q, ti.gr0, &sh->full[b_]);
  };

  if (threadIdx.x == 0) {
    for (int i = 0; i < kPrepBufs; ++i) mbar_init(&sh->full[i], 1);
    sh->abort_flag = 0;
    mbar_fence_init();
  }
  pdl_wait();   // from here on the kernel reads what the launches before it wrote
  if (threadIdx.x == 0) {
    for (int i = 0; i < kPrepBufs; ++i) fetch(i);
  }
  if (threadIdx.x < g.count * 8) {
    const float sg_ = g.mat[threadIdx.x >> 3].scalars[g.ix.sg_X0];
    sh->rcp_tab[threadIdx.x >> 3][threadIdx.x & 7] = __frcp_rn(__fmul_rn((float)(8 + (threadIdx.x & 7)), sg_));
  }
  __syncthreads();

  const PrepLane pl = prep_lane();
  int cur = -1;
  PrepScalars ps;
  ps.tau = ps.inv = ps.tinv = ps.six_sg = ps.rcp_six_sg = ps.sg = 0.0f; ps.rcp_tab = 0; ps.near_limit = 0;
  for (int it = 0; it < my_tiles; ++it) {
    const int b = it % kPrepBufs, use = it / kPrepBufs;
    const PrepTileInfo& ti = sh->info[it & 3];   // written before an earlier barrier
    wait_or_abort(&sh->full[b], (uint32_t)use & 1u, abort_flag);
    const int mi = ti.mi;
    const PrepMatrix& m = g.mat[mi];
    if (mi != cur) {
      cur = mi;
      ps = prep_scalars(g.clip ? m.scalars[g.ix.tau] : __int_as_float(0x7f800000), m.scalars[g.ix.inv], m.scalars[g.ix.sg_X0],
                        smem_u32(&sh->rcp_tab[mi][0]));
    }
    uint8_t* stage = stage_base + b * kPrepStage;
    prep_tile<PF>(g, m, ps, pl, smem_u32(smem + b * kPrepTile), stage, ti);

    // Every warp has read the tile and staged its output: the buffer takes the tile three ahead, the
    // staged bytes go out.
    __syncthreads();
    if (threadIdx.x == kPrepThreads - 32) {
      fence_proxy_async_smem();
      fetch(it + kPrepBufs);
    }
    if (g.write_q) prep_copy_out(g, m, stage, ti);
  }
  if (threadIdx.x == 0 && sh->abort_flag) report_timeout(g.status);
}

// ---- the whole prologue of a group whose matrices fit the shared memories of all SMs, in one cooperative launch.
//
// Every block brings up to three 128 x 128 tiles into shared memory once and keeps them there: it counts them into the
// histogram, compacts candidates and squares from them, and quantises them.  Between those phases the blocks
// meet at (bounded) grid barriers; what a single block did between two launches - the bin of the rank, the select
// among the candidates, the normalisation scalars - every block now computes for its own matrices, which costs less
// than another exchange.  The same sums in the same order (see kp_compact_stats).
//
// Bounds: latency - three barriers, 3200 cycles of shared-memory counting and 4500 of FP64 sums per tile, two radix rounds,
// one tile's quantisation (18 us for one tile per SM, 42 us for three).  Whole 5-iteration calls, six launches before
// and this one now: 512 x 512 121 -> 110-120 us, 1024 x 1024 134 -> 124-128, 2048 x 2048 232 -> 223, 384 x 12160
// 272 -> 262.
constexpr int kResTiles = 3;
constexpr int kResUnion = kTopBins * 4;     // histogram / candidate buffer / select arrays / staged output of a tile
static_assert(kResUnion >= kPrepStage && kResUnion >= 4096 + 1024 * 8, "union area");
struct ResidentShared {
  uint64_t full[kResTiles];
  PrepTileInfo info[kResTiles];
  uint32_t prefix[kResTiles], rank[kResTiles], bin_count[kResTiles], below[kResTiles];   // of the tile's matrix
  float tau[kResTiles], inv[kResTiles], sg[kResTiles];
  float rcp_tab[8];
  double wsum[32];
  float wmax[32];
  uint32_t wtot[32];
  unsigned long long wlo[32], whi[32];
  uint32_t wabove[32];
  uint32_t sel_prefix, sel_rank, cnt, base;
  uint32_t abort_flag;
};
constexpr int kResSmem = kResTiles * kPrepTile + kResUnion + (int)sizeof(ResidentShared) + 1024;
static_assert(kResSmem + 64 <= 232448, "at most 227 KB of shared memory (64 bytes of it static, in the fallback)");

// CLUSTER: at most 16 tiles, one per block of a single cluster, whose hardware barrier takes the place of the counter (and of the
// memset that clears it) and lets the launch be an ordinary one, chained to the kernel before.  Whole 5-iteration calls,
// cooperative launch / cluster: 128 x 128 69.6 / 65.5 us, 256 x 512 82.9 / 77.0, 512 x 512 87.0 / 81.6, 384 x 640 with options
// 111.2 / 106.5.
constexpr int kResCluster = 16;
int g_cluster_blocks[64];   // per device: blocks of the largest such cluster it holds, or 0 (set once, before the device's first launch)
template <bool PF, bool CLUSTER>
__global__ void __launch_bounds__(kPrepThreads, 1) kp_resident(const __grid_constant__ PrepGroup g) {
  extern __shared__ uint8_t prep_smem_raw[];
  // The offset is rounded up, not the pointer: through an integer the compiler loses that this is shared memory, and the
  // counters' atomics on equal values, which the shared ones combine per warp, are done one by one (an all-zero
  // matrix 1024 x 1024, 2 iterations: 292 us instead of 1620).
  uint8_t* smem = prep_smem_raw + ((0u - smem_u32(prep_smem_raw)) & 1023u);
  uint8_t* uni = smem + kResTiles * kPrepTile;
  ResidentShared* sh = reinterpret_cast<ResidentShared*>(uni + kResUnion);
  volatile uint32_t* abort_flag = &sh->abort_flag;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int mine = (g.tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // 1 .. kResTiles (CLUSTER: 0 or 1)
  uint32_t* counter = &g.mat[0].hdr->barrier;
  uint32_t round = 0;
  auto all_blocks = [&]() {
    if (CLUSTER) {
      __syncthreads();
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
      grid_barrier(counter, ++round * gridDim.x, abort_flag);
    }
  };
  if (CLUSTER) {
    pdl_launch_dependents();
    pdl_wait();
  }
  if (tid == 0) {
    for (int i = 0; i < kResTiles; ++i) mbar_init(&sh->full[i], 1);
    sh->abort_flag = 0;
    mbar_fence_init();
    for (int it = 0; it < mine; ++it) {
      const PrepTileInfo ti = place_tile(g, (int)blockIdx.x + it * (int)gridDim.x, 0);
      sh->info[it] = ti;
      mbar_expect_tx(&sh->full[it], kPrepTile);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        tma_load_2d(smem + it * kPrepTile + q * kPrepBox, &g.tmG[ti.mi], ti.gc0 + 32 * q, ti.gr0, &sh->full[it]);
    }
  }
  // clear headers (all but the status word of all but the call's first matrix, and the barrier), scalars, histograms
  constexpr int kBarrierWord = (int)(offsetof(NsHeader, barrier) / 4);
  for (int j = 0; j < g.count; ++j) {
    uint32_t* w = reinterpret_cast<uint32_t*>(g.mat[j].hdr);
    for (int i = (g.mat[j].clear_status ? 0 : 4) + (int)blockIdx.x * kPrepThreads + tid; i < g.zero_words;
         i += (int)gridDim.x * kPrepThreads)
      if (i != kBarrierWord) w[i] = 0;
  }
  if (CLUSTER && mine == 0) {   // a cluster has a power of two of blocks: one without a tile clears its share, too
    for (int i = 0; i < (g.clip ? 3 : 2); ++i) all_blocks();
    return;
  }
  __syncthreads();
  // a thread's four 16-byte pieces of a tile: columns 4 lane .. 4 lane + 3 of rows warp, warp + 32, ...; f(value)
  auto pieces = [&](int it, auto&& f) {
    const PrepTileInfo ti = sh->info[it];
    const PrepMatrix& m = g.mat[ti.mi];
    const int rows = (m.tall ? m.l0 : m.s0) - ti.gr0, cols = (m.tall ? m.s0 : m.l0) - ti.gc0;
    const uint32_t at = smem_u32(smem + it * kPrepTile);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 v = lds128f(prep_piece(at, warp + 32 * k, lane));
      if (warp + 32 * k < rows && lane * 4 < cols) { f(v.x); f(v.y); f(v.z); f(v.w); }
    }
  };
  for (int it = 0; it < mine; ++it) wait_or_abort(&sh->full[it], 0, abort_flag);

  bool cleared = false;   // a barrier has been passed since the headers were cleared
  if (g.clip) {
    // ---- histogram of the top magnitude bits
    uint32_t* hist = reinterpret_cast<uint32_t*>(uni);
    for (int it = 0; it < mine; ++it) {
      const int mi = sh->info[it].mi;
      const bool first = it == 0 || sh->info[it - 1].mi != mi, last = it == mine - 1 || sh->info[it + 1].mi != mi;
      if (!g.mat[mi].hist_top) {
        if (first) {
          for (int i = tid; i < kTopBins; i += kPrepThreads) hist[i] = 0;
          __syncthreads();
        }
        pieces(it, [&](float x) { atomicAdd(&hist[mag_bits(x) >> kTopShift], 1u); });
        __syncthreads();
      }
      if (!cleared) { all_blocks(); cleared = true; }
      if (last && !g.mat[mi].hist_top) {
        for (int i = tid; i < kTopBins; i += kPrepThreads)
          if (hist[i]) atomicAdd(&g.mat[mi].hist[i], hist[i]);
        __syncthreads();
      }
    }
    all_blocks();
    // ---- the bin that holds the rank
    for (int it = 0; it < mine; ++it) {
      const int mi = sh->info[it].mi;
      if (it > 0 && sh->info[it - 1].mi == mi) {
        if (tid == 0) {
          sh->prefix[it] = sh->prefix[it - 1]; sh->rank[it] = sh->rank[it - 1];
          sh->bin_count[it] = sh->bin_count[it - 1]; sh->below[it] = sh->below[it - 1];
        }
        __syncthreads();
        continue;
      }
      // a warp takes 256 bins, a lane two groups of four; the warp that holds the rank looks closer
      const uint32_t* h = (g.mat[mi].hist_top ? g.mat[mi].hist_top : g.mat[mi].hist) + warp * 256 + lane * 4;
      uint32_t c[8];
      if ((reinterpret_cast<uintptr_t>(h) & 15) == 0) {
        const uint4 a = ld_cg(reinterpret_cast<const uint4*>(h)), b = ld_cg(reinterpret_cast<const uint4*>(h + 128));
        c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w; c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
      } else {   // a caller's histogram need only be 4-byte aligned
#pragma unroll
        for (int q = 0; q < 8; ++q) c[q] = ld_cg(h + (q >> 2) * 128 + (q & 3));
      }
      const uint32_t s0 = c[0] + c[1] + c[2] + c[3], s1 = c[4] + c[5] + c[6] + c[7];
      const uint32_t all = __reduce_add_sync(0xffffffffu, s0 + s1);
      if (lane == 0) sh->wtot[warp] = all;
      __syncthreads();
      const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? sh->wtot[lane] : 0u);
      if (g.mat[mi].clip_rank > before && g.mat[mi].clip_rank <= before + all) {
        uint32_t run = before;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const uint32_t v = half ? s1 : s0;
          uint32_t incl = v;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
          }
          uint32_t at = run + incl - v;
          if (g.mat[mi].clip_rank > at && g.mat[mi].clip_rank <= at + v) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint32_t n = c[half * 4 + q];
              if (g.mat[mi].clip_rank > at && g.mat[mi].clip_rank <= at + n) {
                sh->prefix[it] = (uint32_t)(warp * 256 + half * 128 + lane * 4 + q) << kTopShift;
                sh->rank[it] = g.mat[mi].clip_rank - at;
                sh->bin_count[it] = n;
                sh->below[it] = at;
              }
              at += n;
            }
          }
          run += __shfl_sync(0xffffffffu, incl, 31);
        }
      }
      __syncthreads();
    }
  } else {
    all_blocks();
  }

  // ---- squares below the bin, candidates of the bin
  for (int it = 0; it < mine; ++it) {
    const PrepTileInfo ti = sh->info[it];
    const PrepMatrix& m = g.mat[ti.mi];
    const uint32_t bin = g.clip ? sh->prefix[it] >> kTopShift : 0xFFFFFFFFu;
    uint32_t* buf = reinterpret_cast<uint32_t*>(uni);
    constexpr uint32_t kBuf = kResUnion / 4;
    if (tid == 0) sh->cnt = 0;
    __syncthreads();
    double acc = 0.0;
    float mx = 0.0f;
    pieces(it, [&](float x) {
      const uint32_t k = mag_bits(x), kb = k >> kTopShift;
      if (kb < bin) {
        acc += (double)x * (double)x;
        mx = fmaxf(mx, __uint_as_float(k));
      } else if (kb == bin) {
        const uint32_t pos = atomicAdd(&sh->cnt, 1u);
        if (pos < kBuf) {
          buf[pos] = k;
        } else {
          const uint32_t gpos = atomicAdd(&m.hdr->cand_count, 1u);
          if (gpos < m.cand_cap) m.cand[gpos] = k;
        }
      }
    });
    acc = warp_sum(acc);
    mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
    if (lane == 0) { sh->wsum[warp] = acc; sh->wmax[warp] = mx; }
    __syncthreads();
    const uint32_t nbuf = sh->cnt < kBuf ? sh->cnt : kBuf;
    if (warp == 0) {
      acc = warp_sum(sh->wsum[lane]);
      mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sh->wmax[lane])));
      if (lane == 0) {
        m.partial[ti.index] = acc;
        atomicMax(&m.hdr->maxabs_bits, __float_as_uint(mx));
        sh->base = nbuf ? atomicAdd(&m.hdr->cand_count, nbuf) : 0u;
      }
    }
    __syncthreads();
    for (uint32_t j = tid; j < nbuf; j += kPrepThreads) {
      const uint32_t gpos = sh->base + j;
      if (gpos < m.cand_cap) m.cand[gpos] = buf[j];
    }
    __syncthreads();
  }
  all_blocks();

  // ---- tau among the candidates, normalisation scalars: every block for its own matrices; the block of a matrix's
  // first tile writes them
  for (int it = 0; it < mine; ++it) {
    const int mi = sh->info[it].mi;
    const PrepMatrix& m = g.mat[mi];
    NsHeader* hdr = m.hdr;
    if (it > 0 && sh->info[it - 1].mi == mi) {
      if (tid == 0) { sh->tau[it] = sh->tau[it - 1]; sh->inv[it] = sh->inv[it - 1]; sh->sg[it] = sh->sg[it - 1]; }
      __syncthreads();
      continue;
    }
    const bool owner = sh->info[it].index == 0;
    if (owner && g.clip && m.hist_top)   // the caller's counters are consumed, whichever way tau is found: every block has read them
      for (int i = tid; i < kTopBins; i += kPrepThreads) m.hist_top[i] = 0;
    const uint32_t count = g.clip ? ld_cg(&hdr->cand_count) : 0u;
    if (count > m.cand_cap) {
      // so many equal magnitudes that the list overflowed: the owner finishes alone, the others wait for it
      if (owner) {
        if (tid == 0) { hdr->sel_prefix = sh->prefix[it]; hdr->sel_rank = sh->rank[it]; }
        __syncthreads();
        fallback_select_and_stats(g, m, reinterpret_cast<uint32_t*>(uni), reinterpret_cast<double*>(uni + 8192));
        __syncthreads();
        if (tid == 0) {
          __threadfence();
          asm volatile("st.release.gpu.global.u32 [%0], 1;" ::"l"(&hdr->overflow) : "memory");
        }
      } else if (tid == 0) {
        const uint64_t t0 = globaltimer_ns();
        for (;;) {
          uint32_t v;
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&hdr->overflow) : "memory");
          if (v) break;
          if (*abort_flag || globaltimer_ns() - t0 > kWaitLimitNs) { *abort_flag = 1; break; }
        }
      }
      __syncthreads();
      if (tid == 0) {
        sh->tau[it] = ld_cg(m.scalars + g.ix.tau);
        sh->inv[it] = ld_cg(m.scalars + g.ix.inv);
        sh->sg[it] = ld_cg(m.scalars + g.ix.sg_X0);
      }
      __syncthreads();
      continue;
    }
    uint32_t* hist = reinterpret_cast<uint32_t*>(uni);     // 512 counters
    if (tid == 0) {
      sh->sel_prefix = sh->prefix[it]; sh->sel_rank = sh->rank[it];
    }
    unsigned long long lo = 0, hi = 0;
    uint32_t above = 0, tau_bits = 0;
    const uint32_t efield = g.clip ? sh->prefix[it] >> 23 : 0u;
    const uint32_t implicit = efield ? 0x800000u : 0u;
    if (g.clip) {
      // two radix rounds over the low 18 bits of the candidates; the second also gathers exact squares of those
      // below the sub-bin and counts those above (see kp_finalize)
      for (int r = 0; r < 2; ++r) {
        const int shift = r == 0 ? 9 : 0;
        const uint32_t high_mask = ~((1u << (shift + 9)) - 1u) & 0x7FFFFFFFu;
        if (tid < 512) hist[tid] = 0;
        __syncthreads();
        const uint32_t prefix = sh->sel_prefix, rank = sh->sel_rank;
        for (uint32_t i0 = tid; i0 < count; i0 += 8 * kPrepThreads) {
          uint32_t k[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) k[u] = i0 + u * kPrepThreads < count ? ld_cg(m.cand + i0 + u * kPrepThreads) : 0xFFFFFFFFu;
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            if (k[u] == 0xFFFFFFFFu) continue;
            if ((k[u] & high_mask) == (prefix & high_mask)) {
              atomicAdd(&hist[(k[u] >> shift) & 511u], 1u);
            } else if (r == 1) {
              if (k[u] < prefix) {
                const unsigned long long mant = (k[u] & 0x7FFFFFu) | implicit, sq = mant * mant;
                lo += sq & 0xFFFFFFull;
                hi += sq >> 24;
              } else {
                above += 1;
              }
            }
          }
        }
        __syncthreads();
        const uint32_t c = tid < 512 ? hist[tid] : 0u;
        const uint32_t before = block_prefix(c, sh->wtot);
        if (c && rank > before && rank <= before + c) {
          sh->sel_prefix = prefix | ((uint32_t)tid << shift);
          sh->sel_rank = rank - before;
        }
        __syncthreads();
      }
      tau_bits = sh->sel_prefix;
      // a counter of the second round stands for one exact magnitude
      if (tid < 512 && hist[tid]) {
        const uint32_t cnt = hist[tid], kk = (tau_bits & ~511u) | (uint32_t)tid;
        if (kk <= tau_bits) {
          const unsigned long long mant = (kk & 0x7FFFFFu) | implicit, sq = mant * mant;
          lo += (unsigned long long)cnt * (sq & 0xFFFFFFull);
          hi += (unsigned long long)cnt * (sq >> 24);
        } else {
          above += cnt;
        }
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        lo += __shfl_xor_sync(0xffffffffu, lo, o);
        hi += __shfl_xor_sync(0xffffffffu, hi, o);
        above += __shfl_xor_sync(0xffffffffu, above, o);
      }
      if (lane == 0) { sh->wlo[warp] = lo; sh->whi[warp] = hi; sh->wabove[warp] = above; }
    }
    double acc = sum_partials(m.partial, m.tiles, sh->wsum);
    if (warp == 0) {
      if (g.clip) { lo = sh->wlo[lane]; hi = sh->whi[lane]; above = sh->wabove[lane]; }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        lo += __shfl_xor_sync(0xffffffffu, lo, o);
        hi += __shfl_xor_sync(0xffffffffu, hi, o);
        above += __shfl_xor_sync(0xffffffffu, above, o);
      }
      if (lane == 0) {
        float maxabs = __uint_as_float(ld_cg(&hdr->maxabs_bits)), tau = __int_as_float(0x7f800000);
        if (g.clip) {
          tau = __uint_as_float(tau_bits);
          maxabs = tau;
          // clamped to tau: everything in the bins above the picked one, and the candidates above tau
          const double n_clipped = (double)m.n4 * 4.0 - (double)sh->below[it] - (double)sh->bin_count[it] + (double)above;
          acc = clipped_squares(acc, lo, hi, efield, n_clipped, tau);
        }
        const NormScalars ns = norm_scalars(acc, maxabs, g.eps, g.q.widen);
        sh->tau[it] = tau; sh->inv[it] = ns.inv; sh->sg[it] = ns.sg;
        if (owner) {
          if (g.clip) m.scalars[g.ix.tau] = tau;
          write_norm_scalars(m.scalars, g.ix, ns);
        }
      }
    }
    __syncthreads();
  }

  // ---- operand copies of X0 from the resident tiles
  const PrepLane pl = prep_lane();
  for (int it = 0; it < mine; ++it) {
    const PrepTileInfo& ti = sh->info[it];
    const PrepMatrix& m = g.mat[ti.mi];
    if (tid < 8) sh->rcp_tab[tid] = __frcp_rn(__fmul_rn((float)(8 + tid), sh->sg[it]));
    __syncthreads();
    const PrepScalars ps = prep_scalars(sh->tau[it], sh->inv[it], sh->sg[it], smem_u32(&sh->rcp_tab[0]));
    prep_tile<PF>(g, m, ps, pl, smem_u32(smem + it * kPrepTile), uni, ti);
    __syncthreads();
    if (g.write_q) prep_copy_out(g, m, uni, ti);
    __syncthreads();
  }
  if (tid == 0 && sh->abort_flag) report_timeout(g.status);
}

}  // namespace

// Whether a matrix of this many tiles is summed tile by tile, as the single launch does it (at most 1024 partials), and whether
// matrices of `tiles` in all fit that launch.
static bool tiled_sum(int64_t matrix_tiles, int device_sms) { return matrix_tiles <= (int64_t)kResTiles * device_sms && matrix_tiles <= 1024; }
static bool fits_resident(int64_t tiles, int coop_sms) { return tiles <= (int64_t)kResTiles * coop_sms; }

// Estimated time in us: one launch, per tile that a block takes; or six launches, bound by HBM and by their instructions.
// Measured: 8 / 256 / 405 tiles 18 / 29 / 40 us; 8192 x 2048 71 us, sixteen 3072 x 3072 437.
double prologue_us(const WorkShape* w, int count, int device_sms, int coop_sms) {
  int64_t tiles = 0;
  bool tiled = true;
  for (int j = 0; j < count; ++j) {
    const int64_t n = w[j].s / 128 * (w[j].l / 128);
    tiled = tiled && tiled_sum(n, device_sms);
    tiles += n;
  }
  if (tiled && fits_resident(tiles, coop_sms)) return 7.0 + 11.0 * (double)((tiles + coop_sms - 1) / coop_sms);
  return 28.0 + 2.7e-6 * 16384.0 * (double)tiles;
}

cudaError_t prologue_set_attributes() {
  cudaError_t e = cudaFuncSetAttribute(kp_prep_operands<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPrepSmem);
  if (e != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(kp_prep_operands<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPrepSmem))) return e;
  if ((e = cudaFuncSetAttribute(kp_resident<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmem))) return e;
  if ((e = cudaFuncSetAttribute(kp_resident<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmem))) return e;
  if ((e = cudaFuncSetAttribute(kp_resident<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmem))) return e;
  if ((e = cudaFuncSetAttribute(kp_resident<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmem))) return e;
  if ((e = cudaFuncSetAttribute(kp_resident<false, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1))) return e;
  if ((e = cudaFuncSetAttribute(kp_resident<true, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1))) return e;
  // blocks of the largest cluster that the device holds
  int dev = 0;
  if ((e = cudaGetDevice(&dev))) return e;
  for (int blocks = kResCluster; blocks >= 8 && g_cluster_blocks[dev] == 0; blocks /= 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3(kPrepThreads); cfg.dynamicSmemBytes = kResSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)blocks; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int plain = 0, opts = 0;
    if (cudaOccupancyMaxActiveClusters(&plain, kp_resident<false, true>, &cfg) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&opts, kp_resident<true, true>, &cfg) == cudaSuccess && plain > 0 && opts > 0)
      g_cluster_blocks[dev] = blocks;
    else
      cudaGetLastError();
  }
  return cudaSuccess;
}

// Enqueue the prologue for `count` matrices that share clip, eps and options.
cudaError_t launch_prologue_group(const PrologueItem* items, int count, int write_q, const QuantOpts& q,
                                  uint32_t* status, int coop_sms, int sms, cudaStream_t st) {
  for (int i0 = 0; i0 < count; i0 += kMaxPack) {
    const int nn = count - i0 < kMaxPack ? count - i0 : kMaxPack;
    PrepGroup g;
    memset(&g, 0, sizeof(g));
    g.count = nn;
    g.clip = items[i0].pl->clip;
    g.eps = items[i0].pl->eps;
    g.write_q = write_q;
    g.zero_words = (int)(items[i0].pl->zero_bytes / 4);
    g.ix = items[i0].pl->ix;
    g.q = q;
    g.status = status;
    bool all_counted = true, all_tiled = true, none_tiled = true;
    int hist_blocks = 1, stat_tiled = 1, stat_other = 1, select_blocks = 1;
    for (int j = 0; j < nn; ++j) {
      const PrologueItem& it = items[i0 + j];
      const NsPlan& pl = *it.pl;
      const fp4_ws_layout& L = pl.lay;
      PrepMatrix& m = g.mat[j];
      // The candidate list lives in workspace that nothing else uses before the first product: the A buffer
      // (s x s words) or, for a matrix much longer than high, the second set of transposed operand codes
      // (s x l / 8 words).  An eighth of the elements is more than any bin of a spread-out distribution holds.
      const bool cand_in_qxt = pl.s * pl.l / 8 > pl.s * pl.s;
      const int64_t region = cand_in_qxt ? pl.s * pl.l / 8 : pl.s * pl.s;
      m.cand_cap = (uint32_t)(pl.s0 * pl.l0 / 8 < region ? pl.s0 * pl.l0 / 8 : region);
      m.G = it.G; m.X = it.X;
      m.hdr = reinterpret_cast<NsHeader*>(it.ws + L.header);
      m.scalars = reinterpret_cast<float*>(it.ws + L.scalars);
      m.hist = reinterpret_cast<uint32_t*>(it.ws + pl.off_hist);
      m.partial = reinterpret_cast<double*>(it.ws + pl.off_partial);
      m.cand = reinterpret_cast<uint32_t*>(it.ws + (cand_in_qxt ? L.qXt_codes[1] : L.A));
      m.qx_codes = it.ws + L.qX_codes; m.qx_sf = it.ws + L.qX_scales;
      m.qt_codes = it.ws + L.qXt_codes[0]; m.qt_sf = it.ws + L.qXt_scales[0];
      m.tall = pl.tall;
      m.clear_status = it.clear_status ? 1 : 0;
      m.store_x = it.store_x ? 1 : 0;
      m.x_rows = (int)it.x_rows; m.x_cols = (int)it.x_cols;
      m.hist_top = it.hist_top;
      m.n4 = pl.s0 * pl.l0 / 4;
      m.s = (int)pl.s; m.l = (int)pl.l;
      m.s0 = (int)pl.s0; m.l0 = (int)pl.l0;
      m.clip_rank = (uint32_t)pl.clip_rank;
      const int64_t tiles = (pl.l / 128) * (pl.s / 128);
      m.tiled = tiled_sum(tiles, pl.sms);
      m.tiles = (int)tiles;
      m.first_tile = g.tiles;
      g.tiles += m.tiles;
      const int64_t hb = (m.n4 + 512 * 4 - 1) / (512 * 4);
      m.hist_blocks = (int)(hb < (int64_t)sms * 4 ? (hb < 1 ? 1 : hb) : (int64_t)sms * 4);
      m.stat_blocks = m.tiled ? m.tiles : pl.stat_blocks;
      // a block of the select per 4 M elements: some 10 k candidates of a Gaussian matrix
      const int64_t fb = m.n4 >> 20;
      m.select_blocks = (int)(fb < 1 ? 1 : fb < 64 ? fb : 64);
      if (!it.hist_top) {
        all_counted = false;
        hist_blocks = hist_blocks > m.hist_blocks ? hist_blocks : m.hist_blocks;
      }
      int& stat = m.tiled ? stat_tiled : stat_other;
      stat = stat > m.stat_blocks ? stat : m.stat_blocks;
      (m.tiled ? none_tiled : all_tiled) = false;
      select_blocks = select_blocks > m.select_blocks ? select_blocks : m.select_blocks;
      g.tmG[j] = *it.tmG;
    }
    if (all_tiled && fits_resident(g.tiles, coop_sms)) {
      // everything fits the shared memories: one launch
      ProfScope ps(FP4_PROF_PREP, st);
      const bool pf = q.rht || q.four_six;
      cudaLaunchConfig_t cfg = {};
      cfg.blockDim = dim3(kPrepThreads);
      cfg.dynamicSmemBytes = kResSmem; cfg.stream = st;
      cudaLaunchAttribute attr[2];
      cfg.attrs = attr;
      cudaError_t e;
      int dev = 0;
      if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
      if (g.tiles <= g_cluster_blocks[dev] && sms == items[i0].pl->sms) {   // (where a part of the device may lack such a cluster)
        int blocks = 1;
        while (blocks < g.tiles) blocks *= 2;
        cfg.gridDim = dim3((unsigned)blocks);
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)blocks; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
        cfg.numAttrs = 2;
        count_launches(1);
        e = cudaLaunchKernelEx(&cfg, pf ? kp_resident<true, true> : kp_resident<false, true>, g);
        if (e != cudaSuccess) return e;
        continue;
      }
      e = cudaMemsetAsync(&g.mat[0].hdr->barrier, 0, 4, st);
      if (e != cudaSuccess) return e;
      cfg.gridDim = dim3((unsigned)(g.tiles < coop_sms ? g.tiles : coop_sms));
      attr[0].id = cudaLaunchAttributeCooperative;
      attr[0].val.cooperative = 1;
      cfg.numAttrs = 1;
      count_launches(1);
      e = cudaLaunchKernelEx(&cfg, pf ? kp_resident<true, false> : kp_resident<false, false>, g);
      if (e != cudaSuccess) return e;
      continue;
    }
    const dim3 gy1(1, (unsigned)nn), gh((unsigned)hist_blocks, (unsigned)nn);
    {
      ProfScope ps(FP4_PROF_CLIP, st);
      launch_chained(kp_init, dim3(4, (unsigned)nn), dim3(256), 0, st, g);
      count_launches(1);
      if (g.clip) {
        if (!all_counted) launch_chained(kp_hist_top, gh, dim3(512), 0, st, g);
        launch_chained(kp_pick_top, gy1, dim3(512), 0, st, g);
        count_launches(all_counted ? 1 : 2);
      }
    }
    {
      ProfScope ps(FP4_PROF_STATS, st);
      // a pass for each kind of sum
      if (!none_tiled) launch_chained(kp_compact_stats<true>, dim3((unsigned)stat_tiled, (unsigned)nn), dim3(256), 0, st, g);
      if (!all_tiled) launch_chained(kp_compact_stats<false>, dim3((unsigned)stat_other, (unsigned)nn), dim3(256), 0, st, g);
      launch_chained(kp_finalize, dim3((unsigned)select_blocks, (unsigned)nn), dim3(1024), 0, st, g);
      count_launches(none_tiled || all_tiled ? 2 : 3);
    }
    {
      ProfScope ps(FP4_PROF_PREP, st);
      const unsigned gp = (unsigned)(g.tiles < sms ? g.tiles : sms);
      if (q.rht || q.four_six) launch_chained(kp_prep_operands<true>, dim3(gp), dim3(kPrepThreads), kPrepSmem, st, g);
      else launch_chained(kp_prep_operands<false>, dim3(gp), dim3(kPrepThreads), kPrepSmem, st, g);
      count_launches(1);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace fp4
