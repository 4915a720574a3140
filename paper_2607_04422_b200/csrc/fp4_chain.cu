// All iterations of the Newton-Schulz step (Section 3.4, display equations) for a small group of
// matrices, of one or of several shapes, in ONE launch (cooperative, or a single cluster).
//
// A matrix of up to a few million elements has fewer 256 x 256 tiles than the GPU has SM pairs, and with a
// launch per product its time is launch latency, cold instruction fetches and the epilogue of one large tile.
// Here one persistent block per SM walks the products of all iterations in order, in tiles of 128 x 64 or
// 128 x 128 (chosen so that a product fills the SMs).  Nothing is launched between products: a tile of a
// product waits, on a counter in the matrix's workspace header, until all tiles of the matrix's product
// before it are stored.
//
// Work list: product 0, 1, 2, ... and within a product the tiles of all matrices; block b takes the tiles
// b, b + grid, ... of every product.  Every dependency points to an earlier product and all blocks are
// resident (cooperative launch), so the earliest unfinished tile can always run.  Since G1 and G2 list the
// same tiles, and every G3 lists the same tiles, the FP32 values a tile combines with (A in G2, X in G3) were
// written by the very thread that reads them.  So they stay where they are: beside the accumulators the tensor memory has room
// for 6 tiles of 64 columns or 2 of 128, and a block's first tiles of A and X live there from product to product
// (residents); only the caller's matrix in the first G3, the result in the last, and tiles beyond that room
// move through memory (and, stored only, what the workspace keeps of the last iteration).  A block of those is fetched while
// the tile before it is worked on, the first one of a product that has no resident tile before its dependency is even looked
// at; the copies that wrote them have arrived by then, because the warp waits for all its own at the end of the product before.
//
// Warp roles: 0-15 epilogue, 16 operand producer (TMA; also the only thread that polls the counter), 17 MMA
// issuer and TMEM owner, 18 stores.  Epilogue warp w owns the TMEM lanes of quadrant w % 4 and the 16-column
// (or two 16-column) pieces w / 4 of the tile; what moves through memory it moves with its own TMA loads and
// stores, and it shares nothing with the other epilogue warps but the staging area in which the tile's
// quantised outputs are collected.  The store warp sends that area off, waits until it has arrived, publishes
// the running maximum and counts the tile.
//
// Bounds: latency.  A 5-iteration call is a chain of 15 dependent products.  At 256 x 512 a product takes about 4 us:
// operand copies 0.75, MMAs 0.3, the one tile's epilogue 0.75-1.1, its stores and the release 1.1, the counter's way to the
// slowest of the other blocks 0.8.  The epilogue has 96 registers per thread for 16 values in flight: with both passes' values
// in registers at once it spilled, and the spill area of 608 threads does not fit the L1 that the shared memory leaves.  Resident tiles with
// a path of their own that needs nothing else, and the second pass's values read after the first, whole calls: 256 x 512
// 94.7 -> 82.2 us, 1024 x 1024 114.4 -> 101.6, 2048 x 2048 217 -> 198, with the signs of the transform in shared memory 640 x 768
// with the quantiser options 137.6 -> 115.8, 1040 x 2896 212 -> 187; G1 and G2 of 2048 x 6144 with options 510 -> 470.
// With the proxy fence on the reading side and one lane storing everything the iterations of 256 x 512 took 87 us
// instead of 78, of 1408 x 2176 156 instead of 141.  Whole calls against three launches per iteration: 256 x 512
// 152 -> 74 us, 1024 x 1024 178 -> 101, 1040 x 2896 with the paper's quantiser options 300 -> 186.
#include "fp4_gemm_common.cuh"

namespace fp4 {

namespace {

constexpr int BM = 128, BK = 256, KSTEPS = BK / 64;
constexpr int CHUNK = 16;
constexpr int NACC = 2;                       // accumulator buffers at most (ChainLaunch::nacc)
constexpr int EPI_WARPS = 16;
constexpr int W_LOAD = EPI_WARPS, W_MMA = EPI_WARPS + 1, W_STORE = EPI_WARPS + 2;
constexpr int NTHREADS = (EPI_WARPS + 3) * 32;
constexpr int DEP_RING = 16;
constexpr int XBUF = 32 * 64;                 // a warp's 32 x 16 FP32 block: 64-byte rows, 64-byte swizzle
constexpr int MAX_STAGES = 5;
constexpr int SHARED_BYTES = 2304;            // of ChainShared
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t SF_COLS = KSTEPS * 8;      // per stage: 4 columns per MMA for each operand
constexpr uint32_t SF_RING = 2 * SF_COLS;     // copies and MMAs execute in issue order: two stages' columns in turn
constexpr uint32_t ACC_COL = SF_RING;         // then the accumulators, then the resident tiles
// Tiles of A and X that stay in the tensor memory beside nacc accumulators
__host__ __device__ constexpr int resident_slots(int bn, int nacc) { return ((int)TMEM_COLS - (int)SF_RING - nacc * bn) / bn; }

template <int BN>
struct ChainLay {
  static constexpr int STAGES = BN == 64 ? 5 : 3;
  static constexpr int A_BYTES = BM * BK / 2, B_BYTES = BN * BK / 2, SF_BYTES = KSTEPS * 512;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES + 2 * SF_BYTES;
  static constexpr int CHUNKS = BN / 64;      // 16-column chunks per epilogue warp
  // staging area of a tile's quantised outputs: row codes [64-column half][128 rows][32 bytes], column codes
  // [BN columns][64 bytes] with a 64-byte swizzle, row scale atoms, column scales [2 atoms][32][BN / 32 words]
  static constexpr int RQ = BM * BN / 2, CQ = BN * BM / 2, RSF = BN / 64 * 512, CSF = BN * 8;
  static constexpr int OUT = RQ + CQ + 1024 * ((RSF + CSF + 1023) / 1024);
  static constexpr int OFF_X = STAGES * STAGE_BYTES;         // two blocks per epilogue warp
  static constexpr int OFF_OUT = OFF_X + EPI_WARPS * 2 * XBUF;  // two areas, used by alternate tiles
  static constexpr int OFF_BAR = OFF_OUT + 2 * OUT;
  static constexpr int SMEM = OFF_BAR + SHARED_BYTES + 1024;
  static_assert(SMEM <= 232448 && STAGE_BYTES % 1024 == 0 && OFF_OUT % 1024 == 0 && OUT % 1024 == 0, "shared memory");
  static_assert(STAGES <= MAX_STAGES && resident_slots(BN, NACC) >= 1, "tensor memory columns");
  // M = 128, N = BN, E2M1 x E2M1, UE4M3 scales, K-major operands
  static constexpr uint32_t IDESC = (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
};

struct ChainShared {
  uint64_t full[MAX_STAGES], empty[MAX_STAGES];
  uint64_t acc_full[NACC], acc_empty[NACC];
  uint64_t dep[DEP_RING];          // the tile's dependency is met (one arrival by the producer per tile)
  uint64_t xfull[EPI_WARPS * 2];   // an FP32 block has landed
  uint64_t out_done[2], out_free[2];
  alignas(16) uint32_t amax[2][4]; // running maximum of the tile in a staging area (bit pattern), at its place among four slots
  alignas(16) float signs[EPI_WARPS][16];   // of the product at hand, a copy per epilogue warp
  float clip[EPI_WARPS][2];                 // threshold and reciprocal norm of the matrix at hand, a copy per epilogue warp
  uint32_t tmem_base, abort_flag;
  uint32_t tiles[2][kChainTiles];  // this block's tiles of a symmetric product / of G3: p << 28 | ti << 16 | tj
  uint16_t depth[3][kChainTiles];  // their contraction lengths in G1, G2, G3, in blocks of 128
};
static_assert(sizeof(ChainShared) <= SHARED_BYTES, "shared block");

// Tile t of a product of all matrices; the symmetric products list the tiles whose 128-column block is on or above the diagonal.
template <int BN>
__device__ __forceinline__ uint32_t chain_tile(int t, bool sym, const ChainProblem* probs, int count) {
  int p = 0;
  while (p + 1 < count && t >= (sym ? probs[p + 1].first_sym : probs[p + 1].first_full)) ++p;
  t -= sym ? probs[p].first_sym : probs[p].first_full;
  const int cols = (sym ? probs[p].s : probs[p].l) / BN;
  int ti, tj;
  if (!sym) {
    ti = t / cols;
    tj = t - ti * cols;
  } else {
    constexpr int R = BM / BN;
    int row = 0, len = cols;
    while (t >= len) { t -= len; ++row; len -= R; }
    ti = row;
    tj = row * R + t;
  }
  return (uint32_t)p << 28 | (uint32_t)ti << 16 | (uint32_t)tj;
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_add(uint32_t* p, uint32_t v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// running maxima (non-negative floats order like unsigned integers): four words at once, 16-byte aligned
__device__ __forceinline__ void bulk_max16_s(void* dst, uint32_t src) {
  asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.max.u32 [%0], [%1], 16;" ::"l"(dst), "r"(src) : "memory");
}
__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// scalars written by other blocks of this launch: never from L1
__device__ __forceinline__ float ld_scalar(const float* p) {
  return __uint_as_float(ld_relaxed(reinterpret_cast<const uint32_t*>(p)));
}
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ void sts_f4(uint32_t a, float x, float y, float z, float w) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
__device__ __forceinline__ void sts_u2(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void sts_b(uint32_t a, uint32_t x) {
  asm volatile("st.shared.b8 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}
__device__ __forceinline__ float4 lds_f4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float lds_f1(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void tma_load_s(uint32_t dst, const void* tmap, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(tmap), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_store_s(const void* tmap, int x, int y, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(tmap), "r"(x), "r"(y),
               "r"(src)
               : "memory");
}
__device__ __forceinline__ void bulk_store_s(void* dst, uint32_t src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_expect_s(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// A resident block of FP32 values -> 32 lanes x 16 columns of the tensor memory (lane = row), rounded to BF16 on request;
// done when the warp's next tcgen05.wait::st returns.
__device__ __forceinline__ void tc_st16(uint32_t taddr, const float (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]), "f"(r[8]), "f"(r[9]), "f"(r[10]),
      "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15])
      : "memory");
}
__device__ __forceinline__ void store_state(uint32_t taddr, const float (&v)[16], bool round) {
  if (!round) {
    tc_st16(taddr, v);
    return;
  }
  float h[16];
#pragma unroll
  for (int i = 0; i < 16; i += 2) {
    const uint32_t z = cvt_bf16x2(v[i], v[i + 1]);
    h[i] = bf16_lo(z);
    h[i + 1] = bf16_hi(z);
  }
  tc_st16(taddr, h);
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Root's parameter update of a tall matrix: the parameter has the caller's orientation, so the 16 values of this
// lane's row lie a row of the parameter apart.
__device__ __noinline__ void chain_update_tall(uint16_t* w, int64_t ld, const float (&v)[16], float decay, float step) {
#pragma unroll 4
  for (int i = 0; i < 16; ++i, w += ld)
    *w = (uint16_t)cvt_bf16x2(param_update_value(bf16_lo(*w), v[i], decay, step), 0.0f);
}

// SYM: the products [a.first, a.end) only, G1 and G2 of an iteration (loop bounds the compiler cannot unroll by); else all products of all iterations
template <int BN, bool PF, bool SYM, int MAX>
__global__ void __launch_bounds__(NTHREADS, 1)
k_chain(const __grid_constant__ ChainPackOf<MAX> pack, const __grid_constant__ ChainLaunch a) {
  using L = ChainLay<BN>;
  constexpr int STAGES = L::STAGES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  ChainShared* sh = reinterpret_cast<ChainShared*>(smem + L::OFF_BAR);
  volatile uint32_t* abort_flag = &sh->abort_flag;
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int grid = (int)gridDim.x;
  // tiles of this block
  const int my_sym = (a.sym_tiles - (int)blockIdx.x + grid - 1) / grid;
  const int my_full = (a.full_tiles - (int)blockIdx.x + grid - 1) / grid;
  const int products = 3 * a.steps;
  const int first = SYM ? a.first : 0, end = SYM ? a.end : products;
  const bool two_acc = a.nacc == 2;

  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) { mbar_init(&sh->full[i], 1); mbar_init(&sh->empty[i], 1); }
    for (int i = 0; i < NACC; ++i) { mbar_init(&sh->acc_full[i], 1); mbar_init(&sh->acc_empty[i], EPI_WARPS); }
    for (int i = 0; i < DEP_RING; ++i) mbar_init(&sh->dep[i], 1);
    for (int i = 0; i < EPI_WARPS * 2; ++i) mbar_init(&sh->xfull[i], 1);
    for (int i = 0; i < 2; ++i) { mbar_init(&sh->out_done[i], EPI_WARPS); mbar_init(&sh->out_free[i], 1); for (int q = 0; q < 4; ++q) sh->amax[i][q] = 0; }
    sh->abort_flag = 0;
    mbar_fence_init();
  }
  for (int i = (int)threadIdx.x - 64; i >= 0 && i < 2 * kChainTiles; i += NTHREADS) {
    const int list = i / kChainTiles, j = i % kChainTiles;
    if (j < (list ? my_full : my_sym)) {
      const uint32_t tile = chain_tile<BN>((int)blockIdx.x + j * grid, list == 0, pack.p, a.count);
      const ChainProblem& pr = pack.p[tile >> 28];
      sh->tiles[list][j] = tile;
      sh->depth[list ? 2 : 1][j] = (uint16_t)(pr.s / 128);
      if (!list) sh->depth[0][j] = (uint16_t)(pr.l / 128);
    }
  }
  for (int i = (int)threadIdx.x; i < a.count * kChainMaps; i += NTHREADS)   // descriptors come first in a problem
    tma_prefetch_desc(reinterpret_cast<const CUtensorMap*>(&pack.p[i / kChainMaps]) + i % kChainMaps);
  if (warp == W_MMA) {
    tmem_alloc(&sh->tmem_base, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = sh->tmem_base;
  pdl_wait();   // set-up done; from here on the kernel reads what the launch before it wrote

  if (warp == W_LOAD) {
    // ------------------------------------------------------------ operand producer
    if (elect_one()) {
      // until `need` tiles of a matrix are stored
      auto wait_tiles = [&](const uint32_t* done, uint32_t need) {
        bool met = ld_acquire(done) >= need;
        if (met) return;
        const uint64_t t0 = globaltimer_ns();
        for (;;) {
          for (int i = 0; i < 64 && !met; ++i) met = ld_acquire(done) >= need;
          if (met) break;
          if (*abort_flag || globaltimer_ns() - t0 > kWaitLimitNs) { *abort_flag = 1; break; }
        }
      };
      int st = 0; uint32_t ph = 0, n = 0;
      for (int pi = first; pi < end; ++pi) {
        const int k = pi / 3, mode = pi - 3 * k + kG1;
        const bool sym = mode != kG3;
        const int mine = sym ? my_sym : my_full;
        int seen = -1;
        for (int j = 0; j < mine; ++j, ++n) {
          const uint32_t tile = sh->tiles[sym ? 0 : 1][j];
          const int p = (int)(tile >> 28), ti = (int)(tile >> 16) & 0xFFF, tj = (int)(tile & 0xFFFF);
          const ChainProblem& pr = pack.p[p];
          const int K = sh->depth[mode - kG1][j] * 128;
          const int num_kb = (K + BK - 1) / BK;
          const CUtensorMap* ma = mode == kG1 ? &pr.tm_qX : mode == kG2 ? &pr.tm_qA : &pr.tm_qB;
          const CUtensorMap* mb = mode == kG1 ? &pr.tm_qX : mode == kG2 ? &pr.tm_qA : &pr.tm_qXt[k & 1];
          const uint8_t* sfa = (mode == kG1 ? pr.qx_sf : mode == kG2 ? pr.qa_sf : pr.qb_sf) + (size_t)ti * (K / 64) * 512;
          const uint8_t* sfb = (mode == kG1 ? pr.qx_sf : mode == kG2 ? pr.qa_sf : pr.qt_sf[k & 1]) +
                               (size_t)(tj * BN / 128) * (K / 64) * 512;
          // A half-full last stage: the operand boxes are zero-filled beyond K (and still credit their full
          // size), only the scale atoms that exist are fetched.
          auto sf_bytes = [&](int kb) { return (uint32_t)((K - kb * BK < BK ? K - kb * BK : BK) / 64) * 512; };
          auto load_rows = [&](int s_, int kb) {
            uint8_t* d = smem + s_ * L::STAGE_BYTES;
            tma_load_2d(d, ma, kb * (BK / 2), ti * BM, &sh->full[s_]);
            tma_load_2d(d + L::A_BYTES / 2, ma, kb * (BK / 2), ti * BM + 64, &sh->full[s_]);
            bulk_load_1d(d + L::A_BYTES + L::B_BYTES, sfa + (size_t)kb * L::SF_BYTES, sf_bytes(kb), &sh->full[s_]);
          };
          auto load_cols = [&](int s_, int kb) {
            uint8_t* d = smem + s_ * L::STAGE_BYTES;
            mbar_expect_tx(&sh->full[s_], L::A_BYTES + L::B_BYTES + 2 * sf_bytes(kb));
#pragma unroll
            for (int h = 0; h < BN / 64; ++h)
              tma_load_2d(d + L::A_BYTES + h * (64 * BK / 2), mb, kb * (BK / 2), tj * BN + h * 64, &sh->full[s_]);
            bulk_load_1d(d + L::A_BYTES + L::B_BYTES + L::SF_BYTES, sfb + (size_t)kb * L::SF_BYTES, sf_bytes(kb), &sh->full[s_]);
          };
          // tiles of the matrix's earlier products (SYM: what the launches before have left is complete)
          const uint32_t before = (uint32_t)(k * (2 * pr.nsym + (pr.s / BM) * (pr.l / BN)));
          const uint32_t need = SYM ? (mode == kG1 ? 0u : (uint32_t)((2 * k + 1) * pr.nsym)) : before + (uint32_t)((mode - kG1) * pr.nsym);
          int ahead = 0;
          if (p != seen && need != 0) {
            if (!SYM && mode == kG3) {
              // The column operand of G3 comes from the iteration before: its first stages are fetched while B is still under way.
              // 1024 x 1024 101.7 -> 99.8 us, 256 x 512 82.9 -> 82.2, 1040 x 2896 with options 186.2 -> 184.4, 2048 x 2048 196.4 -> 195.9.
              if (before != 0) wait_tiles(pr.done, before);
              ahead = num_kb < STAGES ? num_kb : STAGES;
              int s_ = st; uint32_t ph_ = ph;
              for (int kb = 0; kb < ahead; ++kb) {
                wait_or_abort(&sh->empty[s_], ph_ ^ 1, abort_flag);
                load_cols(s_, kb);
                if (++s_ == STAGES) { s_ = 0; ph_ ^= 1; }
              }
            }
            wait_tiles(pr.done, need);
          }
          seen = p;
          mbar_arrive(&sh->dep[n % DEP_RING]);
          for (int kb = 0; kb < num_kb; ++kb) {
            if (kb >= ahead) {
              wait_or_abort(&sh->empty[st], ph ^ 1, abort_flag);
              load_cols(st, kb);
            }
            load_rows(st, kb);
            if (++st == STAGES) { st = 0; ph ^= 1; }
          }
        }
      }
    }
  } else if (warp == W_MMA) {
    // ------------------------------------------------------------ MMA issuer
    if (elect_one()) {
      int st = 0; uint32_t ph = 0, n = 0;
      for (int pi = first; pi < end; ++pi) {
        const int mode = pi % 3 + kG1;
        const bool sym = mode != kG3;
        const int mine = sym ? my_sym : my_full;
        int p = 0;
        for (int j = 0; j < mine; ++j, ++n) {
          // from the block's index and the parameters, which the compiler knows to be uniform, as the descriptors have to be
          const int t = (int)blockIdx.x + j * grid;
          while (p + 1 < a.count && t >= (sym ? pack.p[p + 1].first_sym : pack.p[p + 1].first_full)) ++p;
          const int K = mode == kG1 ? pack.p[p].l : pack.p[p].s;
          const int num_kb = (K + BK - 1) / BK;
          // scale atoms cover 128 rows of the column operand: an odd 64-column tile uses their upper half
          const uint32_t sfb_shift = BN == 64 ? 2u * (sh->tiles[sym ? 0 : 1][j] & 1u) : 0u;
          const uint32_t ab = two_acc ? n & 1u : 0u;
          wait_or_abort(&sh->acc_empty[ab], ((two_acc ? n >> 1 : n) & 1) ^ 1, abort_flag);
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + ACC_COL + ab * BN;
          for (int kb = 0; kb < num_kb; ++kb) {
            wait_or_abort(&sh->full[st], ph, abort_flag);
            tc_fence_after();
            const uint32_t sf_t = tmem_base + (uint32_t)(kb & 1) * SF_COLS;
            const uint32_t d = smem_u32(smem + st * L::STAGE_BYTES);
            const int ksteps = (K - kb * BK < BK ? K - kb * BK : BK) / 64;
            const uint64_t adesc = umma_desc(d, 1024, 2), bdesc = umma_desc(d + L::A_BYTES, 1024, 2);
#pragma unroll
            for (int i = 0; i < KSTEPS; ++i) {
              if (i < ksteps) {
                tc_cp_sf(sf_t + i * 4, umma_desc(d + L::A_BYTES + L::B_BYTES + i * 512, 128, 0));
                tc_cp_sf(sf_t + KSTEPS * 4 + i * 4, umma_desc(d + L::A_BYTES + L::B_BYTES + L::SF_BYTES + i * 512, 128, 0));
                tc_mma_nvf4(d_tmem, adesc + 2 * i, bdesc + 2 * i, L::IDESC, sf_t + i * 4, sf_t + KSTEPS * 4 + i * 4 + sfb_shift,
                            (kb | i) != 0 ? 1u : 0u);
              }
            }
            tc_commit(&sh->empty[st]);
            if (++st == STAGES) { st = 0; ph ^= 1; }
          }
          tc_commit(&sh->acc_full[ab]);
        }
      }
    }
  } else if (warp == W_STORE) {
    // ------------------------------------------------------------ stores of the quantised outputs
    uint32_t n = 0;
    for (int pi = first; pi < end; ++pi) {
      const int k = pi / 3, mode = pi - 3 * k + kG1;
      const bool sym = mode != kG3;
      const int mine = sym ? my_sym : my_full;
      if (pi == products - 1 && !a.keep) break;
      for (int j = 0; j < mine; ++j, ++n) {
        const uint32_t tile = sh->tiles[sym ? 0 : 1][j];
        const int p = (int)(tile >> 28), ti = (int)(tile >> 16) & 0xFFF, tj = (int)(tile & 0xFFFF);
        const ChainProblem& pr = pack.p[p];
        const bool mirror = mode == kG3 || tj * BN / 128 != ti;
        uint8_t* ob = smem + L::OFF_OUT + (n & 1) * L::OUT;
        const uint32_t os = smem_u32(ob);
        const CUtensorMap* mr = mode == kG1 ? &pr.st_qA : mode == kG2 ? &pr.st_qB : &pr.st_qX;
        const CUtensorMap* mc = mode == kG1 ? &pr.st_qAc : mode == kG2 ? &pr.st_qBc : &pr.st_qXt[(k & 1) ^ 1];
        uint8_t* sym_sf = mode == kG1 ? pr.qa_sf : pr.qb_sf;
        uint8_t* rsf = (sym ? sym_sf : pr.qx_sf) + ((int64_t)ti * ((sym ? pr.s : pr.l) / 64) + tj * (BN / 64)) * 512;
        uint8_t* csf = (sym ? sym_sf : pr.qt_sf[(k & 1) ^ 1]) + ((int64_t)(tj * BN / 128) * (pr.s / 64) + ti * 2) * 512;
        const int slot = mode == kG1 ? a.ix.amax_A0 + k : a.ix.amax_X0 + k + 1;
        float* maxima = pr.scalars + (slot & ~3);
        uint32_t* done = pr.done;
        wait_or_abort(&sh->out_done[n & 1], (n >> 1) & 1, abort_flag);
        if (lane == 0) {
#pragma unroll
          for (int h = 0; h < BN / 64; ++h) tma_store_s(mr, tj * (BN / 2) + h * 32, ti * BM, os + h * 4096);
          bulk_store_s(rsf, os + L::RQ + L::CQ, L::RSF);
          if (mirror) {
#pragma unroll
            for (int h = 0; h < BN / 64; ++h) tma_store_s(mc, ti * 64, tj * BN + h * 64, os + L::RQ + h * 4096);
            if (BN == 128) bulk_store_s(csf, os + L::RQ + L::CQ + L::RSF, L::CSF);
          }
          if (mode != kG2) bulk_max16_s(maxima, smem_u32(&sh->amax[n & 1][0]));
          bulk_commit();
        } else if (BN == 64 && mirror && lane >= 16) {
          // The scales of 64 rows are the 8-byte halves of the 16-byte rows of two atoms: stored by other lanes than
          // the one that waits for the copies (its release would wait for its own stores again), and fenced here,
          // because the next product's TMA loads read what the generic proxy wrote.
          uint8_t* dst = csf + (lane - 16) * 16 + (tj & 1) * 8;
          const uint8_t* src = ob + L::RQ + L::CQ + L::RSF + (lane - 16) * 8;
#pragma unroll
          for (int q = 0; q < 4; ++q)
            *reinterpret_cast<uint2*>(dst + (q >> 1) * 512 + (q & 1) * 256) = *reinterpret_cast<const uint2*>(src + q * 128);
          fence_proxy_async_global();
        }
        __syncwarp();
        if (lane == 0) {
          bulk_wait_all<0>();
          sh->amax[n & 1][slot & 3] = 0;
        }
        __syncwarp();
        if (lane == 0) {
          red_release_add(done, 1u);
          mbar_arrive(&sh->out_free[n & 1]);
        }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue warps
    const int quad = warp & 3, team = warp >> 2;
    const int cq = lane & 15, g = lane >> 4;
    const uint32_t area = smem_u32(smem + L::OFF_X + warp * 2 * XBUF);
    const uint32_t xfull = smem_u32(&sh->xfull[warp * 2]);
    // row-per-lane view of a block: 16-byte group j of this lane's row at row_addr ^ (j << 4)
    const uint32_t row_addr = area + lane * 64 + (((lane >> 1) & 3) << 4);
    // column view: at step k the lane reads row k ^ g of its 16-row group (in step the half-warps, whose rows are
    // 16 apart, would hit the same banks), at col_base | (col_lane ^ (k << 6 | (k >> 1 & 3) << 4))
    const uint32_t col_base = area + g * (16 * 64);
    const uint32_t col_lane = (uint32_t)(g << 6 | cq << 2);
    const uint32_t tm_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
    const uint32_t tm_state = tm_lane + ACC_COL + (two_acc ? 2u : 1u) * BN;   // resident tiles: X first, then A
    // staging offsets of this lane's outputs (chunk 0 of the warp)
    const uint32_t out0 = smem_u32(smem + L::OFF_OUT);
    const int row = quad * 32 + lane;
    const uint32_t signs = smem_u32(&sh->signs[warp & (EPI_WARPS - 1)][0]);

    // Lane 0 starts the copy of the FP32 block a unit (tile, chunk) combines with.
    auto fetch = [&](int mode, int k, uint32_t tile, int c, int b) {
      if (lane == 0) {
        const ChainProblem& pr = pack.p[tile >> 28];
        const int y = ((int)(tile >> 16) & 0xFFF) * BM + quad * 32;
        const int x = (int)(tile & 0xFFFF) * BN + (team * L::CHUNKS + c) * CHUNK;
        const CUtensorMap* m = mode == kG2 ? &pr.tm_A : k == 0 ? &pr.tm_G : &pr.tm_X;
        const bool tr = mode == kG3 && k == 0 && pr.tall;
        mbar_expect_s(xfull + b * 8, XBUF);
        tma_load_s(area + b * XBUF, m, tr ? y : x, tr ? x : y, xfull + b * 8);
      }
    };

    uint32_t n = 0, unit = 0, xph = 0;   // tiles, units, phases of the two block barriers
    bool have = false;                   // the copy of the unit at hand is under way
    for (int pi = first; pi < end; ++pi) {
      // The workspace keeps A of the last iteration and, of a tall matrix whose result leaves transposed, the X before that.  While
      // the other blocks finish the product before the last one (SYM: before the last G2), the resident tiles of both are copied
      // out, through the buffer that holds no fetched block.  (X of a wide matrix lies in `out`, where nothing would order such
      // a copy and the result.  With a.keep the tiles of G1 store A themselves, and the last G3 X.)  Had the tiles stored them in
      // the last iteration, 256 x 512 would take 1.4 us more instead of 0.4, 2048 x 2048 5 instead of 0.3.
      if (!a.keep && pi == products - (SYM ? 2 : 1)) {
        const int tiles_a = min(my_sym, a.na), tiles_x = !SYM && a.tall && a.steps > 1 ? min(my_full, a.nx) : 0;
        const uint32_t dst = (unit & 1) ? 0u : (uint32_t)XBUF;
#pragma unroll 1
        for (int i = 0; i < (tiles_a + tiles_x) * L::CHUNKS; ++i) {
          const int j = i / L::CHUNKS, ch = team * L::CHUNKS + i % L::CHUNKS;
          const bool is_a = j < tiles_a;
          const uint32_t tile = sh->tiles[is_a ? 0 : 1][is_a ? j : j - tiles_a];
          const ChainProblem& pr = pack.p[tile >> 28];
          if (!is_a && !pr.tall) continue;
          float v[16];
          tc_ld16(tm_state + (uint32_t)(is_a ? a.nx + j : j - tiles_a) * BN + ch * CHUNK, v);
          if (lane == 0) bulk_wait_read<0>();
          __syncwarp();
#pragma unroll
          for (int q = 0; q < 4; ++q) sts_f4((row_addr + dst) ^ (q << 4), v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_s(is_a ? &pr.tm_A : &pr.tm_X, (int)(tile & 0xFFFF) * BN + ch * CHUNK,
                        ((int)(tile >> 16) & 0xFFF) * BM + quad * 32, area + dst);
            bulk_commit();
          }
        }
      }
      const int k = pi / 3, mode = pi - 3 * k + kG1;
      const bool sym = mode != kG3;
      const int mine = sym ? my_sym : my_full;
      const bool last = pi == products - 1;
      const bool do_q = !last || a.keep;
      const bool raw = mode == kG3 && k == 0;
      int cur_p = -1;
      float scale = 0.0f, inv_sg = 1.0f, beta = 0.0f, gamma = 0.0f;
      bool fused = false;
      if (PF && a.q.rht) {
        const int j = mode == kG1 ? 2 * k + 1 : mode == kG2 ? 2 * k : 2 * k + 2;
        const uint32_t mask = rht_signs(a.seed, (uint64_t)j);
        if (lane < 16) sh->signs[warp][lane] = (mask >> lane & 1u) ? -1.0f : 1.0f;
        __syncwarp();
      }
      for (int j = 0; j < mine; ++j, ++n) {
        const uint32_t tile = sh->tiles[sym ? 0 : 1][j];
        const int p = (int)(tile >> 28), ti = (int)(tile >> 16) & 0xFFF, tj = (int)(tile & 0xFFFF);
        const ChainProblem& pr = pack.p[p];
        const bool xposed = raw && pr.tall;
        const bool mirror = do_q && (mode == kG3 || tj * BN / 128 != ti);
        const bool out_t = last && pr.tall;              // the result of a tall matrix leaves transposed
        wait_or_abort(&sh->dep[n % DEP_RING], (n / DEP_RING) & 1, abort_flag);
        if (p != cur_p) {
          cur_p = p;
          const float* sc = pr.scalars;
          float sg_out, bound;
          if (mode == kG1) {
            const float sgx = ld_scalar(sc + a.ix.sg_X0 + k), ax = ld_scalar(sc + a.ix.amax_X0 + k);
            scale = __fmul_rn(sgx, sgx);
            bound = fminf(__fmul_rn(__fmul_rn(__fmul_rn(2.0f, pr.l_cols), ax), ax), 4.0f);
          } else if (mode == kG2) {
            const float sga = ld_scalar(sc + a.ix.sg_A0 + k), aa = ld_scalar(sc + a.ix.amax_A0 + k);
            scale = __fmul_rn(sga, sga);
            bound = __fmul_rn(__fadd_rn(fabsf(pr.cb), __fmul_rn(4.0f, fabsf(pr.cc))), aa);
            beta = pr.cb;
            gamma = __fmul_rn(pr.cc, scale);   // exact: sga is a power of two
          } else {
            const float sgb = ld_scalar(sc + a.ix.sg_B0 + k), sgx = ld_scalar(sc + a.ix.sg_X0 + k);
            const float ax = ld_scalar(sc + a.ix.amax_X0 + k);
            scale = __fmul_rn(sgb, sgx);
            bound = __fmul_rn(__fmul_rn(4.0f, fabsf(pr.ca)), ax);
            beta = pr.ca;
            gamma = scale;
            // Fetched with the matrix, not with every tile of the first G3, where nothing covers the two loads: one launch of
            // 1280 x 8192 318 -> 305 us, 8192 x 1280 with BF16 storage 323 -> 311, 1024 x 10240 316 -> 302.  In shared memory:
            // registers for the one product that needs them would be spilled in all (309, 313, 306).
            if (raw && lane == 0) {
              sh->clip[warp & (EPI_WARPS - 1)][0] = a.clip ? ld_scalar(sc + a.ix.tau) : __int_as_float(0x7f800000);
              sh->clip[warp & (EPI_WARPS - 1)][1] = ld_scalar(sc + a.ix.inv);
            }
            __syncwarp();
          }
          sg_out = scale_predicted(__fmul_rn(a.q.widen, bound));
          inv_sg = __frcp_rn(sg_out);
          // a power-of-two scale multiplies exactly, so fl(fl(a x) + fl(acc scale)) is one fused operation
          fused = mode == kG3 && (__float_as_uint(scale) & 0x007FFFFFu) == 0 && scale > 1e-30f && scale < 1e30f;
          // the matrix's first tile publishes its output scale (all epilogue warps of the block arrive on
          // out_done after this, and the store warp counts the tile after that)
          if (ti == 0 && tj == 0 && threadIdx.x == 0)
            pr.scalars[mode == kG1 ? a.ix.sg_A0 + k : mode == kG2 ? a.ix.sg_B0 + k : a.ix.sg_X0 + k + 1] = sg_out;
        }
        const uint32_t ab = two_acc ? n & 1u : 0u;
        // This tile's X (G3) or A (G1, G2) lies in the tensor memory; the first G3 reads the caller's matrix, the last
        // one writes the caller's result.
        const bool resident = mode == kG3 ? j < a.nx : j < a.na;
        const bool from_tm = resident && (mode == kG2 || (mode == kG3 && !raw));
        const bool to_tm = resident && (mode == kG1 || (mode == kG3 && !last));
        const uint32_t state = tm_state + (uint32_t)(mode == kG3 ? j : a.nx + j) * BN;
        const uint32_t os = out0 + (n & 1) * L::OUT;
        float amax = 0.0f;
        // ---- the common tile: nothing but its quantised outputs leaves the SM.  What it needs is in registers before the
        // accumulator is waited for, and the FP32 block goes through shared memory for the pass down the columns only.
        if (resident && !raw && !last && !(a.keep && mode == kG1)) {
          wait_or_abort(&sh->out_free[n & 1], ((n >> 1) & 1) ^ 1, abort_flag);   // the stores of the tile two back
          if (lane == 0) bulk_wait_read<0>();
          const bool has_x = mode != kG1, round = a.bf16 && to_tm;
          const float g1 = mode == kG1 ? scale : gamma;
          const uint64_t b2 = pack2(beta, beta), g2 = pack2(g1, g1);
          // The second 16 rows of the block are stored with neighbouring rows swapped: the half-warps, whose rows are 16 apart, then
          // read down their columns in the same order and never meet in a bank.
          const uint32_t put = area + (((uint32_t)lane ^ (uint32_t)g) << 6) + (((lane >> 1) & 3) << 4);
          const uint32_t get = area + (uint32_t)(g << 10 | g << 6 | cq << 2);
          // the next tile's block, when it comes from memory: into the warp's second buffer, this tile uses the first
          have = has_x && j + 1 < mine && j + 1 >= (mode == kG3 ? a.nx : a.na);
          if (have) fetch(mode, k, sh->tiles[sym ? 0 : 1][j + 1], 0, 1);
          unit = 1;
          __syncwarp();
          wait_or_abort(&sh->acc_full[ab], (two_acc ? n >> 1 : n) & 1, abort_flag);
          tc_fence_after();
#pragma unroll 1
          for (int c = 0; c < L::CHUNKS; ++c) {
            const int ch = team * L::CHUNKS + c;
            uint32_t acc[16];
            float v[16];
            tc_ld16_issue(tm_lane + ACC_COL + ab * BN + ch * CHUNK, acc);
            if (has_x) {
              uint32_t x[16];
              tc_ld16_issue(state + ch * CHUNK, x);
              tc_wait_ld16(acc);
              tc_wait_ld16(x);
#pragma unroll
              for (int i = 0; i < 16; i += 2) {
                const uint64_t ac2 = pack2(__uint_as_float(acc[i]), __uint_as_float(acc[i + 1]));
                const uint64_t bx = mul2(b2, pack2(__uint_as_float(x[i]), __uint_as_float(x[i + 1])));
                if (fused) {
                  unpack2(fma2(ac2, g2, bx), v[i], v[i + 1]);
                } else {
                  float t0, t1, u0, u1;
                  unpack2(bx, t0, t1);
                  unpack2(mul2(ac2, g2), u0, u1);
                  v[i] = __fadd_rn(t0, u0);
                  v[i + 1] = __fadd_rn(t1, u1);
                }
              }
            } else {
              tc_wait_ld16(acc);
#pragma unroll
              for (int i = 0; i < 16; i += 2)
                unpack2(mul2(pack2(__uint_as_float(acc[i]), __uint_as_float(acc[i + 1])), g2), v[i], v[i + 1]);
            }
            if (c == L::CHUNKS - 1) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&sh->acc_empty[ab]);
            }
            if (mirror) {
              if (L::CHUNKS > 1) __syncwarp();   // every lane has read its column of the block before
#pragma unroll
              for (int i = 0; i < 4; ++i) sts_f4(put ^ (i << 4), v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
              __syncwarp();
            }
            if (to_tm) store_state(state + ch * CHUNK, v, round);
            uint32_t lo, hi, sb;
            float bmax;
            if (PF) sb = quantize_block16_opts_p2<false>(v, a.q, inv_sg, lo, hi, bmax, signs);
            else sb = quantize_block16_p2(v, inv_sg, lo, hi, bmax);
            amax = fmaxf(amax, bmax);
            sts_u2(os + (ch >> 2) * 4096 + row * 32 + (((ch & 3) * 8) ^ ((lane & 4) << 2)), lo, hi);
            sts_b(os + L::RQ + L::CQ + (ch >> 2) * 512 + lane * 16 + quad * 4 + (ch & 3), sb);
            if (mirror) {
#pragma unroll
              for (int i = 0; i < 16; ++i) v[i] = lds_f1(get ^ (uint32_t)(i << 6 | ((i >> 1) & 3) << 4));
              if (PF) sb = quantize_block16_opts_p2<false>(v, a.q, inv_sg, lo, hi, bmax, signs);
              else sb = quantize_block16_p2(v, inv_sg, lo, hi, bmax);
              const int col = ch * CHUNK + cq;
              sts_u2(os + L::RQ + col * 64 + ((quad ^ ((col >> 1) & 3)) << 4) + g * 8, lo, hi);
              sts_b(os + L::RQ + L::CQ + L::RSF + (quad >> 1) * (BN * 4) + (col & 31) * (BN / 8) + (col >> 5) * 4 + (quad & 1) * 2 + g, sb);
            }
          }
          if (mode != kG2) {
            const int slot = mode == kG1 ? a.ix.amax_A0 + k : a.ix.amax_X0 + k + 1;
            const uint32_t wm = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));
            if (lane == 0) atomicMax(&sh->amax[n & 1][slot & 3], wm);
          }
          fence_proxy_async_smem();   // staged outputs and the block, before what the copies read and write there
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh->out_done[n & 1]);
          if (to_tm) tc_wait_st();
          continue;
        }
#pragma unroll 1
        for (int c = 0; c < L::CHUNKS; ++c, ++unit) {
          const int ch = team * L::CHUNKS + c;             // chunk of the tile
          const int y = ti * BM + quad * 32, x0 = tj * BN + ch * CHUNK;
          const int b = (int)(unit & 1);
          const uint32_t boff = (uint32_t)b * XBUF;
          // both blocks' earlier stores have been read; the next unit of the same product is fetched now
          if (lane == 0) bulk_wait_read<0>();
          if (mode != kG1) {
            if (!have && !from_tm) fetch(mode, k, tile, c, b);
            const bool more = c + 1 < L::CHUNKS ? !from_tm : j + 1 < mine && (raw || j + 1 >= (mode == kG3 ? a.nx : a.na));
            if (more) fetch(mode, k, c + 1 < L::CHUNKS ? tile : sh->tiles[sym ? 0 : 1][j + 1], c + 1 < L::CHUNKS ? c + 1 : 0, b ^ 1);
            have = more;
          }
          __syncwarp();
          if (c == 0) {
            wait_or_abort(&sh->acc_full[ab], (two_acc ? n >> 1 : n) & 1, abort_flag);
            tc_fence_after();
          }
          uint32_t acc[16];
          tc_ld16_issue(tm_lane + ACC_COL + ab * BN + ch * CHUNK, acc);
          float x[16];
          if (from_tm) {
            tc_ld16(state + ch * CHUNK, x);
          } else if (mode != kG1) {
            wait_or_abort(xfull + b * 8, (xph >> b) & 1, abort_flag);
            xph ^= 1u << b;
            if (xposed) {
#pragma unroll
              for (int i = 0; i < 16; ++i) x[i] = lds_f1(area + boff + i * 128 + lane * 4);
              __syncwarp();  // every lane has its row before the result rows are staged over the block
            } else {
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float4 f = lds_f4((row_addr + boff) ^ (i << 4));
                x[4 * i] = f.x; x[4 * i + 1] = f.y; x[4 * i + 2] = f.z; x[4 * i + 3] = f.w;
              }
            }
            if (raw) {
              const float tau = sh->clip[warp & (EPI_WARPS - 1)][0], inv = sh->clip[warp & (EPI_WARPS - 1)][1];
#pragma unroll
              for (int i = 0; i < 16; ++i) x[i] = __fmul_rn(fminf(fmaxf(x[i], -tau), tau), inv);
            }
          }
          tc_wait_ld16(acc);
          if (c == L::CHUNKS - 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->acc_empty[ab]);
          }
          float v[16];
          if (mode == kG1) {
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = __fmul_rn(__uint_as_float(acc[i]), scale);
          } else {
            const uint64_t b2 = pack2(beta, beta), g2 = pack2(gamma, gamma);
#pragma unroll
            for (int i = 0; i < 16; i += 2) {
              const uint64_t ac2 = pack2(__uint_as_float(acc[i]), __uint_as_float(acc[i + 1]));
              const uint64_t bx = mul2(b2, pack2(x[i], x[i + 1]));
              if (fused) {
                unpack2(fma2(ac2, g2, bx), v[i], v[i + 1]);
              } else {
                float t0, t1, u0, u1;
                unpack2(bx, t0, t1);
                unpack2(mul2(ac2, g2), u0, u1);
                v[i] = __fadd_rn(t0, u0);
                v[i + 1] = __fadd_rn(t1, u1);
              }
            }
          }
          const bool round = a.bf16 && !last && mode != kG2;  // stored rounded to BF16
          if (to_tm) store_state(state + ch * CHUNK, v, round);
          bool send = mode == kG1 && (!to_tm || a.keep);
          if (mode == kG3) {
            // the caller's matrix has no padding; X of a tall matrix lies in the workspace and has
            send = !to_tm && ((y < pr.s0 && x0 < pr.l0) || (pr.tall && !out_t));
            if (last && a.update && pr.W) {
              const bool in = y + lane < pr.s0 && x0 < pr.l0;
              if (pr.tall) {
                if (in) chain_update_tall(pr.W + (int64_t)x0 * pr.s0 + y + lane, pr.s0, v, a.upd_decay, a.upd_step);
              } else if (in) {
                uint4* w = reinterpret_cast<uint4*>(pr.W + ((int64_t)y + lane) * pr.l0 + x0);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  uint4 o = w[h];
                  uint32_t* e = &o.x;
#pragma unroll
                  for (int i = 0; i < 4; ++i)
                    e[i] = cvt_bf16x2(param_update_value(bf16_lo(e[i]), v[8 * h + 2 * i], a.upd_decay, a.upd_step),
                                      param_update_value(bf16_hi(e[i]), v[8 * h + 2 * i + 1], a.upd_decay, a.upd_step));
                  w[h] = o;
                }
              }
              send = send && !a.no_out;
            }
          }
          // ---- stage the block (for the TMA store and for the pass down the columns) and send it off
          if (out_t && !a.keep) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              asm volatile("st.shared.f32 [%0], %1;" ::"r"(area + boff + i * 128 + lane * 4), "f"(v[i]) : "memory");
          } else if (send || mirror) {
#pragma unroll
            for (int i = 0; i < 4; ++i) sts_f4((row_addr + boff) ^ (i << 4), v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
          }
          // The FP32 block leaves by TMA; only this warp reads it back.  With several units per product (BN = 128) it
          // is sent now, so that its buffer is free in time; else after the outputs that other blocks wait for.
          auto send_block = [&]() {
            if (mode == kG1) tma_store_s(&pr.tm_A, x0, y, area + boff);
            else if (!out_t || a.keep) tma_store_s(&pr.tm_X, x0, y, area + boff);
            else tma_store_s(&pr.tm_outT, y, x0, area + boff);
            bulk_commit();
          };
          const bool early = BN == 128 && !round;
          if (send && early) fence_proxy_async_smem();
          __syncwarp();
          if (send && early && lane == 0) send_block();
          uint32_t rounded[8];   // what is stored rounded to BF16 takes the block's place after the pass down the columns
          if (round && send) {
#pragma unroll
            for (int i = 0; i < 8; ++i) rounded[i] = cvt_bf16x2(v[2 * i], v[2 * i + 1]);
          }
          if (do_q) {
            uint32_t lo, hi;
            float bmax;
            uint32_t sb;
            if (PF) sb = quantize_block16_opts_p2<false>(v, a.q, inv_sg, lo, hi, bmax, signs);
            else sb = quantize_block16_p2(v, inv_sg, lo, hi, bmax);
            amax = fmaxf(amax, bmax);
            // the stores of the tile two back have read the staging area
            if (c == 0) wait_or_abort(&sh->out_free[n & 1], ((n >> 1) & 1) ^ 1, abort_flag);
            sts_u2(os + (ch >> 2) * 4096 + row * 32 + (((ch & 3) * 8) ^ ((lane & 4) << 2)), lo, hi);
            sts_b(os + L::RQ + L::CQ + (ch >> 2) * 512 + lane * 16 + quad * 4 + (ch & 3), sb);
            if (mirror) {
              // the block again, down the columns (into the registers of the row pass: both at once would not fit)
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const uint32_t at = (col_base + boff) | (col_lane ^ (uint32_t)(i << 6 | ((i >> 1) & 3) << 4));
                v[i] = lds_f1(at);
                v[i + 8] = lds_f1(at + 512);
              }
            }
            if (round && send) {
              __syncwarp();
#pragma unroll
              for (int i = 0; i < 4; ++i)
                sts_f4((row_addr + boff) ^ (i << 4), bf16_lo(rounded[2 * i]), bf16_hi(rounded[2 * i]), bf16_lo(rounded[2 * i + 1]),
                       bf16_hi(rounded[2 * i + 1]));
            }
            if (mirror) {
              if (PF) {
                // the transform and the error sums need the block in row order
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                  const float c0 = v[i], c1 = v[i + 1];
                  v[i] = g ? c1 : c0;
                  v[i + 1] = g ? c0 : c1;
                }
              }
              if (PF) sb = quantize_block16_opts_p2<false>(v, a.q, inv_sg, lo, hi, bmax, signs);
              else sb = quantize_block16_p2(v, inv_sg, lo, hi, bmax);
              if (!PF && g) { lo = swap_nibbles(lo); hi = swap_nibbles(hi); }   // back into row order
              const int col = ch * CHUNK + cq;
              sts_u2(os + L::RQ + col * 64 + ((quad ^ ((col >> 1) & 3)) << 4) + g * 8, lo, hi);
              sts_b(os + L::RQ + L::CQ + L::RSF + (quad >> 1) * (BN * 4) + (col & 31) * (BN / 8) + (col >> 5) * 4 + (quad & 1) * 2 + g, sb);
            }
          }
          if (to_tm) tc_wait_st();
          // The fence orders this lane's reads and writes of shared memory before what the copies (another proxy)
          // read and write there.
          fence_proxy_async_smem();
          if (c == L::CHUNKS - 1 && do_q) {
            if (mode != kG2) {
              const int slot = mode == kG1 ? a.ix.amax_A0 + k : a.ix.amax_X0 + k + 1;
              const uint32_t wm = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));
              if (lane == 0) atomicMax(&sh->amax[n & 1][slot & 3], wm);
              fence_proxy_async_smem();
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->out_done[n & 1]);
          }
          __syncwarp();
          if (send && !early && lane == 0) send_block();
        }
      }
      // What the next product reads from memory: blocks this warp has stored itself (A in G1, X in the G3 before), so every store
      // of the warp has to have arrived - also when the product begins with resident tiles and fetches later.  A product
      // that begins beyond them has its first block fetched here.  (a.keep: resident tiles of A are stored in every
      // iteration, to the same place.)
      if (mine > 0) for (int np = pi + 1; np < end && np <= pi + 3; ++np) {
        const int nk = np / 3, nmode = np - 3 * nk + kG1;
        const int nmine = nmode != kG3 ? my_sym : my_full;
        if (nmine == 0) continue;
        const int in_tm = nmode == kG1 ? nmine : nmode == kG2 ? a.na : nk > 0 ? a.nx : 0;
        if (nmine > in_tm || a.keep) {
          if (lane == 0) bulk_wait_all<0>();
          if (in_tm == 0) {
            fetch(nmode, nk, sh->tiles[nmode != kG3 ? 0 : 1][0], 0, (int)(unit & 1));
            have = true;
          }
        }
        break;
      }
    }
    if (lane == 0) bulk_wait_all<0>();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == W_MMA) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
  if (threadIdx.x == 0 && sh->abort_flag) report_timeout(a.status);
}

// The blocks wait on one another, so all have to be resident: a cooperative launch - or, up to kChainCluster blocks, a single
// cluster, which is an ordinary launch whose set-up overlaps with the prologue (a power of two of blocks, some without a tile): 256 x 512
// 77.2 -> 74.6 us, with options 100.2 -> 97.7.  A cooperative launch takes any SMs that are free, a cluster those of one GPC, so beside other work
// it may start later, or finish sooner.  Two of the caller's streams, time per call of the second, cooperative / cluster: 512 x 512 beside 1024 x
// 1024 146 / 163 us, beside 640 x 1024 93 / 96, beside 2048 x 2048 266 / 264; 256 x 512 beside 1024 x 1024 88 / 79, beside 2048 x 2048 262 / 169.
// The second stream of FP4_FLAG_OVERLAP_GROUPS: eight groups of one to 16 tiles 353 / 326, two larger and four such groups 322 / 313, 4096 x
// 4096 and six of them 921 / 909, two 1536 wide and two such groups 517 / 520.
constexpr int kChainCluster = 16;
int g_cluster_blocks[64];   // per device: blocks of the largest such cluster it holds, or 0 (set once, before the device's first launch)
template <int BN, bool PF, bool SYM = false>
cudaError_t launch_one(const ChainPack& pack, const ChainLaunch& a, int grid, bool whole_device, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(NTHREADS); cfg.dynamicSmemBytes = ChainLay<BN>::SMEM; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (whole_device && grid <= g_cluster_blocks[dev]) {
    int blocks = 1;
    while (blocks < grid) blocks *= 2;
    cfg.gridDim = dim3((unsigned)blocks);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)blocks; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
    cfg.numAttrs = 2;
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.numAttrs = 1;
  }
  count_launches(1);
  if (a.count == 1) return cudaLaunchKernelEx(&cfg, k_chain<BN, PF, SYM, 1>, ChainPackOf<1>{{pack.p[0]}}, a);
  return cudaLaunchKernelEx(&cfg, k_chain<BN, PF, SYM, kChainMax>, pack, a);
}

int64_t sym_tiles(int64_t s, int bn) {
  int64_t n = 0;
  for (int64_t r = 0; r < s / BM; ++r) n += (s - r * BM) / bn;
  return n;
}
int64_t rounds(int64_t tiles, int sms) { return (tiles + sms - 1) / sms; }
}  // namespace

template <int BN, bool PF, bool SYM, int MAX>
static cudaError_t chain_set_attribute(int dev) {
  const auto kernel = k_chain<BN, PF, SYM, MAX>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ChainLay<BN>::SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  // blocks of the largest cluster that the device holds, of any of the kernels
  int blocks = kChainCluster;
  for (; blocks >= 8; blocks /= 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3(NTHREADS); cfg.dynamicSmemBytes = ChainLay<BN>::SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)blocks; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters > 0) break;
    cudaGetLastError();
  }
  if (blocks < 8) blocks = 0;
  if (blocks < g_cluster_blocks[dev]) g_cluster_blocks[dev] = blocks;
  return cudaSuccess;
}
template <int BN, bool PF, bool SYM>
static cudaError_t chain_set_attribute(int dev) {
  const cudaError_t e = chain_set_attribute<BN, PF, SYM, 1>(dev);
  return e != cudaSuccess ? e : chain_set_attribute<BN, PF, SYM, kChainMax>(dev);
}
cudaError_t chain_set_attributes() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  g_cluster_blocks[dev] = kChainCluster;
  if ((e = chain_set_attribute<64, false, false>(dev))) return e;
  if ((e = chain_set_attribute<64, true, false>(dev))) return e;
  if ((e = chain_set_attribute<128, false, true>(dev))) return e;
  if ((e = chain_set_attribute<128, true, true>(dev))) return e;
  if ((e = chain_set_attribute<128, false, false>(dev))) return e;
  return chain_set_attribute<128, true, false>(dev);
}

// Which tiles stay in the tensor memory, when every block takes up to `full` tiles of G3 and `sym` of a symmetric product: A
// first, which serves two products of an iteration (2048 x 2048 201 us, X first 215).  One accumulator instead of two where that lets
// more of them stay: a tile's accumulator is read at the very start of its epilogue (201 us, with two accumulators 211).
struct Residents { int nacc, na, nx; };
static Residents residents(int bn, int64_t full, int64_t sym) {
  const int nacc = full + sym <= resident_slots(bn, 2) ? 2 : 1;
  const int64_t slots = resident_slots(bn, nacc), na = sym < slots ? sym : slots;
  return {nacc, (int)na, (int)(full < slots - na ? full : slots - na)};
}

// Estimated times in us.  A product costs a dependency round trip and a block's tiles, each an epilogue - short where its FP32 values
// stay in the tensor memory, long where they move through memory - or a main loop, whichever is longer.  The constants here
// and of the CTA-pair kernel's estimate beside the caller are fitted to the times of all routes and both widths at 213 shapes and
// groups (short sides 128 to 2304, long sides to 32768, 1 to 14 matrices, plain and with the quantiser options): choosing by them
// loses 0.1 % on average against always knowing the fastest, 3.5 % at worst, and 0.7 % (9 %) at 100 others drawn at random.  Calls of mixed
// shapes, which they were not fitted to: at 119 drawn ones (2 to 4 shapes, up to 14 matrices) route and merging lose 0.4 % (14 %).
struct TileUs {
  double product, resident, memory;
  TileUs(int bn, bool opts)
      : product(bn == 64 ? 4.0 : 5.0), resident((bn == 64 ? 0.65 : 1.0) * (opts ? 1.45 : 1.0)),
        memory((bn == 64 ? 1.7 : 4.75) * (opts ? 1.45 : 1.0)) {}
  static double k1(int64_t l) { return 0.22 * (double)((l + 255) / 256); }   // main loop of G1
  static double k2(int64_t s) { return 0.26 * (double)((s + 255) / 256); }   // of G2 and G3
};
// Mean times of a tile of one product, resident or not
struct MeanTile {
  double resident = 0.0, memory = 0.0;
  void add(double share, const TileUs& t, double k) {
    resident += share * (t.resident > k ? t.resident : k);
    memory += share * (t.memory > k ? t.memory : k);
  }
  double tiles(int64_t n, int in_tm) const { return in_tm * resident + (double)(n - in_tm) * memory; }
};
// one iteration of a single launch with tiles of bn columns; 0 when a block would take more tiles than its list holds
static double width_us(int bn, const WorkShape* w, int count, bool opts, int sms) {
  int64_t sym = 0, full = 0;
  for (int j = 0; j < count; ++j) { sym += sym_tiles(w[j].s, bn); full += w[j].s / BM * (w[j].l / bn); }
  const int64_t rs = rounds(sym, sms), rf = rounds(full, sms);
  if (rf > kChainTiles) return 0.0;
  const Residents r = residents(bn, rf, rs);
  const TileUs t(bn, opts);
  MeanTile g1, g2, g3;
  for (int j = 0; j < count; ++j) {
    const double share = (double)sym_tiles(w[j].s, bn) / (double)sym;
    g1.add(share, t, TileUs::k1(w[j].l));
    g2.add(share, t, TileUs::k2(w[j].s));
    g3.add((double)(w[j].s / BM * (w[j].l / bn)) / (double)full, t, TileUs::k2(w[j].s));
  }
  return 3 * t.product + g1.tiles(rs, r.na) + g2.tiles(rs, r.na) + g3.tiles(rf, r.nx);
}
// The width of a single launch's tiles.  Measured, 5 iterations, 64 / 128 columns: 256 x 512 83 / 101 us (now 72 as one cluster), 1024 x 4096 159 / 185 (with the
// quantiser options 200 / 243), 8 x 768 x 768 155 / 179, 1152 x 8192 290 / 324, 1536 x 1536 148 / 139, 1536 x 2816 196 / 188,
// 2048 x 2048 210 / 196 (250 / 249).
static bool narrow_tiles(const WorkShape* w, int count, bool opts, int sms) {
  const double narrow = width_us(64, w, count, opts, sms), wide = width_us(128, w, count, opts, sms);
  return narrow > 0.0 && narrow <= wide;
}
double chain_iteration_us(const WorkShape* w, int count, bool opts, int sms) {
  return width_us(narrow_tiles(w, count, opts, sms) ? 64 : 128, w, count, opts, sms);
}
// G1 and G2 of an iteration in a launch of their own, where every SM has at most one tile (else 0)
double chain_symmetric_us(const WorkShape* w, int count, bool opts, int sms) {
  int64_t sym = 0, s = 0, l = 0;
  for (int j = 0; j < count; ++j) {
    sym += sym_tiles(w[j].s, 128);
    s = w[j].s > s ? w[j].s : s;
    l = w[j].l > l ? w[j].l : l;
  }
  if (sym > sms) return 0.0;
  const TileUs t(128, opts);
  const double k1 = TileUs::k1(l), k2 = TileUs::k2(s);
  return 12.5 + (t.resident > k1 ? t.resident : k1) + (t.resident > k2 ? t.resident : k2);
}

// Places of the matrices in the launch's tile lists
static void place_tiles(ChainPack& pack, ChainLaunch& a, int bn) {
  a.sym_tiles = a.full_tiles = 0;
  for (int j = 0; j < a.count; ++j) {
    ChainProblem& pr = pack.p[j];
    pr.nsym = (int)sym_tiles(pr.s, bn);
    pr.first_sym = a.sym_tiles;
    pr.first_full = a.full_tiles;
    a.sym_tiles += pr.nsym;
    a.full_tiles += pr.s / BM * (pr.l / bn);
  }
}

cudaError_t launch_chain(ChainPack& pack, const ChainLaunch& launch, int sms, bool whole_device, cudaStream_t st) {
  if (launch.count < 1 || launch.count > kChainMax || launch.steps < 1) return cudaErrorInvalidValue;
  ChainLaunch a = launch;
  const bool pf = a.q.rht || a.q.four_six;
  WorkShape w[kChainMax];
  for (int j = 0; j < a.count; ++j) w[j] = {pack.p[j].s, pack.p[j].l};
  const bool narrow = narrow_tiles(w, a.count, pf, sms);
  const int bn = narrow ? 64 : 128;
  place_tiles(pack, a, bn);
  const int grid = a.full_tiles < sms ? a.full_tiles : sms;
  const Residents r = residents(bn, rounds(a.full_tiles, grid), rounds(a.sym_tiles, grid));
  a.nacc = r.nacc; a.na = r.na; a.nx = r.nx;
  if (narrow) return pf ? launch_one<64, true>(pack, a, grid, whole_device, st) : launch_one<64, false>(pack, a, grid, whole_device, st);
  return pf ? launch_one<128, true>(pack, a, grid, whole_device, st) : launch_one<128, false>(pack, a, grid, whole_device, st);
}

// G1 and G2 of iteration `step` in one launch with a 128 x 128 tile per SM.
cudaError_t launch_chain_symmetric(ChainPack& pack, const ChainLaunch& launch, int step, int sms, bool whole_device, cudaStream_t st) {
  if (launch.count < 1 || launch.count > kChainMax || launch.steps < 1) return cudaErrorInvalidValue;
  ChainLaunch a = launch;
  place_tiles(pack, a, 128);
  a.first = 3 * step; a.end = a.first + 2;
  if (a.sym_tiles > sms) return cudaErrorInvalidValue;
  const int grid = a.sym_tiles;
  const Residents r = residents(128, 0, 1);
  a.nacc = r.nacc; a.na = r.na; a.nx = r.nx;
  return a.q.rht || a.q.four_six ? launch_one<128, true, true>(pack, a, grid, whole_device, st) : launch_one<128, false, true>(pack, a, grid, whole_device, st);
}

}  // namespace fp4
