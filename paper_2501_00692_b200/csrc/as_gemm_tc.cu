// bf16 tensor-core contractions for sm_100a, by CTA pairs (tcgen05 cta_group::2): TMA (cp.async.bulk.tensor, 128-byte swizzle)
// feeds a shared-memory ring in each CTA of a pair, one elected thread of the pair issues tcgen05.mma into both CTAs' TMEM
// accumulators, sixteen warps per CTA drain them with tcgen05.ld, apply the fused epilogue into a shared-memory staging tile
// and hand that tile to TMA (bulk tensor store, or bulk tensor reduce-add for the split-K weight gradients), so that global
// memory only sees whole rows of 128 bytes.  One kernel template covers the three token-dimension contractions of the layer:
//   PROJ : [Delta | B | C] = X Wcat^T              (A K-major, B K-major;  softplus+bias epilogue)
//   DW   : dWcat^T = X^T Gcat  over all tokens     (A MN-major, B MN-major; split-K, fp32 reduction)
//   DX   : dx = dx_dir + Gcat Wcat                 (A K-major, B MN-major; add + bf16 store)
// with Wcat = [W_delta; W_B; W_C] ([P+32, P]) and Gcat = [du | dB | dC] ([tokens, P+32]), both bf16.
//
// Bound: the path between L2 and the SM, 128 bytes in some 2.4 cycles whatever moves (operands, dx_dir, results).  A single CTA
// (128 x 256) has to fill 48 KB per 64-deep block for 512 cycles of MMA; in a pair (256 x 256) each CTA holds its own 128 rows
// of A and half of B, 32 KB.  The rows of A a pair needs next are sent for into L2 a tile ahead (131,072 x 768, projections: 184 us
// without, 172 with).  At large K the sustained tensor rate (power) bounds it.  Measured, us, single CTAs of 128 x 256 with the
// issuing loops in lane-0 branches before: 131,072 x 768 projections 200 -> 172, dW 130 -> 124, dx 158 -> 145; 262,144 x 2,048
// 1,937 -> 1,600, 1,690 -> 1,600, 1,758 -> 1,560; 40,000 x 512 54 -> 43, 27 -> 30, 33 -> 33; 1,024 x 512 14.6 -> 9.8, 9.1 -> 8.9,
// 10.4 -> 9.1.  Slower: stores turned around in shared memory and made by the warps instead of TMA (193 against 178, 155
// against 145).
// Widths that are not a multiple of 32 take the fp32-accurate softplus: a deep bf16 stack turns rounding differences of one
// layer's Delta into differences of some per cent of its outputs, and these widths never had the shorter one.
// Widths that are not a multiple of 32 keep all 24 bits of dB and dC: Gcat then ends in three such pairs (the fp32 sums
// split into three bf16 terms, which is exact) and the Wcat of the input gradient repeats W_B and W_C three times
// (Plan.gsplit), so the contraction of the split equals the contraction of the fp32 values.
// No load is multicast.  Every mbarrier wait is bounded; on timeout the kernel records AS_ERR_TIMEOUT in the status block,
// stops issuing work, gives the copies in flight one more bounded wait, frees its TMEM and returns.
#include <cuda.h>

#include <type_traits>

#include "as_tc.cuh"

namespace as {
namespace {

constexpr int BM = 256, BK = 64, UK = 16;                 // rows of a pair's tile; depth of a block, of one MMA
constexpr int MAXN = 256;                                 // widest tile
constexpr int EPI_WARPS = 16, NTHREADS = 64 + 32 * EPI_WARPS;
constexpr int A_BYTES = BM / 2 * BK * 2, B_BYTES = MAXN / 2 * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;   // per CTA
constexpr int STAGES = 5;
constexpr int STG_BYTES = 32 * 128;                       // staging tile of one epilogue warp: 32 rows of 128 bytes
constexpr int TMEM_COLS = 512;                            // two accumulators
constexpr int SMEM_DYN = STAGES * STAGE_BYTES + 1024 + EPI_WARPS * STG_BYTES;   // + alignment slack + staging

// one contraction of a launch
struct Job {
  int64_t M;            // output rows per layer (PROJ, DX: tokens; DW: P, the columns of X)
  int N;                // output columns (PROJ: P + 32; DX: P; DW: columns of Gcat)
  int mt;               // 256-row tiles per layer
  int nt, nbase, nrem;  // column tiles: nbase units of columns each, one more in the first nrem
  int kblocks;          // BK-blocks of the contraction
  int splitk, kper;     // DW: splits of the contraction, blocks per split
  int ntiles;           // of all layers
};
struct TcArgs {
  Job job[2];           // PROJ: the first; gradients: DW, then DX (no tiles where dx is not wanted)
  int P;                // d_model
  int direct;           // W_delta, W_B, W_C are read where they lie, no Wcat: rows past P in pieces of 16 (P % 16 == 0)
  const float* bias;    // PROJ: b_delta [layers, P]
  float* bc;            // PROJ: [B | C] rows, for the plain stores where P is not a multiple of 32
  int* status;
  ZeroList zero;        // PROJ: regions to clear for the later kernels, where the call has no kernel before this one; the
                        // status word is among them, which is why the CTAs report through bytes of their own
};
// tensor maps of a launch
enum { PM_A, PM_B, PM_B1, PM_DELTA, PM_BC, PM_WB, PM_WC, PM_N };                                    // PROJ
enum { GM_X, GM_G, GM_DW, GM_DB, GM_DC, GM_GK, GM_W, GM_DX, GM_DIR, GM_W1, GM_WB, GM_WC, GM_N };    // gradients (DW, then DX)
template <bool GRAD> struct TcMaps { CUtensorMap m[GRAD ? (int)GM_N : (int)PM_N]; };
// columns of a tile come in units: 32 (one chunk of fp32 output), for the bf16 output of DX 64
__host__ __device__ constexpr int unit(bool dx) { return dx ? 64 : 32; }

struct Tile { int64_t m0; int n0, w, kb0, nkb, lay; bool dx; };   // first row, first column, columns, blocks, layer, contraction

// ---- the pair: addresses in, and signals to, the leader (rank 0) ----
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t leader_addr(const void* p) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
  return r;
}
__device__ __forceinline__ void arrive_at(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ void pair_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// into this CTA's shared memory; the bytes are counted at the leader's barrier
__device__ __forceinline__ void pair_load(void* dst, const CUtensorMap* tm, int c0, int c1, int c2, uint32_t leader_bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_u32(dst)), "l"(tm), "r"(c0), "r"(c1), "r"(c2), "r"(leader_bar) : "memory");
}
__device__ __forceinline__ void prefetch_l2(const CUtensorMap* tm, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(tm), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void pair_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void pair_commit(uint64_t* bar) {   // arrives at this barrier of both CTAs
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
// byte offset of 16-byte piece q of row r in a [rows][128 B] tile under the 128-byte swizzle
__device__ __forceinline__ uint32_t swz128(int r, int q) { return (uint32_t)(r * 128 + ((q ^ (r & 7)) << 4)); }

// Persistent, warp-specialised; pair p walks tiles t = p, + pairs, ...  In each CTA
//   warp 0 (elected lane): TMA producer over a STAGES-deep ring that runs on across tiles: the CTA's 128 rows of A, its half of B
//   warp 1 (elected lane, leader only): tcgen05.mma issuer; the accumulator alternates between two 256-column TMEM buffers
//   warps 2..17      : epilogue (four warps per TMEM lane quarter, each taking every fourth chunk of columns); they read a
//                      tile into registers and hand the buffer back before they work on it
// A full barrier of the leader counts the bytes of both CTAs; the MMAs' commits free the stage in both.
// Tile order: n fastest, then m, then the K split, so concurrently running pairs share A rows (DW: tokens) through L2.
// GRAD: the gradient contractions, one or both in a launch: DW's tiles (few and long) first, DX's fill up behind them.
// SP: softplus of the projections; SP_FINE also is the form for a P that is not a multiple of 32.
template <bool GRAD, int SP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NTHREADS, 1)
gemm_tc_kernel(const __grid_constant__ TcMaps<GRAD> maps, const __grid_constant__ TcArgs a) {
  constexpr bool OFF = SP == SP_FINE;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[STAGES];       // leader's: both CTAs' copies of the stage have landed
  __shared__ __align__(8) uint64_t empty_bar[STAGES];      // the MMAs have read the stage
  __shared__ __align__(8) uint64_t tmem_full_bar[2];       // the accumulator is complete
  __shared__ __align__(8) uint64_t tmem_empty_bar[2];      // leader's: the epilogue warps of both CTAs have read it
  __shared__ __align__(8) uint64_t ld_bar[EPI_WARPS];      // DX: the dx_dir tile has landed in the staging buffer
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;

  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();
  const int pair = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;
  volatile int* abortp = &abort_s;
  uint8_t* const cta_bytes = reinterpret_cast<uint8_t*>(a.status) + STATUS_CTA;   // PROJ: where its CTAs report

  // nothing up to pdl_wait() touches global memory.  The allocation cannot block: this CTA has its SM's shared memory to itself, and
  // the kernels of the library that hold TMEM all use some.
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&tmem_full_bar[b], 1); mbar_init(&tmem_empty_bar[b], 2 * EPI_WARPS); }
    for (int w2 = 0; w2 < EPI_WARPS; ++w2) mbar_init(&ld_bar[w2], 1);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
#pragma unroll
    for (const CUtensorMap& m : maps.m) prefetch_map(&m);
  }
  if (warp == 1) {   // TMEM allocation, by both CTAs of the pair
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "n"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  pair_sync();   // the peer's barriers are initialised, its TMEM is allocated
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = tmem_base_s;
  pdl_wait();
  if (!GRAD && a.zero.n > 0) {
    static_assert(NTHREADS >= STATUS_CTAS, "one CTA alone clears all bytes");
    const unsigned i = blockIdx.x + gridDim.x * threadIdx.x;   // this CTA's byte, and its share of those without a CTA
    if (i < STATUS_CTAS) cta_bytes[i] = 0;
    clear_regions(a.zero, (int64_t)blockIdx.x * NTHREADS + threadIdx.x, (int64_t)gridDim.x * NTHREADS);
  }

  const int ntiles = a.job[0].ntiles + (GRAD ? a.job[1].ntiles : 0);
  auto decode = [&](int t) {
    Tile q;
    q.dx = GRAD && t >= a.job[0].ntiles;
    if (q.dx) t -= a.job[0].ntiles;
    const Job& j = a.job[q.dx ? 1 : 0];
    const int in = t % j.nt;
    t /= j.nt;
    const int im = t % j.mt;
    t /= j.mt;
    q.n0 = unit(q.dx) * (in * j.nbase + min(in, j.nrem));
    q.w = unit(q.dx) * (j.nbase + (in < j.nrem ? 1 : 0));
    q.m0 = (int64_t)im * BM;
    q.kb0 = 0; q.nkb = j.kblocks;
    if (GRAD && !q.dx) {
      q.kb0 = t % j.splitk * j.kper;
      q.nkb = min(j.kblocks - q.kb0, j.kper);
      t /= j.splitk;
    }
    q.lay = t;
    return q;
  };

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    int it = 0;
    bool ok = true;
    // one tile; the contraction is a compile-time choice (which maps an instruction names at run time cost 250 cycles a block)
    auto load_tile = [&](const Tile& q, int t, auto dw_c) {
      constexpr bool DW = decltype(dw_c)::value;
      const CUtensorMap& tmA = maps.m[GRAD ? (DW ? (int)GM_X : (int)GM_GK) : (int)PM_A];
      const CUtensorMap& tmB = maps.m[GRAD ? (DW ? (int)GM_G : (int)GM_W) : (int)PM_B];
      const int half = q.w / 2, m0 = (int)q.m0 + rank * (BM / 2), n0 = q.n0 + rank * half;
      const int nq = (half + 63) / 64;   // MN-major B: 64-column pieces of this CTA's half
      const uint32_t bytes = 2u * (uint32_t)(A_BYTES + (GRAD ? nq * 64 * BK * 2 : half * BK * 2));   // of both CTAs
      // PROJ, DX: the pair's next tile, if it is the first of its rows: its rows of A go to L2 while this tile is loaded (DW: blocks
      // ahead of the ring slowed it down, 128 against 169 us at 131,072 x 768)
      Tile ahead = q;
      bool pre = false;
      if (!DW && t + pairs < ntiles) { ahead = decode(t + pairs); pre = ahead.n0 == 0; }
      const int ma = (int)ahead.m0 + rank * (BM / 2);
      for (int i = 0; i < q.nkb; ++i, ++it) {
        const int s = it % STAGES, round = it / STAGES;
        if (round > 0 && !mbar_wait(&empty_bar[s], (round - 1) & 1, abortp)) { ok = false; break; }
        uint8_t* sa = smem + s * STAGE_BYTES;
        uint8_t* sb = sa + A_BYTES;
        const int k = (q.kb0 + i) * BK;
        if (elect_one()) {
          const uint32_t bar = leader_addr(&full_bar[s]);
          if (rank == 0) mbar_expect_tx(&full_bar[s], bytes);
          if (pre) prefetch_l2(&tmA, k, ma, ahead.lay);
          if (!DW) {
            pair_load(sa, &tmA, k, m0, q.lay, bar);
          } else {
            pair_load(sa, &tmA, m0, k, q.lay, bar);
            pair_load(sa + A_BYTES / 2, &tmA, m0 + 64, k, q.lay, bar);
          }
          if (!GRAD) {   // the box has the narrow tiles' rows; a wide tile's last rows by a second one
            const int rows = unit(false) / 2 * a.job[0].nbase;
            if (a.direct && n0 + half > a.P) {
              for (int r = 0; r < half; r += 16) {   // rows of W_delta, W_B, W_C; past them the zero fill of the last
                const int e = n0 + r - a.P;
                const CUtensorMap& m = maps.m[GRAD ? 0 : e < 0 ? (int)PM_B1 : e == 0 ? (int)PM_WB : (int)PM_WC];
                pair_load(sb + r * (BK * 2), &m, k, e < 0 ? n0 + r : e < 32 ? 0 : 16, q.lay, bar);
              }
            } else {
              pair_load(sb, &tmB, k, n0, q.lay, bar);
              if (half > rows) pair_load(sb + rows * (BK * 2), &maps.m[PM_B1], k, n0 + rows, q.lay, bar);
            }
          } else if (!DW && a.direct && k + BK > a.P) {
            for (int r = 0; r < BK; r += 16) {
              const int e = k + r - a.P;   // the contraction of the split repeats W_B and W_C; past them the zero fill of the last
              const CUtensorMap& m = maps.m[!GRAD ? 0 : e < 0 ? (int)GM_W1 : (e & 16) == 0 ? (int)GM_WB : (int)GM_WC];
              const int row = e < 0 ? k + r : e < a.job[0].N - a.P ? 0 : NS;
              for (int j = 0; j < nq; ++j) pair_load(sb + j * (64 * BK * 2) + r * 128, &m, n0 + 64 * j, row, q.lay, bar);
            }
          } else {
            pair_load(sb, &tmB, n0, k, q.lay, bar);
            if (nq > 1) pair_load(sb + 64 * BK * 2, &tmB, n0 + 64, k, q.lay, bar);
          }
        }
        __syncwarp();
      }
    };
    for (int t = pair; t < ntiles && ok; t += pairs) {
      const Tile q = decode(t);
      if (GRAD && !q.dx) load_tile(q, t, std::true_type{});
      else load_tile(q, t, std::false_type{});
    }
    pdl_launch();
    if (!ok && lane == 0) {
      *abortp = 1;
      if (GRAD) atomicExch(a.status, AS_ERR_TIMEOUT);
      // the leader's barriers see the copies of both CTAs: one more bounded wait for those in flight
      if (rank == 0)
        for (int i = it > STAGES ? it - STAGES : 0; i < it; ++i) mbar_wait(&full_bar[i % STAGES], (i / STAGES) & 1);
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ---------------- MMA issuer ----------------
      int it = 0, ti = 0;
      bool ok = true;
      auto issue_tile = [&](const Tile& q, auto dw_c) {
        constexpr bool DW = decltype(dw_c)::value;   // A is MN-major
        const int ab = ti & 1, around = ti >> 1;
        if (around > 0 && !mbar_wait(&tmem_empty_bar[ab], (around - 1) & 1, abortp)) { ok = false; return; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc = tmem_base + (uint32_t)(ab * MAXN);
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(DW ? MAJ_MN : MAJ_K) << 15) |
                               ((uint32_t)(GRAD ? MAJ_MN : MAJ_K) << 16) | ((uint32_t)(q.w >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
        for (int i = 0; i < q.nkb; ++i, ++it) {
          const int s = it % STAGES, round = it / STAGES;
          if (!mbar_wait(&full_bar[s], round & 1, abortp)) { ok = false; return; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sa = smem_u32(smem + s * STAGE_BYTES);
          const uint32_t sb = sa + A_BYTES;
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < BK / UK; ++k) {
              const uint64_t ad = DW ? make_desc(sa + k * UK * 128, A_BYTES / 2, 1024) : make_desc(sa + k * UK * 2, 16, 1024);
              const uint64_t bd = GRAD ? make_desc(sb + k * UK * 128, 64 * BK * 2, 1024) : make_desc(sb + k * UK * 2, 16, 1024);
              pair_mma(acc, ad, bd, idesc, (i > 0 || k > 0) ? 1u : 0u);
            }
            pair_commit(&empty_bar[s]);   // frees the stage once these MMAs have read it
            if (i + 1 == q.nkb) pair_commit(&tmem_full_bar[ab]);   // accumulator of this tile complete
          }
          __syncwarp();
        }
      };
      for (int t = pair; t < ntiles && ok; t += pairs, ++ti) {
        const Tile q = decode(t);
        if (GRAD && !q.dx) issue_tile(q, std::true_type{});
        else issue_tile(q, std::false_type{});
      }
      if (!ok && lane == 0) { *abortp = 1; if (GRAD) atomicExch(a.status, AS_ERR_TIMEOUT); }
    }
  } else {
    // ---------------- epilogue warps ----------------
    // A warp owns TMEM lanes [32 quarter, 32 quarter + 32) = 32 output rows, one row per lane, and every fourth chunk of the
    // tile's columns.  A chunk (PROJ, DW: 32 columns; DX: 64) goes registers -> the warp's staging tile (rows of 128 bytes;
    // DW: the transpose, a row per column) -> TMA; lane 0 issues and tracks the bulk operations.  Rows and columns past the
    // output's extent are clipped by TMA.
    const int quarter = warp & 3, cw = (warp - 2) >> 2;   // the TMEM lane quarter this warp may read; its chunks cw, cw + 4
    uint8_t* buf = smem + STAGES * STAGE_BYTES + (warp - 2) * STG_BYTES;
    uint64_t* lbar = &ld_bar[warp - 2];
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    uint32_t ld_phase = 0;
    bool ok = true;
    // DX: dx_dir of the warp's chunk of a tile, requested as soon as the staging buffer is free; false if it has none
    auto request = [&](const Tile& q) {
      const int nb = q.n0 + 64 * cw, mrow = (int)q.m0 + rank * (BM / 2) + quarter * 32;
      if (!q.dx || 64 * cw >= q.w || nb >= a.job[1].N || mrow >= a.job[1].M) return false;
      if (lane == 0) {
        bulk_wait_read<0>();
        mbar_expect_tx(lbar, STG_BYTES);
        tma_load_3d(buf, &maps.m[GM_DIR], nb, mrow, q.lay, lbar);
      }
      return true;
    };
    bool has = GRAD && pair < ntiles && request(decode(pair));
    int ti = 0;
    for (int t = pair; t < ntiles; t += pairs, ++ti) {
      const Tile q = decode(t);
      const int ab = ti & 1;
      const Job& j = a.job[q.dx ? 1 : 0];
      const int mrow = (int)q.m0 + rank * (BM / 2) + quarter * 32;      // first output row of this warp
      if (!mbar_wait(&tmem_full_bar[ab], (ti >> 1) & 1, abortp)) { ok = false; break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t acc = lane_addr + (uint32_t)(ab * MAXN);
      // first and second 32 columns of the warp in this tile
      const int c0 = q.dx ? 64 * cw : 32 * cw, c1 = q.dx ? 64 * cw + 32 : 32 * cw + 128;
      const bool two = c1 < q.w;
      if (has && !mbar_wait(lbar, ld_phase, abortp)) { ok = false; break; }
      if (c0 >= q.w && lane == 0) arrive_at(leader_addr(&tmem_empty_bar[ab]));   // nothing for this warp in a narrow tile
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        if (h ? !two : c0 >= q.w) break;                  // warp-uniform
        const int c = h ? c1 : c0, nb = q.n0 + c;
        const bool last = h || !two, none = nb >= j.N || mrow >= j.M;
        if (!q.dx && !none) {
          if (lane == 0) bulk_wait_read<0>();             // the operation that last used the buffer has read it
          __syncwarp();
        }
#pragma unroll 1
        for (int g = 0; g < 2; ++g) {                     // 16 columns at a time
          uint32_t r[16];
          tmem_ld16(acc + c + 16 * g, r);
          if (last && g) {                                // the warp's last: hand the accumulator back to the issuer
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) arrive_at(leader_addr(&tmem_empty_bar[ab]));
          }
          if (none) continue;
          if (GRAD && q.dx) {
#pragma unroll
            for (int p = 0; p < 2; ++p) {
              uint4* pq = reinterpret_cast<uint4*>(buf + swz128(lane, 4 * h + 2 * g + p));
              const uint4 sv = *pq;
              const __nv_bfloat162* s2 = reinterpret_cast<const __nv_bfloat162*>(&sv);
              uint4 ov;
              __nv_bfloat162* o2 = reinterpret_cast<__nv_bfloat162*>(&ov);
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const float2 f = __bfloat1622float2(s2[e]);
                o2[e] = __floats2bfloat162_rn(f.x + __uint_as_float(r[8 * p + 2 * e]), f.y + __uint_as_float(r[8 * p + 2 * e + 1]));
              }
              *pq = ov;
            }
          } else if (GRAD) {
#pragma unroll
            for (int i = 0; i < 16; ++i) *reinterpret_cast<uint32_t*>(buf + (16 * g + i) * 128 + lane * 4) = r[i];
          } else {
            const int col = nb + 16 * g;
            const bool border = OFF && col + 16 > a.P;   // holds the border between Delta and [B | C], or lies behind it
            if (col < a.P || border) {
              const int64_t row = mrow + lane;
              const float* bias_l = a.bias + (int64_t)q.lay * a.P + col;
#pragma unroll
              for (int p = 0; p < 4; ++p) {
                // four columns: all inside one part (its border is a multiple of 8) or all outside
                if (!border || col + 4 * p < a.P) {
                  const f2x2 bv = split4(__ldg(reinterpret_cast<const float4*>(bias_l + 4 * p)));
                  float v[4];
                  upk(softplus2<SP>(add2(pk(__uint_as_float(r[4 * p]), __uint_as_float(r[4 * p + 1])), bv.x)), v[0], v[1]);
                  upk(softplus2<SP>(add2(pk(__uint_as_float(r[4 * p + 2]), __uint_as_float(r[4 * p + 3])), bv.y)), v[2], v[3]);
#pragma unroll
                  for (int e = 0; e < 4; ++e) r[4 * p + e] = __float_as_uint(v[e]);
                } else if (col + 4 * p < a.P + NBC && row < j.M) {
                  // where the border is no multiple of 32 a TMA store would have to start left of the [B | C] rows
                  *reinterpret_cast<uint4*>(a.bc + ((int64_t)q.lay * j.M + row) * NBC + col + 4 * p - a.P) =
                      make_uint4(r[4 * p], r[4 * p + 1], r[4 * p + 2], r[4 * p + 3]);
                }
              }
            }
#pragma unroll
            for (int p = 0; p < 4; ++p)
              *reinterpret_cast<uint4*>(buf + swz128(lane, 4 * g + p)) = make_uint4(r[4 * p], r[4 * p + 1], r[4 * p + 2], r[4 * p + 3]);
          }
        }
        if (none || q.dx) continue;
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (!GRAD) {
            if (nb < a.P) tma_store_3d(&maps.m[PM_DELTA], buf, nb, mrow, q.lay);                  // Delta, clipped at column P
            else if (!OFF) tma_store_3d(&maps.m[PM_BC], buf, nb - a.P, mrow, q.lay);              // [B | C]
          } else {
            // columns of Gcat: [0, P) dW_delta, then 16 dW_B and 16 dW_C (three such pairs with the split: their sums add up
            // in the output).  The rows of a chunk that lie past P are clipped from dW_delta and go out eight at a time:
            // eight columns never straddle two outputs.
            if (nb < a.P) tma_reduce_add_3d(&maps.m[GM_DW], buf, mrow, nb, q.lay);
            if (nb + 32 > a.P) {
#pragma unroll 1
              for (int i = 0; i < 32; i += 8) {
                const int e = nb + i - a.P;
                if (e >= 0 && nb + i < j.N) tma_reduce_add_3d(&maps.m[(e & 16) == 0 ? GM_DB : GM_DC], buf + i * 128, mrow, e & 15, q.lay);
              }
            }
          }
          bulk_commit();
        }
      }
      if (GRAD) {
        if (has) {
          ld_phase ^= 1;
          fence_async_smem();
          __syncwarp();
          if (lane == 0) { tma_store_3d(&maps.m[GM_DX], buf, q.n0 + c0, mrow, q.lay); bulk_commit(); }
        }
        has = t + pairs < ntiles && request(decode(t + pairs));
      }
    }
    if (lane == 0) {
      bulk_wait_read<0>();                     // staging tiles must outlive the bulk operations that read them
      if (!ok && has) mbar_wait(lbar, ld_phase);
    }
    if (!ok) { *abortp = 1; if (GRAD && lane == 0) atomicExch(a.status, AS_ERR_TIMEOUT); }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  pair_sync();   // nobody signals this CTA any more, both CTAs are done with TMEM
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(TMEM_COLS) : "memory");
  }
  // the projections report here and not where a role gives up: a choice of the place inside the roles cost a forward of
  // 2,048 x 512 3 us of 45
  if (!GRAD && threadIdx.x == 0 && *abortp) cta_bytes[blockIdx.x] = 1;
}

// ---- small helpers -------------------------------------------------------------------------------
// [dB | dC] fp32 sums -> the last bf16 columns of Gcat; eight values per thread (P and the row pitch are multiples of 8
// elements, so every access is 16-byte aligned).  SPLIT: as three bf16 terms, 32 columns each, that add up to the fp32 value.
template <int SPLIT>
__global__ void cvt_dbc_kernel(int64_t rows, int ldg, int P, const float* __restrict__ dbc, __nv_bfloat16* __restrict__ gcat) {
  pdl_begin();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // one group of 8 columns
  if (i >= rows * (NBC / 8)) return;
  const int64_t row = i / (NBC / 8);
  const int c = (int)(i % (NBC / 8)) * 8;
  const float4 a = __ldg(reinterpret_cast<const float4*>(dbc + row * NBC + c));
  const float4 b = __ldg(reinterpret_cast<const float4*>(dbc + row * NBC + c + 4));
  float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
  for (int t = 0; t < SPLIT; ++t) {
    uint4 o;
    __nv_bfloat162* o2 = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      o2[k] = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
      const float2 f = __bfloat1622float2(o2[k]);
      v[2 * k] -= f.x; v[2 * k + 1] -= f.y;
    }
    *reinterpret_cast<uint4*>(gcat + row * ldg + P + t * NBC + c) = o;
  }
}

// [layers, rows, cols] row-major, rows `ld` elements apart; box = {box_cols, box_rows, 1}.  Reads outside a layer give 0, writes
// are dropped.
int map3(CUtensorMap* tm, bool f32, CUtensorMapSwizzle swz, const void* base, int64_t layers, int64_t rows, int64_t cols, int64_t ld,
         int box_cols, int box_rows) {
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return 1;
  const cuuint64_t e = f32 ? 4 : 2;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)layers};
  cuuint64_t strides[2] = {(cuuint64_t)ld * e, (cuuint64_t)rows * (cuuint64_t)ld * e};
  cuuint32_t box[3] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(tm, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims,
             strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS ? 0 : 1;
}
int operand(CUtensorMap* tm, const void* base, int64_t layers, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  return map3(tm, false, CU_TENSOR_MAP_SWIZZLE_128B, base, layers, rows, cols, ld, BK, box_rows);
}
int output(CUtensorMap* tm, bool f32, CUtensorMapSwizzle swz, const void* base, int64_t layers, int64_t rows, int64_t cols, int box_cols,
           int box_rows) {
  return map3(tm, f32, swz, base, layers, rows, cols, cols, box_cols, box_rows);
}

int64_t cdiv(int64_t x, int64_t y) { return (x + y - 1) / y; }
int pair_count() { return sm_count() / 2 < STATUS_CTAS / 2 ? sm_count() / 2 : STATUS_CTAS / 2; }

// Tile widths and splits.  A block of 64 costs the longer of its MMAs, 2 w cycles, and the fill of its operands, 256 rows of A and w
// of B by two CTAs at 128 bytes in two cycles each: 256 + w.  An epilogue takes some EPI_CYCLES per round of four chunks, twice
// that for the reduce-adds of DW.  Of the widths from the widest tile down, and of DW's splits into one, two or three waves, the
// one with the least time is taken: long runs get an even cut of N into tiles of at most 256 columns, short ones tiles narrow
// enough that every pair has work (1,024 x 512, projections: 14.6 us at 208 columns, 9.8 at 32; 256 x 256: 12.8 and 9).
// Returns that time in cycles.
constexpr int64_t EPI_CYCLES = 1500;
enum { CUT_PROJ, CUT_DW, CUT_DX };
constexpr int64_t ONE_LAUNCH_BLOCKS = 400;   // see tc_gradients
int64_t cut_columns(int what, Job* j, int layers, int pairs) {
  const int u = unit(what == CUT_DX), units = (int)cdiv(j->N, u);
  const bool split = what == CUT_DW;
  j->mt = (int)cdiv(j->M, BM);
  int64_t best = -1, count = 0;
  for (int nt = (int)cdiv(units, MAXN / u); nt <= units; ++nt) {
    const int64_t w = cdiv(units, nt) * u, out = cdiv(w, 4 * u) * EPI_CYCLES * (split ? 2 : 1);
    const int64_t tiles = (int64_t)j->mt * nt * layers;
    for (int target = 1; target <= (split ? 3 : 1); ++target) {   // waves the splits aim at
      int64_t sk = split ? target * pairs / tiles : 1;
      if (sk > j->kblocks) sk = j->kblocks;
      if (sk < 1) sk = 1;
      const int64_t kper = cdiv(j->kblocks, sk), real = cdiv(j->kblocks, kper);
      // a wave costs its blocks, or its epilogue where that takes longer; the last epilogue is not hidden
      const int64_t blocks = kper * (256 + w), cost = cdiv(tiles * real, pairs) * (blocks > out ? blocks : out) + out;
      if (best < 0 || cost < best) {
        best = cost;
        j->nt = nt; j->nbase = units / nt; j->nrem = units % nt;
        j->splitk = (int)real; j->kper = (int)kper;
        count = tiles * real;
      }
    }
    if (tiles >= 4 * pairs) break;   // narrower tiles only cost fill from here on
  }
  j->ntiles = count > 0x3fffffff ? -1 : (int)count;
  return best;
}

template <bool GRAD, int SP>
int launch_tc(const TcMaps<GRAD>& maps, const TcArgs& a, cudaStream_t st) {
  if (a.job[0].ntiles < 0 || a.job[1].ntiles < 0) return 1;
  auto kern = gemm_tc_kernel<GRAD, SP>;
  static DeviceFlags done = {};
  if (ensure_dynamic_smem(kern, SMEM_DYN, done)) return 1;
  const int pairs = pair_count(), ntiles = a.job[0].ntiles + a.job[1].ntiles;
  const unsigned grid = 2u * (unsigned)(ntiles < pairs ? ntiles : pairs);   // one persistent CTA per SM
  return launch_dependent(kern, dim3(grid), dim3(NTHREADS), SMEM_DYN, st, maps, a);
}

}  // namespace

int tc_projections(const Plan& pl, const as_params_t* pr, const void* wcat, int wreps, const void* x,
                   const ZeroList& z, char* ws, cudaStream_t st) {
  const int P = pl.P, NW = P + wreps * NBC;
  TcArgs a{};
  Job& j = a.job[0];
  j.M = (int64_t)pl.Bg * pl.T; j.N = P + NBC; j.kblocks = (P + BK - 1) / BK;
  a.P = P;
  a.bias = pr->b_delta; a.bc = (float*)(ws + pl.off_bc); a.status = (int*)(ws + pl.off_status); a.zero = z;
  cut_columns(CUT_PROJ, &j, pl.KL, pair_count());
  TcMaps<false> t;
  if (operand(&t.m[PM_A], x, pl.KL, j.M, P, P, BM / 2)) return 1;
  a.direct = !wcat;
  const void* wd = wcat ? wcat : pr->W_delta;
  if (operand(&t.m[PM_B], wd, pl.KL, wcat ? NW : P, P, P, j.nbase * (unit(false) / 2))) return 1;
  if (operand(&t.m[PM_B1], wd, pl.KL, wcat ? NW : P, P, P, unit(false) / 2)) return 1;
  t.m[PM_WB] = t.m[PM_WC] = t.m[PM_B];
  if (!wcat && (operand(&t.m[PM_WB], pr->W_B, pl.KL, NS, P, P, 16) || operand(&t.m[PM_WC], pr->W_C, pl.KL, NS, P, P, 16))) return 1;
  if (output(&t.m[PM_DELTA], true, CU_TENSOR_MAP_SWIZZLE_128B, ws + pl.off_delta, pl.KL, j.M, P, 32, 32)) return 1;
  if (output(&t.m[PM_BC], true, CU_TENSOR_MAP_SWIZZLE_128B, ws + pl.off_bc, pl.KL, j.M, NBC, 32, 32)) return 1;
  if (P % 32) return launch_tc<false, SP_FINE>(t, a, st);
  return pl.ordered ? launch_tc<false, SP_LOG>(t, a, st) : launch_tc<false, SP_POLY>(t, a, st);
}

int tc_gradients(const Plan& pl, const as_params_t* pr, const void* wcat, const void* x, const as_grads_t* out, char* ws, cudaStream_t st,
                 cudaEvent_t between) {
  const int64_t rows = (int64_t)pl.Bg * pl.T, all = rows * pl.KL;
  const int P = pl.P, NW = pl.gcols;   // columns of Gcat, rows of Wcat
  auto cvt = pl.gsplit == 3 ? cvt_dbc_kernel<3> : cvt_dbc_kernel<1>;
  if (launch_dependent(cvt, dim3((unsigned)((all * (NBC / 8) + 255) / 256)), dim3(256), 0, st, all, pl.du_ld, P,
                       (const float*)(ws + pl.off_dbc), (__nv_bfloat16*)(ws + pl.off_du)))
    return 1;
  TcArgs a{};
  a.P = P; a.status = (int*)(ws + pl.off_status); a.direct = !wcat;
  Job &dw = a.job[0], &dx = a.job[1];
  dw.M = P; dw.N = NW; dw.kblocks = (int)((rows + BK - 1) / BK);
  const int pairs = pair_count();
  const int64_t cdw = cut_columns(CUT_DW, &dw, pl.KL, pairs);
  if (out->dx) {
    dx.M = rows; dx.N = P; dx.kblocks = (NW + BK - 1) / BK;
    const int64_t cdx = cut_columns(CUT_DX, &dx, pl.KL, pairs);
    const int rest = pairs - dx.ntiles;
    if (dx.ntiles > 0 && rest > 0 && !between) {   // short runs: side by side, if DW on the other pairs takes no longer than both in turn
      Job side = dw;
      if (cut_columns(CUT_DW, &side, pl.KL, rest) < cdw + cdx) dw = side;
    }
  }
  TcMaps<true> t;
  const char* gcat = ws + pl.off_du;
  if (operand(&t.m[GM_X], x, pl.KL, rows, P, P, BK)) return 1;                  // X as [K = tokens, M = P]
  if (operand(&t.m[GM_G], gcat, pl.KL, rows, NW, pl.du_ld, BK)) return 1;       // Gcat as [K = tokens, N]
  if (output(&t.m[GM_DW], true, CU_TENSOR_MAP_SWIZZLE_NONE, out->dW_delta, pl.KL, P, P, 32, 32)) return 1;
  if (output(&t.m[GM_DB], true, CU_TENSOR_MAP_SWIZZLE_NONE, out->dW_B, pl.KL, NS, P, 32, 8)) return 1;
  if (output(&t.m[GM_DC], true, CU_TENSOR_MAP_SWIZZLE_NONE, out->dW_C, pl.KL, NS, P, 32, 8)) return 1;
  if (out->dx) {
    if (operand(&t.m[GM_GK], gcat, pl.KL, rows, NW, pl.du_ld, BM / 2)) return 1;   // Gcat as [M = tokens, K]
    const void* wd = wcat ? wcat : pr->W_delta;                                    // Wcat or its parts as [K, N = P]
    if (operand(&t.m[GM_W], wd, pl.KL, wcat ? NW : P, P, P, BK)) return 1;
    t.m[GM_W1] = t.m[GM_WB] = t.m[GM_WC] = t.m[GM_W];
    if (!wcat && (operand(&t.m[GM_W1], wd, pl.KL, P, P, P, 16) || operand(&t.m[GM_WB], pr->W_B, pl.KL, NS, P, P, 16) ||
                  operand(&t.m[GM_WC], pr->W_C, pl.KL, NS, P, P, 16)))
      return 1;
    if (output(&t.m[GM_DX], false, CU_TENSOR_MAP_SWIZZLE_128B, out->dx, pl.KL, rows, P, 64, 32)) return 1;
    if (output(&t.m[GM_DIR], false, CU_TENSOR_MAP_SWIZZLE_128B, ws + pl.off_dxdir, pl.KL, rows, P, 64, 32)) return 1;
  } else {
    t.m[GM_GK] = t.m[GM_W] = t.m[GM_DX] = t.m[GM_DIR] = t.m[GM_W1] = t.m[GM_WB] = t.m[GM_WC] = t.m[GM_X];
  }
  // One launch for both up to ONE_LAUNCH_BLOCKS blocks of the input gradient a pair: it saves a launch and its ramp, and DX fills DW's
  // last wave.  Longer runs have nothing to gain, and the two pairs without a tile of DW that then run ahead cost them.  Both
  // gradients, us, two launches | one, by blocks a pair: 588 x 128 (whole call) 52 | 46, 3,447 x 64 71 | 66, 3 x 5,003 x 1,000 554 | 546;
  // 40,000 x 512 [38] 68 | 60; 2 x 32,768 x 768 [135] 146 | 142; 262,144 x 384 [194] 249 | 243, x 512 [249] 310 | 304; 131,072 x 768
  // [270] 278 | 277; 43,690 x 1,536 [347] 314 | 310; 98,304 x 1,024 [354] 343 | 340; 400,000 x 512 [380] 473 | 472; 200,000 x 768 [412]
  // 429 | 432; 32,768 x 2,048 [457] 388 | 390; 131,072 x 1,024 [470] 460 | 460; 65,536 x 1,536 [520] 466 | 468; 49,152 x 2,048 [686]
  // 589 | 605; 262,144 x 2,048 [3,650] 3,258 | 3,400.
  // With phase timing always two launches, so that the phases can be told apart.
  if (dw.ntiles < 0 || ((int64_t)dx.ntiles * dx.kblocks <= ONE_LAUNCH_BLOCKS * pairs && !between)) return launch_tc<true, SP_LOG>(t, a, st);
  TcArgs first = a;
  first.job[1].ntiles = 0;
  dw.ntiles = 0;
  if (dx.ntiles < 0 || launch_tc<true, SP_LOG>(t, first, st)) return 1;
  if (between && cudaEventRecord(between, st) != cudaSuccess) return 1;
  return out->dx ? launch_tc<true, SP_LOG>(t, a, st) : 0;
}

}  // namespace as
