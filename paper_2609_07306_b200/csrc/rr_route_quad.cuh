// Full routing of a set of rows in ONE kernel, two sweeps over the key chunks, FOUR THREADS PER QUERY ROW: score
// GEMM on the tensor cores (Eq. 1), per-row TopK (Eq. 2), near-miss sentinels (Section 3.1 item 1), k-th score
// and margin (Section 3.3), mandatory global and random sentinels (Section 3.1 items 2, 3); with TEST also a relay's
// challenge test (Eq. 5) on the scores of the first sweep.  The score matrix never leaves the SM.
//
// One CTA owns 128 query rows of one problem (consecutive rows, or a segment of the compacted refresh list,
// Section 4.2; with TEST on a small grid 32 or 64 consecutive rows, rows_per_test_cta in rr_route_quad.cu) and walks the key chunks in tiles of 64, stopping at the last chunk any of its rows may select.
//   warp 0     : TMA producer (Kc tiles, 128-byte swizzle, one copy per tile)
//   warp 1     : issues tcgen05.mma (M=128, N=64, K=16) into a ring of 3 TMEM accumulators; the Qc tile is the
//                MMA's A operand in TMEM
//   warps 2-17 : selection.  Thread j of a row takes columns 32 (j % 2) .. + 31 of the tiles t with t % 2 == j / 2.
// The work per row is that of the kernel with two threads (rr_route_rows.cu), bound by the latency of its phases
// and, inside the sorts, by the half-rate ALU pipe; what four threads change: every phase is half as long, 32
// selection warps share an SM instead of 16 (56 registers a thread, two CTAs), and no phase is left to one thread of a
// row but the draws.  It pays where the phases are long: beyond 28 kept chunks (256 x 512 x 512, six layers: keep
// 30 921 -> 813 us, keep 48 1215 -> 1017; keep 20 736 -> 782 and keep 28 832 -> 898 the other way round).
//
// Sweep 1 (threshold before filtering): each thread keeps packed bf16 maxima of 32 NG groups of columns (32 positions
// x NG classes of its tiles), 128 NG groups per row.  The keep-th largest of the row's maxima (keep = k + max(m, 1))
// is a lower bound tau of its keep-th largest score.  It is found exactly: packed sorting network and merge inside a
// thread, merge of a pair's lists through shared memory, binary search over the two lists of 64.
// Sweep 2: scores >= tau go as {score, chunk id} into the row's column of CAP entries.  The search says how many groups
// of each pair of threads reach the bound; each pair gets that much of the column and half of the rest, and its
// two threads fill it from both ends.  (Four shares would overflow far more often, one shared counter costs an
// atomic and a second pass over the scores.)
// Sort: a quarter of the column per thread, in registers, by 23 bits of fixed point and the slot; three bitonic merges
// with the lists exchanged through the idle accumulators in TMEM leave the column in rank order.  Entries that
// agree in 23 bits matter only next to a cut, where they are looked at with their exact scores.
// Ids are ordered by chunk in packed registers and leave with 16-byte stores, while the row's other two threads mark
// the excluded chunks and draw the sentinels.
// Rows the fast path cannot finish exactly (a pair's part overflowed, three entries in a row that agree in 23 bits at
// a cut) take an exact slow path: one more sweep stores their complete score rows in shared memory, and a warp
// per row runs the radix select of the two-pass path.  Every mbarrier wait is bounded.
//
// 256 x 1024 x 1024, keep 48: 277 us (two threads) -> 261; 64 x 2048 x 2048, keep 96: 408 -> 300; the list of 17 % of
// 256 x 1024 rows: 130 -> 96; 32 x 1024 x 1024 55 -> 50.
// TEST, 8 x 256 x 256 (twelve layers): 371 us with the test and the list before the routing kernel, 260 in it with
// 128 rows per CTA, 251 with 32.
//
// Tried and taken back: 64 rows per CTA with every query row twice in the MMA, two threads per row, four CTAs per
// SM (high drift 5625 -> 6753 us per 16 layers: every Kc tile comes twice and waits longer); a pair's share of
// the column at 128 groups and 48 kept chunks (one row in 4000 overflows: 256 CTAs of one wave 1070 -> 1370 us); hashes of
// the draws spread over two threads ahead of their acceptance (1112 -> 1122); sleeping or hinted waits of the
// producer and the issuer (no difference).
#pragma once
#include <algorithm>
#include <type_traits>
#include "rr_common.cuh"
#include "rr_networks.cuh"
#include "rr_route_select.cuh"
#include "rr_sm100.cuh"
#include "rr_test_marks.cuh"
#include "rr_warp_topk.cuh"

using namespace sm100;
using namespace rr_select;

typedef void (*rr_quad_kernel)(RRParams, const __nv_bfloat16*, const CUtensorMap, const int32_t*, uint32_t, int, int, int, int);
rr_quad_kernel rr_quad_kernel_d64(int variant, bool test);     // (the kernels of the two head widths are compiled apart)
rr_quad_kernel rr_quad_kernel_d128(int variant, bool test);

namespace {

constexpr int BM = 128, BN = 64, ACC_STAGES = 3;
constexpr int TPR = 4, SLICE = 32;                 // threads per row, columns of a tile per thread
constexpr int SEL_WARPS = TPR * (BM / 32);
constexpr int NT = (2 + SEL_WARPS) * 32;
constexpr int A_COL = ACC_STAGES * BN;             // Qc tile behind the accumulators
constexpr int LIST = 16;                           // words of a thread's sorted maxima
constexpr int PARTS = 2 * TPR;                     // slots through which a row's threads pass their parts of the test
constexpr int LIST_SLOTS = PARTS + TPR * LIST;     // the column has at least as many slots
constexpr int MAX_STAGES = ACC_STAGES;             // of the Kc ring: tiles of 16 KB (d = 128) or 8 KB (d = 64)
constexpr int MAX_HARD = 24;                       // score rows held at once by the slow path
constexpr uint32_t SLOT_PITCH = BM * 8;            // bytes between entries of a row's column
constexpr uint32_t WORD_PITCH = BM * 4;            // [word][row] areas

__host__ __device__ constexpr int stages_of(int d, int ctas) { return d == 64 || ctas == 1 ? 3 : 2; }   // of the Kc ring

struct Ctl {
  uint64_t full[MAX_STAGES], acc_full[ACC_STAGES], acc_empty[ACC_STAGES], drain, decided;
  uint32_t tmem_base, abort_flag, hard_n, pad_;
  uint8_t cnt[TPR][BM];                 // survivors per thread; after the cuts [0], [1]: cut k / k + m undecided
  uint8_t hard_rows[BM];                // rows handed to the slow path, in registration order
  int8_t hard_slot[BM];                 // position of a row in hard_rows, -1 = none
  uint8_t gave_up[BM / 32];             // of the test: a warp of the quarter has met a wait that gave up,
  uint32_t any_routed;                  // a row of the CTA failed,
  uint32_t flagged, cand;               // rows that failed, candidates looked at,
  unsigned long long full_pairs;        // valid chunks of the rows that failed
};
constexpr int CTL_BYTES = 1024;
static_assert(sizeof(Ctl) <= CTL_BYTES, "control block too large");

// the four warps that share a quarter of the rows, barrier ids 1..4; its last two, ids 5..8
__device__ __forceinline__ void quarter_sync(int quarter) {
  asm volatile("bar.sync %0, 128;" ::"r"(quarter + 1) : "memory");
}
__device__ __forceinline__ void drawers_sync(int quarter) {
  asm volatile("bar.sync %0, 64;" ::"r"(quarter + 5) : "memory");
}

__device__ __forceinline__ uint32_t swap_halves(uint32_t w) { return __byte_perm(w, w, 0x1032); }

// A bitonic sequence of any length into order: half-cleaners while the length is even (they need no power
// of two), a sorting network for what is left (3 or 5 elements, 9 for lengths of 36).
template <int N, class OP>
__device__ __forceinline__ void bitonic_merge(uint32_t* x) {
  if constexpr (N > 1 && N % 2 == 0) {
#pragma unroll
    for (int i = 0; i < N / 2; ++i) OP::ce(x[i], x[i + N / 2]);
    bitonic_merge<N / 2, OP>(x);
    bitonic_merge<N / 2, OP>(x + N / 2);
  } else if constexpr (N > 1) {
    OESort<0, pow2_at_least(N), OP, N>::run(x);
  }
}
// Packed words whose low and high halves are two lists of N in order: afterwards one list of 2 N, element
// i in the low half of word i, element i + N in its high half.
template <int N, class OP>
__device__ __forceinline__ void merge_halves(uint32_t* x) {
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    uint32_t first = x[i], last = swap_halves(x[N - 1 - i]);
    OP::ce(first, last);                               // (low i, high N-1-i) and (high i, low N-1-i)
    x[i] = __byte_perm(first, last, 0x5410);
    x[N - 1 - i] = __byte_perm(first, last, 0x7632);
  }
  bitonic_merge<N, OP>(x);
}
// The same for words that hold one bitonic sequence of 2 N, element i + N above element i.
template <int N, class OP>
__device__ __forceinline__ void bitonic_merge_halves(uint32_t* x) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    uint32_t first = x[i], last = swap_halves(x[i]);
    OP::ce(first, last);
    x[i] = __byte_perm(first, last, 0x5410);
  }
  bitonic_merge<N, OP>(x);
}

// ---- a row's threads exchange sorted keys through TMEM: N words of this thread to / from columns at a --
template <int N>
__device__ __forceinline__ void tmem_put(uint32_t a, const uint32_t* x) {
  static_assert(N % 2 == 0, "pairs of columns");
#pragma unroll
  for (int i = 0; i + 4 <= N; i += 4)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                 ::"r"(a + i), "r"(x[i]), "r"(x[i + 1]), "r"(x[i + 2]), "r"(x[i + 3]) : "memory");
  if constexpr (N % 4 == 2)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(a + N - 2), "r"(x[N - 2]), "r"(x[N - 1]) : "memory");
  tmem_st_wait();
}
template <int N>
__device__ __forceinline__ void tmem_get(uint32_t a, uint32_t* x) {
#pragma unroll
  for (int i = 0; i + 4 <= N; i += 4)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(x[i]), "=r"(x[i + 1]), "=r"(x[i + 2]), "=r"(x[i + 3]) : "r"(a + i) : "memory");
  if constexpr (N % 4 == 2)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(x[N - 2]), "=r"(x[N - 1]) : "r"(a + N - 2) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < N; ++i) asm volatile("" : "+r"(x[i]) :: "memory");   // no use ahead of the wait
}

// Qc words of a row into TMEM
__device__ __forceinline__ void tmem_st_16(uint32_t a, const uint32_t (&x)[16]) { tmem_put<16>(a, x); }

constexpr int GUARD = 16;                  // scores between two looks at the room left
template <int I, bool EDGE>
__device__ __forceinline__ void filter_all(uint32_t& w, const uint32_t* acc, float tau, uint32_t col0, uint32_t step,
                                           int v) {
  if constexpr (I < GUARD) {
    filter_one<I, EDGE>(w, acc[I], tau, col0, step, v);
    filter_all<I + 1, EDGE>(w, acc, tau, col0, step, v);
  }
}

// ---- gather and order -------------------------------------------------------------------------
// The ids of n consecutive entries at `src`, ordered by chunk id and written to dst [0, width), -1 behind
// the last one.  Ids fit 16 bits: all of it in packed words.
template <int N>
__device__ __forceinline__ void order_ids(uint32_t src, int n, int32_t* dst, int width, bool vec, bool on) {
  uint32_t x[N / 2];
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    uint32_t lo = 0xFFFFu, hi = 0xFFFFu;       // (order behind every id)
    if (i < n) lo = lds32(src + (uint32_t)i * SLOT_PITCH + 4u);
    if (i + N / 2 < n) hi = lds32(src + (uint32_t)(i + N / 2) * SLOT_PITCH + 4u);
    x[i] = __byte_perm(lo, hi, 0x5410);
  }
  OESort<0, N / 2, AscU2, N / 2>::run(x);
  merge_halves<N / 2, AscU2>(x);
  if (!on) return;
  auto id = [&](int i) -> uint32_t { return i < n ? (i < N / 2 ? x[i] & 0xFFFFu : x[i - N / 2] >> 16) : 0xFFFFFFFFu; };
#pragma unroll
  for (int q = 0; q < N; q += 4) {
    if (q < width) {
      if (vec) {
        *reinterpret_cast<uint4*>(dst + q) = make_uint4(id(q), id(q + 1), id(q + 2), id(q + 3));
      } else {
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (q + t < width) dst[q + t] = (int32_t)id(q + t);
      }
    }
  }
}

#ifdef RR_PHASE_TIMING
__device__ unsigned long long g_quad_phase[32];
#define PH_T0() long long ph_t0_ = clock64()
#define PH_LAP(i) do { const long long t1_ = clock64(); if ((threadIdx.x & 31) == 0) atomicAdd(&g_quad_phase[i], (unsigned long long)(t1_ - ph_t0_)); ph_t0_ = t1_; } while (0)
#define PH_CNT(i, val_) atomicAdd(&g_quad_phase[i], (unsigned long long)(val_))
#else
#define PH_CNT(i, val_) do {} while (0)
#define PH_T0() do {} while (0)
#define PH_LAP(i) do {} while (0)
#endif

// NG: classes of a thread's tiles (128 NG groups of columns per row); CAP: entries per row.
// TEST: a relay's challenge test runs on the scores of sweep 1, rows that pass it are left alone.
template <int D, int NG, int CAP, int CTAS, bool TEST>
__global__ void __launch_bounds__(NT, CTAS)
route_quad_kernel(RRParams p, const __nv_bfloat16* __restrict__ qc,
                  const __grid_constant__ CUtensorMap tmap_k, const int32_t* __restrict__ row_list_arg,
                  uint32_t layer, int hooks, int ring_bytes, int cta_stride, int rows_per_cta) {
  constexpr int KH = D / 64;                               // K-halves of a tile
  constexpr int TILE = BN * D * 2;
  constexpr int STAGES = stages_of(D, CTAS);
  static_assert(STAGES >= 2 && STAGES <= ACC_STAGES, "see produce()");
  constexpr int M = CAP / TPR;                             // entries per quarter column
  constexpr int TMEM_COLS = CTAS == 2 ? 256 : 512;
  constexpr int XCH = CTAS == 2 ? 96 : 256;                // second set of columns for the exchanges (first: 0, over the accumulators)
  static_assert(CAP % (2 * TPR) == 0 && TPR * M <= (CTAS == 2 ? 96 : 192), "exchange columns");
  constexpr int S1 = 16;                                   // columns per load of sweep 1
  extern __shared__ __align__(1024) uint8_t smem_raw[];    // (checked below: the swizzle needs it)
  uint8_t* smem = smem_raw;
  uint8_t* sB = smem;                                      // Kc ring; after the sweeps: keys, bitmap
  Ctl* ctl = (Ctl*)(smem + ring_bytes);
  uint8_t* s_col = (uint8_t*)ctl + CTL_BYTES;              // [CAP][BM] entries

  const int tid = threadIdx.x, warp = __shfl_sync(FULL, tid >> 5, 0), lane = tid & 31;
  const CUtensorMap* const tmap_ptr = &tmap_k;             // address in parameter space (what TMA needs)
  if (tid == 0) tma_prefetch_desc(tmap_ptr);               // first thing: the descriptor fetch takes a while
#ifdef RR_PHASE_TIMING
  const long long cta_t0_ = clock64();
#endif
  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) mbar_init(&ctl->full[s], 1);
    for (int s = 0; s < ACC_STAGES; ++s) {
      mbar_init(&ctl->acc_full[s], 1);
      mbar_init(&ctl->acc_empty[s], SEL_WARPS / 2);        // one arrival per warp that reads the tile
    }
    mbar_init(&ctl->drain, 1);
    ctl->abort_flag = 0;
    ctl->hard_n = 0;
    ctl->flagged = 0; ctl->cand = 0; ctl->full_pairs = 0ull;
    for (int q = 0; q < BM / 32; ++q) ctl->gave_up[q] = 0;
    ctl->any_routed = 0;
    mbar_init(&ctl->decided, BM / 32);                     // one arrival per quarter
    mbar_fence_init();
  }
  if ((smem_u32(smem) & 1023u) != 0u) {                    // reported like a wait that gave up
    if (tid == 0) atomicOr(p.status, RR_STATUS_TIMEOUT);
    rr_pdl_wait();
    return;
  }
  // The predecessor writes the refresh list; at an anchor it is the fill, which only writes
  // book-keeping that is not read here, and has triggered after its own wait: the inputs are complete.
  // The wait for it is then at the end of every path (see rr_pdl_wait).
  if (TEST || row_list_arg) rr_pdl_wait();
  // The list's length and this problem's part of it are asked for together: the rows hang on them, and the Qc rows
  // on those.
  const int prob = blockIdx.x % p.P;
  int list_n = 0, list_lo = 0, list_hi = 0;
  if (row_list_arg) { list_n = *p.refresh_count; list_lo = p.problem_offsets[prob]; list_hi = p.problem_offsets[prob + 1]; }
  // a relay call that the forced-anchor policy turned into full routing has the identity list:
  // take the anchor's path (consecutive rows, no gathers through the list)
  const bool forced_call = row_list_arg && p.force_threshold > 0 && p.force_in[0] > 0;
  // A refresh list that holds nearly every row (high drift) is served the same way, with the
  // rows that are not on it masked out: gathering 7/8 of the rows through the list costs more
  // than sweeping the missing eighth for nothing (results per row are the same either way).
  const bool dense_refresh = row_list_arg && !forced_call &&
                             (long long)list_n * 8 >= (long long)p.rows * 7;
  const int32_t* __restrict__ row_list = (forced_call || dense_refresh) ? nullptr : row_list_arg;
  const bool force_hard = hooks & 1, force_timeout = hooks & 2, force_late = hooks & 4;      // test hooks
  // Row tiles are handed out heaviest first (under the causal mask the last tile of a problem
  // walks the most key chunks), so the tail of the grid is made of the short ones and, where a refresh
  // list is short, of the CTAs that find no tile: in front they kept the SMs from the
  // others (17 % of 256 x 1024 rows on the list: 130 -> 120 us).
  const int seg_lo = row_list ? list_lo : 0, seg_hi = row_list ? list_hi : p.n_q;
  const int own = TEST ? rows_per_cta : BM;                // rows of a CTA (fewer than the MMA's: the others are empty)
  const int tm = (seg_hi - seg_lo + own - 1) / own - 1 - (int)(blockIdx.x / p.P);
  if (tm < 0) { if (!TEST && !row_list_arg) rr_pdl_wait(); return; }  // nothing to do (uniform per CTA)
  const bool tested = TEST && !(p.force_threshold > 0 && p.force_in[0] > 0);   // (a forced anchor routes every row)

  // row of the CTA's tile -> query row of the problem and global row id; -1 = no row
  auto locate = [&](int rr, int& row_out, int& g_out) {
    const int local = tm * own + rr;
    row_out = -1; g_out = 0;
    if (TEST && rr >= own) return;
    if (row_list) {
      if (seg_lo + local < seg_hi) { g_out = row_list[seg_lo + local]; row_out = g_out - prob * p.n_q; }
    } else if (local < p.n_q) {
      row_out = local; g_out = prob * p.n_q + local;
    }
  };
  // ---- selection-side geometry (meaningful for warps 2..) -------------------------------------
  const int quarter = warp & 3, j = (warp - 2) >> 2;
  const int pair = j >> 1, side = j & 1;                   // tiles t with t % 2 == pair, columns 32 side .. 32 side + 31 of each
  const int r = quarter * 32 + lane;                       // row inside the CTA
  const bool is_sel = warp >= 2;
  // ---- the Qc tile goes to TMEM: a thread of row r loads its part of the row (two bf16 per
  // 32-bit word, as they lie in memory; refresh rows are not contiguous, so this is also the
  // gather) and stores it to TMEM lane r, where the MMA reads its A operand; rows without a
  // query are 0.  The loads are issued first so that their latency overlaps the rest of the set-up.
  constexpr int QW = 16, QT = D / 2 / QW;                  // 32-bit words per thread, threads per row
  const bool q_loader = is_sel && j < QT;
  uint32_t qv[QW];
  int row = -1, g = 0;
  if (is_sel) locate(r, row, g);
  if (q_loader) {
    const uint4* src = reinterpret_cast<const uint4*>(qc + ((size_t)prob * p.n_q + max(row, 0)) * D) + j * (QW / 4);
#pragma unroll
    for (int i = 0; i < QW / 4; ++i) {
      uint4 t = make_uint4(0, 0, 0, 0);
      if (row >= 0) t = __ldg(src + i);
      qv[4 * i] = t.x; qv[4 * i + 1] = t.y; qv[4 * i + 2] = t.z; qv[4 * i + 3] = t.w;
    }
  }
  if (is_sel && j == 0) ctl->hard_slot[r] = -1;
  // The test's bitmaps lie in the column, word w of both at slot w: the route's in the score words, the
  // sentinels' in the id words.
  const int words = (p.n_k + 31) / 32;
  if (tested && is_sel)
    for (int w = j; w < words; w += TPR) sts64(smem_u32(s_col) + (uint32_t)r * 8u + (uint32_t)w * SLOT_PITCH, 0u, 0u);
  if (warp == 1) {
    tmem_alloc(&ctl->tmem_base, TMEM_COLS);
    rr_pdl_trigger();                                      // (not before: the successor takes TMEM, too)
  }
  // The Kc loads depend on nothing but the number of key tiles (from the tile's last row: rows
  // ascend inside a tile), and the ring's stages are all free: the producer fills the ring before
  // the CTA's first barrier, while the Qc rows are on their way.
  const int last_local = min(seg_hi - seg_lo, (tm + 1) * own) - 1;
  const int last_row = row_list ? row_list[seg_lo + last_local] - prob * p.n_q : last_local;
  const int n_tiles = (rr_valid_count(last_row, p.n_k, p.causal, p.causal_offset) + BN - 1) / BN;
  const uint32_t ring = smem_u32(sB);
  const int pre = min(STAGES, 2 * n_tiles);
  if (warp == 0) {
    __syncwarp();
    for (int gt = 0; gt < pre; ++gt)
      tma_load_tile_warp(ring + gt * TILE, tmap_ptr, (gt >= n_tiles ? gt - n_tiles : gt) * BN, prob, &ctl->full[gt], TILE);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (q_loader) {
    tmem_st_16(ctl->tmem_base + ((uint32_t)(quarter * 32) << 16) + A_COL + j * QW, qv);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  volatile uint32_t* abort_flag = &ctl->abort_flag;

  // Sweep 2 of a CTA that tests its rows begins when its quarters have decided, and does not if all of them pass
  // (a wait that gives up ends it as well).  Called by whole warps.  What fails is sorted meanwhile, so that nobody
  // waits (8 x 256 x 256 at 83 % and 15 x 389 x 777 at 55 % failing: no difference).  With no row failing, six layers:
  // 7 x 1345 x 1915 202 -> 181 us, 1 x 202 x 1362 176 -> 154, 8 x 200 x 256 79 -> 75.
  auto sweep2 = [&]() -> bool {
    return __all_sync(FULL, mbar_wait_spin(&ctl->decided, 0, abort_flag)) && *(volatile uint32_t*)&ctl->any_routed != 0u;
  };
  // Tiles are numbered through all sweeps (gt): stage and phase of every ring follow from gt.
  // A stage of the Kc ring is free again when the MMAs of its tile are done, which is what acc_full
  // says: tile gt may be fetched once tile gt - STAGES is complete.  (That barrier cannot run ahead
  // of the wait: its next completion is tile gt - STAGES + ACC_STAGES >= gt, not fetched yet.)
  // Both roles are run by whole, converged warps (see umma_bf16_ts_warp).
  auto produce = [&](int first, int count, int begin) {
    int t = begin % n_tiles, s = begin % STAGES, gt = begin;
#pragma unroll 1
    for (; gt < first + count; ++gt) {
      const int done = gt - STAGES;
      if (tested && done == n_tiles && !sweep2()) break;   // (first tile that needs an MMA of sweep 2)
      if (done >= first &&
          !__all_sync(FULL, mbar_wait_spin(&ctl->acc_full[done % ACC_STAGES], (done / ACC_STAGES) & 1, abort_flag))) break;
      tma_load_tile_warp(ring + s * TILE, tmap_ptr, t * BN, prob, &ctl->full[s], TILE);
      if (++t == n_tiles) t = 0;
      if (++s == STAGES) s = 0;
    }
    // do not go on while copies into this CTA's shared memory may still be in flight
#pragma unroll 1
    for (int u = max(first, gt - STAGES); u < gt; ++u)
#pragma unroll 1
      for (uint32_t it = 0; it < kSpinLimit && !mbar_try_wait(&ctl->full[u % STAGES], (u / STAGES) & 1); ++it) __nanosleep(64);
    __syncwarp();
  };
  auto issue = [&](int first, int count) {
    constexpr uint32_t idesc = umma_idesc_bf16(BM, BN);
    const uint32_t tmem_u = __shfl_sync(FULL, tmem_base, 0);
    const uint64_t desc0 = umma_desc_k_sw128(ring);
#pragma unroll 1
    for (int gt = first; gt < first + count; ++gt) {
      const int as = gt % ACC_STAGES, s = gt % STAGES;
      if (tested && gt == n_tiles && !sweep2()) return;
      if (!__all_sync(FULL, mbar_wait_spin(&ctl->acc_empty[as], ((gt / ACC_STAGES) & 1) ^ 1, abort_flag))) return;
      if (!__all_sync(FULL, mbar_wait_spin(&ctl->full[s], (gt / STAGES) & 1, abort_flag))) return;
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < KH * 4; ++k)
        umma_bf16_ts_warp(tmem_u + as * BN, tmem_u + A_COL + k * 8,
                          desc0 + (uint64_t)(s * (TILE >> 4) + (k >> 2) * (BN * 128 >> 4) + (k & 3) * 2), idesc,
                          k > 0 ? 1u : 0u);
      umma_commit_warp(&ctl->acc_full[as]);
    }
  };

  const int v = row >= 0 ? rr_valid_count(row, p.n_k, p.causal, p.causal_offset) : 0;
  bool routed = row >= 0 && (!dense_refresh || p.flags[g] != 0);           // this row is (re)routed here
  const float pinf = __int_as_float(0x7f800000), ninf = __int_as_float(0xff800000);
  const uint32_t col = smem_u32(s_col) + (uint32_t)r * 8u;                 // the row's entries
  const uint32_t bits = smem_u32(sB) + (uint32_t)r * 4u;                   // the row's bitmap (ring area)
  const uint32_t acc_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
  const int vmaxw = __reduce_max_sync(FULL, v);
  const int vminw = min(__reduce_min_sync(FULL, row >= 0 ? v : 0x7FFFFFFF), vmaxw);
  bool alive = true;
  // Consumer side of tile gt of the running numbering: wait for it / hand the accumulator back.
  auto tile_wait = [&](int gt) -> bool {
    if (!alive) return false;
    // test hook: the first wait of CTA 0 counts as expired (what a wait that ran out does:
    // raise the CTA's abort flag; every role then leaves its loop at its next poll)
    if (force_timeout && blockIdx.x == 0) *abort_flag = 1u;
    const bool ready = mbar_wait(&ctl->acc_full[gt % ACC_STAGES], (gt / ACC_STAGES) & 1, abort_flag) &&
                       !(force_timeout && blockIdx.x == 0);
    alive = __all_sync(FULL, ready);
    tc_fence_after();
    return alive;
  };
  auto tile_release = [&](int gt) {
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(&ctl->acc_empty[gt % ACC_STAGES]);
  };
  auto acc_addr = [&](int gt) -> uint32_t { return acc_lane + (uint32_t)((gt % ACC_STAGES) * BN + side * SLICE); };

  // The quarter's byte among the flagged counts (stored as soon as it is known: at the kernel's end it was 0.4 us late).
  auto store_count = [&](int n) { ((uint8_t*)(p.tile_counts + prob * p.tiles_per_problem))[(tm * own >> 5) + quarter] = (uint8_t)n; };
  static_assert(RR_ROW_TILE == 128, "a byte of the tile's word per quarter");

  if (warp == 0) {
    // The Kc tiles beyond the ring are asked into L2, and so are the Qc rows of the CTA that will
    // start about when this one ends (CTAs start in index order as SMs fall free: the one that comes
    // cta_stride = CTAs per SM x SMs later), so that its set-up waits for L2 instead of DRAM.  Hints
    // only: nothing depends on them.
    for (int t = pre + lane; t < n_tiles; t += 32) tma_prefetch_l2_tile(tmap_ptr, t * BN, prob);
    const int nb = (int)blockIdx.x + cta_stride;
    if (nb < (int)gridDim.x) {
      const int nprob = nb % p.P;
      int nlo = 0, nhi = p.n_q;
      if (row_list) { nlo = p.problem_offsets[nprob]; nhi = p.problem_offsets[nprob + 1]; }
      const int ntm = (nhi - nlo + own - 1) / own - 1 - nb / p.P;
      for (int i = lane; i < own && ntm >= 0; i += 32) {
        const int local = ntm * own + i;
        if (local >= nhi - nlo) break;
        const size_t grow = row_list ? (size_t)row_list[nlo + local] : (size_t)nprob * p.n_q + local;
        const char* src = reinterpret_cast<const char*>(qc + grow * D);
#pragma unroll
        for (int b = 0; b < D * 2; b += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + b));
      }
    }
    __syncwarp();
    produce(0, 2 * n_tiles, pre);
  } else if (warp == 1) {
    issue(0, 2 * n_tiles);
  } else if (!__any_sync(FULL, routed)) {
    // A quarter without a row to route (the end of a refresh list, a ragged last tile) only hands its
    // accumulators back.  All of its warps come here, so nobody waits for them at its barriers
    // (3 % of 256 x 256 rows on the list: 24.9 -> 24.1 us).
    // (rows behind the problem's last one, in the same row tile, are none of another CTA's)
    if (tested && j == 0 && lane == 0 && tm * own + quarter * 32 >= p.n_q && (tm * own & (RR_ROW_TILE - 1)) + quarter * 32 < RR_ROW_TILE)
      store_count(0);
    if (tested && j == 0 && lane == 0) mbar_arrive(&ctl->decided);
#pragma unroll 1
    for (int first = 0; first < 2 * n_tiles; first += n_tiles) {
      if (tested && first > 0 && !sweep2()) break;
#pragma unroll 1
      for (int t = pair; t < n_tiles && tile_wait(first + t); t += 2) tile_release(first + t);
    }
  } else do {
    PH_T0();
#ifdef RR_PHASE_TIMING
    if (lane == 0) PH_CNT(12, ph_t0_ - cta_t0_);
#endif
    const int keep_cfg = p.k + max(p.m, 1);
    const int T = min(keep_cfg, v), kk = min(p.k, v);        // ranks that the row can fill
    // Empty slots of the column read as -inf in the sort.  (The score words; the id words hold lists first.)
    auto slot = [&](int e) -> uint32_t { return col + (uint32_t)e * SLOT_PITCH; };
    if (tested) {
      // ---- the ledger rows of the quarter's 32 query rows, read as one array, into the bitmaps -------------
      // (two warps the routes, two the sentinels)
      const int row0 = tm * own + quarter * 32, n_rows = max(0, min(32, p.n_q - row0));
      bool bad = false;
      int n_cand = rr_mark_rows<2, SLOT_PITCH>(p, pair == 0 ? p.routes : p.sentinels, pair == 0 ? p.k : p.sw, prob, row0, n_rows,
                                               smem_u32(s_col) + (uint32_t)quarter * 256u + 4u * (uint32_t)pair, 8u, side, lane, bad);
      n_cand = __reduce_add_sync(FULL, n_cand);
      if (lane == 0) atomicAdd(&ctl->cand, (uint32_t)n_cand);
      if (__any_sync(FULL, bad) && lane == 0) atomicOr(p.status, RR_STATUS_BAD_INDEX);
      if (p.debug && row >= 0 && j == 0)
        for (int q = 0; q < p.c; ++q) p.cand_scores[(size_t)g * p.c + q] = __int_as_float(0x7fc00000);
      quarter_sync(quarter);
    }
    float amin = pinf, bmax = ninf;
    // ===== sweep 1: packed group maxima =============================================================
    float tau, scale;
    int split;                                               // first slot of the second pair's part of the column
    {
      constexpr int W = SLICE / 2;                           // words per class
      uint32_t mx[NG * W];
#pragma unroll
      for (int i = 0; i < NG * W; ++i) mx[i] = 0xff80ff80u;
#pragma unroll 1
      for (int t0 = pair; t0 < n_tiles; t0 += 2 * NG) {
#pragma unroll
        for (int c = 0; c < NG; ++c) {
          const int t = t0 + 2 * c;
          if (t < n_tiles && tile_wait(t)) {
            uint32_t wa = 0u, wb = 0u;                       // candidates among the thread's 32 columns
            if (tested && 2 * t + side < words) lds64(slot(2 * t + side), wa, wb);
            const bool candidates = TEST && __any_sync(FULL, (wa | wb) != 0u);
#pragma unroll
            for (int h = 0; h < SLICE / S1; ++h) {
              const int col0 = t * BN + side * SLICE + h * S1;
              uint32_t acc[S1];
              if (col0 < vmaxw) tmem_get<S1>(acc_addr(t) + (uint32_t)(h * S1), acc);
              if (h == SLICE / S1 - 1) tile_release(t);
              if (TEST && candidates) {
#pragma unroll
                for (int i = 0; i < S1; ++i) {
                  min_if(amin, __uint_as_float(acc[i]), wa, 1u << (h * S1 + i));
                  max_if(bmax, __uint_as_float(acc[i]), wb, 1u << (h * S1 + i));
                }
                if (p.debug && row >= 0) {                   // tests: every candidate's score
                  for (int q = 0; q < p.c; ++q) {
                    const int id = q < p.k ? p.routes[(size_t)g * p.k + q] : p.sentinels[(size_t)g * p.sw + q - p.k];
                    if (id < col0 || id >= v || id >= col0 + S1) continue;
#pragma unroll
                    for (int i = 0; i < S1; ++i)
                      if (id - col0 == i) p.cand_scores[(size_t)g * p.c + q] = __uint_as_float(acc[i]);
                  }
                }
              }
              if (col0 + S1 <= vminw) {
#pragma unroll
                for (int i = 0; i < S1 / 2; ++i) {
                  const uint32_t pk = __byte_perm(acc[2 * i], acc[2 * i + 1], 0x7632);   // upper halves: bf16, cut
                  asm("max.bf16x2 %0, %0, %1;" : "+r"(mx[c * W + h * (S1 / 2) + i]) : "r"(pk));
                }
              } else if (col0 < vmaxw) {                     // some row's last chunk lies inside
                const int nv = v - col0;
#pragma unroll
                for (int i = 0; i < S1 / 2; ++i) {
                  const uint32_t pk = __byte_perm(acc[2 * i], acc[2 * i + 1], 0x7632);
                  const uint32_t pm = 2 * i + 1 < nv ? pk : (pk & 0xffffu) | 0xff800000u;
                  asm("max.bf16x2 %0, %0, %1;" : "+r"(mx[c * W + h * (S1 / 2) + i]) : "r"(2 * i < nv ? pm : 0xff80ff80u));
                }
              }
            }
          }
        }
      }
      PH_LAP(0);
      // one sorted list of 32; with two classes the upper half of each pair of lists is kept: fewer
      // groups than there are, a valid bound all the same
      OESort<0, W, DescBF2, W>::run(mx);
      if constexpr (NG == 2) {
        OESort<0, W, DescBF2, W>::run(mx + W);
#pragma unroll
        for (int i = 0; i < W; ++i) asm("max.bf16x2 %0, %0, %1;" : "+r"(mx[i]) : "r"(mx[2 * W - 1 - i]));
        bitonic_merge<W, DescBF2>(mx);
      }
      merge_halves<W, DescBF2>(mx);
      PH_LAP(1);
      // the two threads of a pair merge their lists: the first keeps the upper half, the second the lower
      // one.  Lists go through the (unused) column: score words first, then id words.  (Slots of thread j are
      // those with e % 4 == j: the words of the test's bitmaps that only it reads.)
#pragma unroll
      for (int i = 0; i < LIST; ++i) sts32(slot(TPR * i + j), mx[i]);
      if (tested) { sts32(slot(j) + 4u, __float_as_uint(amin)); sts32(slot(TPR + j) + 4u, __float_as_uint(bmax)); }
      // Whether the test stands is one decision of the quarter, taken at the barrier: the abort flag may rise at any
      // time, and warps that read it for themselves could part here, some of them at barriers that the others never
      // reach.  (A wait that gave up before: the rows stay as they are.  One that gives up later: see tile_wait.)
      if (tested && lane == 0 && (!alive || *abort_flag != 0u)) ctl->gave_up[quarter] = 1;
      quarter_sync(quarter);
      if (tested) {
        const bool stands = ctl->gave_up[quarter] == 0;
        // test hook: a wait expires between the decision and what hangs on it, seen by one warp of the four at first
        if (force_late && blockIdx.x == 0 && j == TPR - 1) *abort_flag = 1u;
#pragma unroll
        for (int t = 0; t < TPR; ++t) {
          amin = fminf(amin, ldsf(slot(t) + 4u));
          bmax = fmaxf(bmax, ldsf(slot(TPR + t) + 4u));
        }
        routed = row >= 0 && stands && rr_challenge(p, g, amin, bmax);
        const unsigned failed = __ballot_sync(FULL, routed); // (the quarter's four warps agree)
        if (j == 0) {
          if (row >= 0 && stands) { p.flags[g] = routed ? 1 : 0; p.alpha[g] = amin; p.beta[g] = bmax; }
          const int n_flag = __popc(failed), v_sum = __reduce_add_sync(FULL, routed ? v : 0);
          if (lane == 0) {
            if (failed) ctl->any_routed = 1;
            mbar_arrive(&ctl->decided);
            store_count(n_flag);
            atomicAdd(&ctl->flagged, (uint32_t)n_flag);
            atomicAdd(&ctl->full_pairs, (unsigned long long)v_sum);
          }
        }
        if (failed == 0u) {                                  // sweep 2's accumulators go back, if another quarter needs it
          if (!sweep2()) break;
#pragma unroll 1
          for (int t = pair; t < n_tiles && tile_wait(n_tiles + t); t += 2) tile_release(n_tiles + t);
          break;
        }
      }
#pragma unroll
      for (int i = 0; i < LIST; ++i) {
        const uint32_t y = swap_halves(lds32(slot(TPR * (LIST - 1 - i) + (j ^ 1))));
        if (side == 0) asm("max.bf16x2 %0, %0, %1;" : "+r"(mx[i]) : "r"(y));
        else asm("min.bf16x2 %0, %0, %1;" : "+r"(mx[i]) : "r"(y));
      }
      bitonic_merge_halves<LIST, DescBF2>(mx);
#pragma unroll
      for (int i = 0; i < LIST; ++i) sts32(slot(PARTS + TPR * i + j) + 4u, mx[i]);
      quarter_sync(quarter);
      // the T-th largest of the two lists of 64 (element e: word e % 16 of thread e / 32, upper half from 16 on)
      auto entry = [&](int list, int e) -> float {
        const uint32_t w = lds32(slot(PARTS + TPR * (e & 15) + 2 * list + (e >> 5)) + 4u);
        return __uint_as_float(e & 16 ? w & 0xffff0000u : w << 16);
      };
      auto A = [&](int e) -> float { return entry(0, e); };
      auto B = [&](int e) -> float { return entry(1, e); };
      const int a = rank_split<64>(T, A, B);
      {
        const float la = A(max(a - 1, 0)), lb = B(max(T - a - 1, 0));
        tau = fminf(a > 0 ? la : pinf, T > a ? lb : pinf);
      }
      float top = fmaxf(A(0), B(0));
      // A pair has as many survivors as groups at or above the bound, and about a fifth more: half of what
      // the column has beyond T goes to each.
      split = a + (CAP - T) / 2;
#pragma unroll
      for (int e = 0; e < M; ++e) sts32(slot(j * M + e), 0xff800000u);
      quarter_sync(quarter);                                 // lists read, column empty
      // a maximum is a score with its low half cut off, i.e. moved towards zero: a negative bound is
      // lowered by one bf16 step, a positive top raised by one
      const uint32_t tb = __float_as_uint(tau);
      if ((tb & 0x80000000u) && tb != 0xff800000u) tau = __uint_as_float(tb + 0x10000u);
      if (top >= 0.f) top = __uint_as_float(__float_as_uint(top + 0.f) + 0x10000u);
      scale = __fdividef(1.0f - 1.0f / 2097152.0f, top - tau);
      if (!(top > tau && scale < 1e30f)) scale = 0.f;        // nothing to tell apart
      if (!routed) tau = pinf;                               // rows without work pass nothing
    }
    PH_LAP(2);

    // ===== sweep 2: threshold filter into the row's column ==========================================
    // A pair's two threads fill its part from both ends.  Running over into the other pair's part only spoils
    // a row that has overflowed; the two in the middle stop where they would leave the column.
    const uint32_t step = side == 0 ? SLOT_PITCH : 0u - SLOT_PITCH;
    const uint32_t first = slot(j == 0 ? 0 : j == 1 ? split - 1 : j == 2 ? split : CAP - 1);   // this thread's entry 0
    const int room = j == 1 ? split : j == 2 ? CAP - split : CAP;
    uint32_t waddr = first;
    bool over = false;                                       // the room did not suffice
    auto filled = [&]() -> int { return (int)(side == 0 ? waddr - first : first - waddr); };     // bytes
#pragma unroll 1
    for (int t = pair; t < n_tiles; t += 2) {
      const int gt = n_tiles + t, col0 = t * BN + side * SLICE;
      if (!tile_wait(gt)) break;
      uint32_t acc[SLICE];
      if (col0 < vmaxw) tmem_ld_32x32(acc_addr(gt), acc);
      tile_release(gt);
#pragma unroll
      for (int h = 0; h < SLICE / GUARD; ++h) {
        const int c0 = col0 + h * GUARD;
        if (c0 < vmaxw) {
          if (!__any_sync(FULL, filled() > (room - GUARD) * (int)SLOT_PITCH)) {
            if (c0 + GUARD <= vminw) filter_all<0, false>(waddr, acc + h * GUARD, tau, (uint32_t)c0, step, v);
            else filter_all<0, true>(waddr, acc + h * GUARD, tau, (uint32_t)c0, step, v);
          } else {                // the room may run out inside this slice
            int n = filled() / (int)SLOT_PITCH;
#pragma unroll
            for (int i = 0; i < GUARD; ++i) {
              const float s = __uint_as_float(acc[h * GUARD + i]);
              if (s >= tau && c0 + i < v) {
                if (n < room) { sts64(waddr, acc[h * GUARD + i], (uint32_t)(c0 + i)); waddr += step; }
                ++n;
              }
            }
            if (n > room) waddr = first + step * (uint32_t)room, over = true;
          }
        }
      }
    }
    ctl->cnt[j][r] = (uint8_t)(over ? 255 : filled() / (int)SLOT_PITCH);
    PH_LAP(3);
    // the bitmap of excluded chunks starts empty once the ring is idle (all of sweep 2 has been consumed)
    quarter_sync(quarter);

    // ===== sort: the column in rank order ================================================================
    const bool have = alive && routed;
    const bool sampling = p.r > 0 || p.n_global > 0;
    const bool top_half = j < 2;
    bool bad;
    {
      const int n0 = ctl->cnt[0][r] + ctl->cnt[1][r], n1 = ctl->cnt[2][r] + ctl->cnt[3][r];
      bad = have && (n0 > split || n1 > CAP - split || n0 + n1 < T);   // (too few only after a wait gave up)
    }
    {
      // Each thread sorts a quarter of the column by keys of 23 bits of fixed point and the slot; the pairs'
      // lists are merged, then the two lists of half the column: thread j ends with ranks M j .. M j + M - 1.
      uint32_t key[M], other[M];
      const uint32_t put0 = acc_lane + (uint32_t)(j * M), put1 = put0 + XCH;
      auto from = [&](int t) -> uint32_t { return acc_lane + (uint32_t)(t * M); };
#pragma unroll
      for (int i = 0; i < M; ++i)
        key[i] = fixed_bits(ldsf(slot(j * M + i)), tau, scale) * 256u + (uint32_t)(j * M + i);
      OESort<0, pow2_at_least(M), DescPos, M>::run(key);
      auto exchange = [&](uint32_t to, uint32_t src) {
        tmem_put<M>(to, key);
        tc_fence_before();
        quarter_sync(quarter);
        tc_fence_after();
        tmem_get<M>(src, other);
      };
      auto keep_larger = [&](bool larger, auto reversed) {
        constexpr bool R = decltype(reversed)::value;
#pragma unroll
        for (int i = 0; i < M; ++i) {
          const float x = __uint_as_float(key[i]), y = __uint_as_float(other[R ? M - 1 - i : i]);
          key[i] = __float_as_uint(larger ? fmaxf(x, y) : fminf(x, y));
        }
      };
      exchange(put0, from(j ^ 1));
      keep_larger(side == 0, std::true_type());
      bitonic_merge<M, DescPos>(key);
      exchange(put1, from(3 - j) + XCH);
      keep_larger(top_half, std::true_type());
      exchange(put0, from(j ^ 1));
      // ranks beyond keep + 2 are not looked at
      const bool wanted = j * M < keep_cfg + 3;
      uint32_t es[M], ei[M];
      if (wanted) {
        keep_larger(side == 0, std::false_type());
        bitonic_merge<M, DescPos>(key);
#pragma unroll
        for (int i = 0; i < M; ++i) lds64(slot((int)(key[i] & 255u)), es[i], ei[i]);
      }
      if (sampling)
        for (int w = j; w < ((v + 31) >> 5); w += TPR) sts32(bits + (uint32_t)w * WORD_PITCH, 0u);
      quarter_sync(quarter);                                 // everyone has read
      if (wanted) {
#pragma unroll
        for (int i = 0; i < M; ++i) sts64(slot(j * M + i), es[i], ei[i]);
      }
    }
    PH_LAP(4);
    quarter_sync(quarter);

    // ===== cuts: thread 0 rank k, thread 1 rank k + m ====================================================
    // Entries that agree in all 23 bits may stand in the wrong order.  That matters only next to a cut: a pair
    // is put right, three in a row are left to the slow path.
    const int n_excl = p.m > 0 ? T : kk;                     // route + near-miss ids of the row
    if (top_half) {
      const int rank = j == 0 ? kk : p.m > 0 ? T : 0;        // (no near-miss sentinels: no second cut)
      bool open = bad;                                       // this cut could not be settled
      if (have && rank > 0 && !bad) {
        uint32_t s_[6], id_[6], q[6];                        // ranks rank - 3 .. rank + 2 (from 0)
#pragma unroll
        for (int e = 0; e < 6; ++e) {
          const int at = rank - 3 + e;
          lds64(slot(min(max(at, 0), CAP - 1)), s_[e], id_[e]);
          q[e] = at < 0 ? 0xFFFFFFF0u - (uint32_t)e : fixed_bits(__uint_as_float(s_[e]), tau, scale);
        }
        const uint32_t none = fixed_bits(ninf, tau, scale);
        auto f = [&](int e) -> float { return __uint_as_float(s_[e]); };
        float last_in = f(2), first_out = f(3);
        if (q[2] > q[3]) {
          if (j == 0) {
            if (q[1] == q[2]) { last_in = fminf(f(1), f(2)); open |= q[0] == q[2]; }
            if (q[3] == q[4] && q[3] != none) { first_out = fmaxf(f(3), f(4)); open |= q[5] == q[3] || p.m == 1; }
          }
        } else if (q[3] != none) {
          open |= q[1] == q[2] || q[4] == q[3];
          if (!open && (f(3) > f(2) || (f(3) == f(2) && id_[3] < id_[2]))) {
            sts64(slot(rank - 1), s_[3], id_[3]);
            sts64(slot(rank), s_[2], id_[2]);
            last_in = f(3); first_out = f(2);
          }
        }
        if (force_hard && g % 5 == 0) open = true;           // test hook: exercise the slow path
        if (j == 0 && !open) {                               // (overwritten by the slow path if it takes the row)
          p.kth[g] = last_in;
          p.margin[g] = v > kk ? last_in - first_out : pinf;
        }
      }
      ctl->cnt[j][r] = open ? 1 : 0;
    }
    quarter_sync(quarter);
    const bool hard = (ctl->cnt[0][r] | ctl->cnt[1][r]) != 0;
    const bool go = have && !hard;
    if (j == 0 && hard) {
      const uint32_t idx = atomicAdd(&ctl->hard_n, 1u);
      ctl->hard_rows[idx] = (uint8_t)r;
      ctl->hard_slot[r] = (int8_t)idx;
    }
    PH_LAP(5);

    // ===== copy-out: thread 0 the route, thread 1 the near-miss sentinels, the other two the draws ========
    int32_t* const sent = p.sentinels + (size_t)g * p.sw;
    if (top_half) {
      const int width = j == 0 ? p.k : p.m, n = !go ? 0 : j == 0 ? kk : n_excl - kk;
      const uint32_t src = slot(j == 0 ? 0 : kk);
      int32_t* const dst = j == 0 ? p.routes + (size_t)g * p.k : sent;
      const bool vec = j == 0 ? (p.k & 3) == 0 : ((p.m | p.sw) & 3) == 0;
      if (width > 0) {
        if (width <= 16) order_ids<16>(src, n, dst, width, vec, go);
        else if (width <= 32) order_ids<32>(src, n, dst, width, vec, go);
        else if (NG == 1 || CTAS == 2 || width <= 64) order_ids<64>(src, n, dst, width, vec, go);
        else if constexpr (NG > 1 && CTAS == 1) order_ids<128>(src, n, dst, width, vec, go);
      }
    } else if (sampling) {
#pragma unroll 8
      for (int e = side; e < (go ? n_excl : 0); e += 2) {
        const uint32_t id = lds32(slot(e) + 4u);
        asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(bits + (id >> 5) * WORD_PITCH), "r"(1u << (id & 31)) : "memory");
      }
      drawers_sync(quarter);                                 // the bitmap is complete
    }
    PH_LAP(6);
    // ===== sentinels (Section 3.1 items 2, 3): the row's third thread ====================================
    if (j == 2 && sampling)
      draw_sentinels<WORD_PITCH, SLOT_PITCH, CAP>(p, bits, col, g, v, n_excl, layer, lane, go);
    PH_LAP(7);
  } while (false);

  // ===== slow path: rows the fast path could not settle ============================================
  // One more sweep per batch of hard_slots rows stores their complete score rows (as order keys)
  // over the column area; a warp per row then runs the exact radix select on them.
  fence_proxy_async_smem();                                // the ring was written by ordinary stores
  tc_fence_before();                                       // (and the accumulators by the exchanges)
  __syncthreads();
  const int n_hard = ctl->abort_flag ? 0 : (int)ctl->hard_n;
  const int nk_words = (p.n_k + 31) / 32;
  const int hard_slots = min(MAX_HARD, (CAP * (int)SLOT_PITCH / 4 - SEL_WARPS * (256 + nk_words)) / (nk_words * 32));
  int next_gt = 2 * n_tiles;
  for (int done = 0; done < n_hard; done += hard_slots) {
    // barrier: the previous batch's rows and scratch are free again; the vote makes the
    // decision to stop after a timed-out wait the same for every thread
    if (__syncthreads_or((int)ctl->abort_flag)) break;
    if (warp == 0) {
      produce(next_gt, n_tiles, next_gt);
    } else if (warp == 1) {
      issue(next_gt, n_tiles);
    } else {
      const int hs = row >= 0 ? (int)ctl->hard_slot[r] - done : -1;
      const bool mine = hs >= 0 && hs < hard_slots && ctl->hard_slot[r] >= 0;
      const uint32_t srow = smem_u32(s_col) + (uint32_t)max(hs, 0) * (uint32_t)(nk_words * 128);
#pragma unroll 1
      for (int t = pair; t < n_tiles; t += 2) {
        const int gt = next_gt + t, col0 = t * BN + side * SLICE;
        if (!tile_wait(gt)) break;
        uint32_t acc[SLICE];
        tmem_ld_32x32(acc_addr(gt), acc);
        if (mine) {
#pragma unroll
          for (int i = 0; i < SLICE; ++i)
            if (col0 + i < v) sts32(srow + (uint32_t)(col0 + i) * 4u, rr_order_key(__uint_as_float(acc[i])));
        }
        __syncwarp();
        tile_release(gt);
      }
    }
    next_gt += n_tiles;
    __syncthreads();
    if (is_sel && !ctl->abort_flag) {
      const int sw = warp - 2;
      uint32_t* scratch = (uint32_t*)s_col + (size_t)hard_slots * nk_words * 32 + sw * (256 + nk_words);
      for (int hs = sw; hs < hard_slots && done + hs < n_hard; hs += SEL_WARPS) {
        const int rr = ctl->hard_rows[done + hs];
        const int hg = row_list ? row_list[seg_lo + tm * own + rr] : prob * p.n_q + tm * own + rr;
        const int hv = rr_valid_count(hg - prob * p.n_q, p.n_k, p.causal, p.causal_offset);
        const uint32_t* keys = (const uint32_t*)s_col + (size_t)hs * nk_words * 32;
        warptopk::route_row(p, keys, scratch, scratch + 256, hg, hv, layer, lane);
        __syncwarp();
      }
    }
  }

  // TMEM must not be freed while an MMA can still write to it: after a wait that gave up the
  // consumers no longer vouch for that, so the issuer waits (bounded) for its own MMAs
  // (when no wait gave up, every issued tile has been waited for by the consumers: nothing is pending)
  if (warp == 1 && ctl->abort_flag) {
    umma_commit_warp(&ctl->drain);
    for (uint32_t it = 0; it < kSpinLimit && !mbar_try_wait(&ctl->drain, 0); ++it) __nanosleep(64);
  }
  tc_fence_before();
  __syncthreads();
#ifdef RR_PHASE_TIMING
  if (tid == 0) { PH_CNT(14, clock64() - cta_t0_); PH_CNT(15, 1); PH_CNT(16, n_hard); PH_CNT(17, n_hard > 0); }
#endif
  if (warp == 1) {                                         // the warp that allocated
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
  if (tid == 0 && ctl->abort_flag) atomicOr(p.status, RR_STATUS_TIMEOUT);
  if (tested && tid == 0) {
    atomicAdd(&p.counters[RR_CNT_FLAGGED_ROWS], (unsigned long long)ctl->flagged);
    atomicAdd(&p.counters[RR_CNT_CAND_PAIRS], (unsigned long long)ctl->cand);
    atomicAdd(&p.counters[RR_CNT_FULL_PAIRS], ctl->full_pairs);
  }
  if (!TEST && !row_list_arg) rr_pdl_wait();               // complete only after the predecessor is
}

constexpr int VARIANTS = 8, CAPS[VARIANTS] = {48, 64, 80, 80, 88, 104, 128, 160}, CTAS_OF[VARIANTS] = {2, 2, 2, 2, 2, 1, 1, 1};

template <int D, bool TEST>
rr_quad_kernel quad_kernels(int variant) {
  static const rr_quad_kernel table[VARIANTS] = {
      route_quad_kernel<D, 1, CAPS[0], CTAS_OF[0], TEST>, route_quad_kernel<D, 1, CAPS[1], CTAS_OF[1], TEST>,
      route_quad_kernel<D, 1, CAPS[2], CTAS_OF[2], TEST>, route_quad_kernel<D, 2, CAPS[3], CTAS_OF[3], TEST>,
      // (a column of 88 entries fits twice at d = 64 only)
      route_quad_kernel<D, 2, D == 64 ? CAPS[4] : CAPS[3], 2, TEST>, route_quad_kernel<D, 2, CAPS[5], CTAS_OF[5], TEST>,
      route_quad_kernel<D, 2, CAPS[6], CTAS_OF[6], TEST>, route_quad_kernel<D, 2, CAPS[7], CTAS_OF[7], TEST>};
  return table[variant];
}

}  // namespace
