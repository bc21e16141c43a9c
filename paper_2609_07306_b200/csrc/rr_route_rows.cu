// Full routing of a set of rows in ONE kernel, two sweeps over the key chunks: score GEMM on
// the tensor cores (Eq. 1), per-row TopK (Eq. 2), near-miss sentinels (Section 3.1 item 1),
// k-th score and margin (Section 3.3), mandatory global and random sentinels (Section 3.1
// items 2, 3) -- the score matrix never leaves the SM.
//
// One CTA owns 128 query rows of one problem (consecutive rows at an anchor; a segment of the
// compacted refresh list at a relay, Section 4.2) and walks the key chunks in tiles of 64,
// stopping at the last chunk any of its rows may select.
//   warp 0    : TMA producer (Kc tiles, 128-byte swizzle, one copy per tile, a ring of 3)
//   warp 1    : issues tcgen05.mma (M=128, N=64, K=16) into a ring of 3 TMEM
//               accumulators; the Qc tile is the MMA's A operand in TMEM
//   warps 2-9 : selection, TWO THREADS PER QUERY ROW: thread j of a row takes the tiles t with
//               t % 2 == j (two tcgen05.ld 32x32b hand it the tile's 64 scores of its row).
// What bounds this kernel is the instruction issue of the selection and the latency of its
// phases, not the GEMM (which is therefore simply issued twice); everything is laid out so that
// TWO CTAs fit an SM (97 KB of shared memory, 96 registers, 256 TMEM columns each) and one CTA's
// latency-bound phases hide behind the other's sweeps.  It serves keep = k + max(m, 1) <= 28; more kept chunks make its
// phases so long that four threads per row are better (rr_route_quad.cuh; the figures are there).
//
// Sweep 1 (threshold before filtering): scores are cut to bf16 (the upper half of the float, one
// byte permute per two scores) and each thread keeps packed running maxima of 64 groups of
// columns (64 positions in a tile): 128 groups per row.  The keep-th
// largest group maximum, keep = k + max(m, 1), has keep distinct scores of the row at or above it:
// a valid lower bound tau of the row's keep-th largest score (about 1.1 keep scores pass it).  The
// maxima are sorted in registers, two lists at a time (packed compare-exchange); each thread takes
// its share of keep from the top of its own two lists (binary search), and the shares are shifted
// once towards the thread that has more above the lower of the two bounds.  Any shares give a
// valid bound; these are close to the exact rank and follow the data when one thread's tiles hold
// most of the row's best chunks.
// Sweep 2: each thread appends its scores >= tau as {score, chunk id} to the row's column of CAP
// entries in shared memory, thread 0 upwards from the bottom, thread 1 downwards from the top.
// Cut: each thread sorts one half of the column in registers, by keys that carry 23 bits of
// fixed point over [tau, row maximum] and the slot, and writes the entries back in rank order
// (which is then checked against the exact scores).  Thread 0 finds rank k, thread 1 rank k + m,
// by binary search over the two sorted halves; route and near-miss ids are gathered, ordered by
// chunk id in registers and leave with 16-byte stores.  The second thread of the row then draws
// the sentinels against the row's bitmap of excluded chunks.
// Rows the fast path cannot finish exactly (the column overflowed, three scores out of order
// within the fixed-point resolution)
// are handed to an exact slow path: one more sweep stores their complete score rows in shared
// memory, and a warp per row runs the radix select of the two-pass path.  Every mbarrier wait is
// bounded.
#include "rr_common.cuh"
#include "rr_networks.cuh"
#include "rr_route_select.cuh"
#include "rr_sm100.cuh"
#include "rr_warp_topk.cuh"

using namespace sm100;
using namespace rr_select;

namespace {

constexpr int BM = 128, BN = 64, ACC_STAGES = 3;
constexpr int TPR = 2, SLICE = 32;                 // threads per row, columns per TMEM load
constexpr int SEL_WARPS = TPR * (BM / 32);
constexpr int NT = (2 + SEL_WARPS) * 32;
constexpr int TMEM_COLS = 256, A_COL = ACC_STAGES * BN;   // Qc tile behind the accumulators
constexpr int MAX_KEEP = 28;                       // largest k + max(m, 1) that a column of 48 entries serves
constexpr int MAX_STAGES = ACC_STAGES;             // of the Kc ring: tiles of 16 KB (d = 128) or 8 KB (d = 64)
constexpr int MAX_HARD = 24;                       // score rows held at once by the slow path
constexpr uint32_t SLOT_PITCH = BM * 8;            // bytes between entries of a row's column
constexpr uint32_t WORD_PITCH = BM * 4;            // [word][row] areas

struct Ctl {
  uint64_t full[MAX_STAGES], acc_full[ACC_STAGES], acc_empty[ACC_STAGES], drain;
  uint32_t tmem_base, abort_flag, hard_n, pad_;
  uint8_t cnt[TPR][BM];                 // survivors per thread
  uint8_t cut[TPR][BM];                 // entries of the first half column in the top k / top k + m; bit 7: slow path
  uint8_t hard_rows[BM];                // rows handed to the slow path, in registration order
  int8_t hard_slot[BM];                 // position of a row in hard_rows, -1 = none
};
constexpr int CTL_BYTES = 1024;
constexpr int MAIL = 20;                // slot of a half column through which its thread gets the other's messages
static_assert(sizeof(Ctl) <= CTL_BYTES, "control block too large");

// the two warps that share a quarter of the rows (64 threads), barrier ids 1..4
__device__ __forceinline__ void quarter_sync(int quarter) {
  asm volatile("bar.sync %0, 64;" ::"r"(quarter + 1) : "memory");
}

template <int I, bool EDGE>
__device__ __forceinline__ void filter_all(uint32_t& w, const uint32_t (&acc)[SLICE], float tau, uint32_t col0,
                                           uint32_t step, int v) {
  if constexpr (I < SLICE) {
    filter_one<I, EDGE>(w, acc[I], tau, col0, step, v);
    filter_all<I + 1, EDGE>(w, acc, tau, col0, step, v);
  }
}

// ---- gather and order -------------------------------------------------------------------------
// n0 ids from entries e0, e0 + 1, ... of the row's column and n1 ids from entries e1, ...: ordered
// by chunk id and written to dst [0, width), -1 behind the last one.  With `mark`, the ids' bits
// are set in the row's bitmap at bits + word * WORD_PITCH.
template <int N>
__device__ __forceinline__ void gather_ids(uint32_t col, int e0, int n0, int e1, int n1, uint32_t bits, bool mark,
                                           int32_t* dst, int width, bool vec, bool on) {
  constexpr uint32_t NONE = 0xFFFFu;
  uint32_t x[N];
  const int n = n0 + n1;
  const uint32_t a0 = col + (uint32_t)e0 * SLOT_PITCH + 4u, a1 = col + (uint32_t)(e1 - n0) * SLOT_PITCH + 4u;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    uint32_t id = NONE;        // (orders behind every id)
    if (i < n) id = lds32((i < n0 ? a0 : a1) + (uint32_t)i * SLOT_PITCH);
    x[i] = id;
    if (mark && i < n)
      asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(bits + (id >> 5) * WORD_PITCH), "r"(1u << (id & 31)) : "memory");
  }
  // ids fit 16 bits: two half lists are sorted at a time, then merged
  uint32_t h[N / 2];
#pragma unroll
  for (int i = 0; i < N / 2; ++i) h[i] = __byte_perm(x[i], x[i + N / 2], 0x5410);
  OESort<0, N / 2, AscU2, N / 2>::run(h);
#pragma unroll
  for (int i = 0; i < N / 2; ++i) { x[i] = h[i] & 0xFFFFu; x[i + N / 2] = h[i] >> 16; }
  OEMerge<0, N, 1, AscPos, N>::run(x);
  if (!on) return;
#pragma unroll
  for (int i = 0; i < N; ++i) x[i] = i < n ? x[i] : 0xFFFFFFFFu;
#pragma unroll
  for (int q = 0; q < N; q += 4) {
    if (q < width) {
      if (vec) {
        *reinterpret_cast<uint4*>(dst + q) = make_uint4(x[q], x[q + 1], x[q + 2], x[q + 3]);
      } else {
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (q + t < width) dst[q + t] = (int32_t)x[q + t];
      }
    }
  }
}

#ifdef RR_PHASE_TIMING
__device__ unsigned long long g_rows_phase[32];
#define PH_T0() long long ph_t0_ = clock64()
#define PH_LAP(i) do { const long long t1_ = clock64(); if ((threadIdx.x & 31) == 0) atomicAdd(&g_rows_phase[i], (unsigned long long)(t1_ - ph_t0_)); ph_t0_ = t1_; } while (0)
#define PH_CNT(i, val_) atomicAdd(&g_rows_phase[i], (unsigned long long)(val_))
#else
#define PH_CNT(i, val_) do {} while (0)
#define PH_T0() do {} while (0)
#define PH_LAP(i) do {} while (0)
#endif

constexpr int CAP = 48, STAGES = ACC_STAGES;         // entries of a row's column, tiles of the Kc ring
template <int D>
__global__ void __launch_bounds__(NT, 2)
route_rows_kernel(RRParams p, const __nv_bfloat16* __restrict__ qc,
                  const __grid_constant__ CUtensorMap tmap_k, const int32_t* __restrict__ row_list_arg,
                  uint32_t layer, int hooks, int ring_bytes, int cta_stride) {
  constexpr int KH = D / 64;                               // K-halves of a tile
  constexpr int TILE = BN * D * 2;
  constexpr int M = CAP / 2;                               // entries per half column
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
      mbar_init(&ctl->acc_empty[s], SEL_WARPS / TPR);      // one arrival per warp that reads the tile
    }
    mbar_init(&ctl->drain, 1);
    ctl->abort_flag = 0;
    ctl->hard_n = 0;
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
  if (row_list_arg) rr_pdl_wait();
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
  const bool force_hard = hooks & 1, force_timeout = hooks & 2;      // test hooks
  // Row tiles are handed out heaviest first (under the causal mask the last tile of a problem
  // walks the most key chunks), so the tail of the grid is made of the short ones and, where a refresh
  // list is short, of the CTAs that find no tile: in front they kept the SMs from the
  // others (17 % of 256 x 1024 rows on the list: 130 -> 120 us).
  const int seg_lo = row_list ? list_lo : 0, seg_hi = row_list ? list_hi : p.n_q;
  const int tm = (seg_hi - seg_lo + BM - 1) / BM - 1 - (int)(blockIdx.x / p.P);
  if (tm < 0) { if (!row_list_arg) rr_pdl_wait(); return; }          // nothing to do (uniform per CTA)

  // row of the CTA's tile -> query row of the problem and global row id; -1 = no row
  auto locate = [&](int rr, int& row_out, int& g_out) {
    const int local = tm * BM + rr;
    row_out = -1; g_out = 0;
    if (row_list) {
      if (seg_lo + local < seg_hi) { g_out = row_list[seg_lo + local]; row_out = g_out - prob * p.n_q; }
    } else if (local < p.n_q) {
      row_out = local; g_out = prob * p.n_q + local;
    }
  };
  // ---- selection-side geometry (meaningful for warps 2..) -------------------------------------
  const int quarter = warp & 3, j = (warp - 2) >> 2;
  const int r = quarter * 32 + lane;                       // row inside the CTA
  const bool is_sel = warp >= 2;
  // ---- the Qc tile goes to TMEM: a thread of row r loads its part of the row (two bf16 per
  // 32-bit word, as they lie in memory; refresh rows are not contiguous, so this is also the
  // gather) and stores it to TMEM lane r, where the MMA reads its A operand; rows without a
  // query are 0.  The loads are issued first so that their latency overlaps the rest of the set-up.
  constexpr int QT = D == 128 ? 2 : 1, QW = 32;            // threads per row, 32-bit words per thread
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
  if (warp == 1) {
    tmem_alloc(&ctl->tmem_base, TMEM_COLS);
    rr_pdl_trigger();                                      // (not before: the successor takes TMEM, too)
  }
  // The Kc loads depend on nothing but the number of key tiles (from the tile's last row: rows
  // ascend inside a tile), and the ring's stages are all free: the producer fills the ring before
  // the CTA's first barrier, while the Qc rows are on their way.
  const int last_local = min(seg_hi - seg_lo, (tm + 1) * BM) - 1;
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
    tmem_st_32x32(ctl->tmem_base + ((uint32_t)(quarter * 32) << 16) + A_COL + j * QW, qv);
    tmem_st_wait();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  volatile uint32_t* abort_flag = &ctl->abort_flag;

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
  const bool routed = row >= 0 && (!dense_refresh || p.flags[g] != 0);     // this row is (re)routed here
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
  auto acc_addr = [&](int gt, int half) -> uint32_t { return acc_lane + (uint32_t)((gt % ACC_STAGES) * BN + half * SLICE); };

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
      const int ntm = (nhi - nlo + BM - 1) / BM - 1 - nb / p.P;
      for (int i = lane; i < BM && ntm >= 0; i += 32) {
        const int local = ntm * BM + i;
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
    // accumulators back.  Both of its warps come here, so nobody waits for them at its barriers
    // (3 % of 256 x 256 rows on the list: 24.9 -> 24.1 us).
#pragma unroll 1
    for (int first = 0; first < 2 * n_tiles; first += n_tiles)
#pragma unroll 1
      for (int t = j; t < n_tiles && tile_wait(first + t); t += TPR) tile_release(first + t);
  } else {
    PH_T0();
#ifdef RR_PHASE_TIMING
    if (lane == 0) PH_CNT(12, ph_t0_ - cta_t0_);
#endif
    const int keep_cfg = p.k + max(p.m, 1);
    const int T = min(keep_cfg, v), kk = min(p.k, v);        // ranks that the row can fill
    // ===== sweep 1: packed group maxima =============================================================
    float tau;
    float scale;
    {
      uint32_t mx[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) mx[i] = 0xff80ff80u;
#pragma unroll 1
      for (int t = j; t < n_tiles; t += TPR) {
        if (!tile_wait(t)) break;
#pragma unroll
        for (int h = 0; h < BN / SLICE; ++h) {
          const int col0 = t * BN + h * SLICE;
          uint32_t acc[SLICE];
          if (col0 < vmaxw) tmem_ld_32x32(acc_addr(t, h), acc);
          if (h == BN / SLICE - 1) tile_release(t);
          if (col0 + SLICE <= vminw) {
#pragma unroll
            for (int i = 0; i < SLICE / 2; ++i) {
              const uint32_t pk = __byte_perm(acc[2 * i], acc[2 * i + 1], 0x7632);   // upper halves: bf16, cut
              asm("max.bf16x2 %0, %0, %1;" : "+r"(mx[h * (SLICE / 2) + i]) : "r"(pk));
            }
          } else if (col0 < vmaxw) {                         // some row's last chunk lies inside
            const int nv = v - col0;
#pragma unroll
            for (int i = 0; i < SLICE / 2; ++i) {
              const uint32_t pk = __byte_perm(acc[2 * i], acc[2 * i + 1], 0x7632);
              const uint32_t pm = 2 * i + 1 < nv ? pk : (pk & 0xffffu) | 0xff800000u;
              asm("max.bf16x2 %0, %0, %1;" : "+r"(mx[h * (SLICE / 2) + i]) : "r"(2 * i < nv ? pm : 0xff80ff80u));
            }
          }
        }
      }
      PH_LAP(0);
      // two sorted lists of 32
      OESort<0, 32, DescBF2, 32>::run(mx);
      // published in this thread's (still unused) half of the column: list A in the low halves of
      // the words, list B in the high halves, two words to a slot
      const uint32_t pub = col + (uint32_t)(j * M) * SLOT_PITCH;
#pragma unroll
      for (int i = 0; i < 32; i += 2) sts64(pub + (uint32_t)(i / 2) * SLOT_PITCH, mx[i], mx[i + 1]);
      PH_LAP(1);
      auto A = [&](int i) -> float { return __uint_as_float(lds32(pub + (uint32_t)(i >> 1) * SLOT_PITCH + (uint32_t)(i & 1) * 4u) << 16); };
      auto B = [&](int i) -> float { return __uint_as_float(lds32(pub + (uint32_t)(i >> 1) * SLOT_PITCH + (uint32_t)(i & 1) * 4u) & 0xffff0000u); };
      // the share-th largest of this thread's maxima (+inf for an empty share)
      auto share_bound = [&](int share) -> float {
        const int a = rank_split<32>(share, A, B), b = share - a;
        const float la = A(max(a - 1, 0)), lb = B(max(b - 1, 0));
        return fminf(a > 0 ? la : pinf, b > 0 ? lb : pinf);
      };
      // shares in proportion to the threads' non-empty groups (64 at most)
      const int q = v / BN, rem = v % BN;
      const int c0 = min(64, ((q + 1) / 2) * BN + ((q & 1) == 0 ? rem : 0));
      const int c1 = min(64, (q / 2) * BN + ((q & 1) == 1 ? rem : 0));
      int share0 = c1 == 0 ? T : c1 == 64 ? (T + 1) / 2 : (int)((float)(T * c0) / (float)(c0 + c1) + 0.5f);
      share0 = min(c0, max(share0, T - c1));
      int share = j == 0 ? share0 : T - share0;
      float bound = share_bound(share);
      // messages: word 0 of the other thread's mail slot = this thread's bound, word 1 = the shift
      const uint32_t mail_in = col + (uint32_t)(j * M + MAIL) * SLOT_PITCH, mail_out = col + (uint32_t)((1 - j) * M + MAIL) * SLOT_PITCH;
      float top = fmaxf(A(0), B(0));
      sts32(mail_out, __float_as_uint(bound));
      quarter_sync(quarter);
      const float other = ldsf(mail_in);
      {                                                      // (the other list is still there)
        const uint32_t w = lds32(col + (uint32_t)((1 - j) * M) * SLOT_PITCH);
        top = fmaxf(top, fmaxf(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)));
      }
      // the thread with the higher bound counts its maxima at or above the other one's and takes
      // half of the surplus
      int ca = 0, cb = 0;
#pragma unroll
      for (int s = 16; s >= 1; s >>= 1) {
        ca += A(ca + s - 1) >= other ? s : 0;
        cb += B(cb + s - 1) >= other ? s : 0;
      }
      ca += A(ca) >= other ? 1 : 0; cb += B(cb) >= other ? 1 : 0;   // ca, cb <= 31 here
      int shift = max(0, (ca + cb - share) >> 1);
      if (j == 1) shift = -shift;
      if (bound > other) sts32(mail_out + 4u, (uint32_t)shift);
      quarter_sync(quarter);
      if (bound < other) shift = (int)lds32(mail_in + 4u);
      if (bound == other) shift = 0;
      share0 = min(min(c0, T), max(share0 + shift, max(T - c1, 0)));
      share = j == 0 ? share0 : T - share0;
      bound = share_bound(share);
      sts32(mail_out, __float_as_uint(bound));
      // the lists are done with: the half column is cleared (empty slots read as -inf in the sort), the
      // mail slot once its last message has been read
#pragma unroll
      for (int e = 0; e < M; ++e)
        if (e != MAIL) sts64(col + (uint32_t)(j * M + e) * SLOT_PITCH, 0xff800000u, 0u);
      quarter_sync(quarter);
      tau = fminf(bound, ldsf(mail_in));
      sts64(mail_in, 0xff800000u, 0u);
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
    const uint32_t step = j == 0 ? SLOT_PITCH : 0u - SLOT_PITCH;
    const uint32_t own = j == 0 ? col : col + (uint32_t)(CAP - 1) * SLOT_PITCH;    // this thread's entry 0
    uint32_t waddr = own;
#pragma unroll 1
    for (int t = j; t < n_tiles; t += TPR) {
      const int gt = n_tiles + t;
      if (!tile_wait(gt)) break;
      uint32_t acc[2][SLICE];
      if (t * BN < vmaxw) tmem_ld_32x64(acc_addr(gt, 0), acc[0], acc[1]);
      tile_release(gt);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int col0 = t * BN + h * SLICE;
        if (col0 < vmaxw) {
          if (!__any_sync(FULL, (j == 0 ? waddr - own : own - waddr) > (uint32_t)(CAP - SLICE) * SLOT_PITCH)) {
            if (col0 + SLICE <= vminw) filter_all<0, false>(waddr, acc[h], tau, (uint32_t)col0, step, v);
            else filter_all<0, true>(waddr, acc[h], tau, (uint32_t)col0, step, v);
          } else {                // the column may run full inside this slice
            int n = (int)((j == 0 ? waddr - own : own - waddr) / SLOT_PITCH);
#pragma unroll
            for (int i = 0; i < SLICE; ++i) {
              const float s = __uint_as_float(acc[h][i]);
              if (s >= tau && n < CAP && col0 + i < v) { sts64(waddr, acc[h][i], (uint32_t)(col0 + i)); waddr += step; ++n; }
            }
          }
        }
      }
    }
    ctl->cnt[j][r] = (uint8_t)((j == 0 ? waddr - own : own - waddr) / SLOT_PITCH);
    PH_LAP(3);
    quarter_sync(quarter);

    // ===== sort: each thread one half of the column, in rank order =======================================
    const bool have = alive && routed;
    const int n = (int)ctl->cnt[0][r] + (int)ctl->cnt[1][r];
    bool bad = have && (n > CAP || n < T);                   // (too few only after a wait gave up)
    const uint32_t half = col + (uint32_t)(j * M) * SLOT_PITCH;
    {
      // equal keys keep the ascending chunk ids of their thread: slots ascend with the ids in thread
      // 0's half, descend in thread 1's
      const uint32_t flip = j == 0 ? 255u : 0u;
      uint32_t key[M];
#pragma unroll
      for (int i = 0; i < M; ++i)
        key[i] = fixed_bits(ldsf(half + (uint32_t)i * SLOT_PITCH), tau, scale) * 256u + (uint32_t)(j == 0 ? 255 - i : i);
      OESort<0, pow2_at_least(M), DescPos, M>::run(key);
      uint32_t es[M], ei[M];
#pragma unroll
      for (int i = 0; i < M; ++i) lds64(half + ((key[i] & 255u) ^ flip) * SLOT_PITCH, es[i], ei[i]);
      bool wrong = false;
#pragma unroll
      for (int i = 0; i + 1 < M; ++i)
        wrong |= !(__uint_as_float(es[i]) > __uint_as_float(es[i + 1]) || (es[i] == es[i + 1] && ei[i] <= ei[i + 1]));
#pragma unroll
      for (int i = 0; i < M; ++i) sts64(half + (uint32_t)i * SLOT_PITCH, es[i], ei[i]);
      // Keys that agree in all 23 bits leave their two entries in slot order: about one row in 5000
      // has such a pair.  One pass of exchanges repairs pairs; what is out of order after it (a run of
      // three) is left to the slow path.
      if (__any_sync(FULL, have && wrong)) {
        wrong = false;
        uint32_t s0, i0;
        lds64(half, s0, i0);
        float above = pinf;
        uint32_t above_id = 0;
        auto follows = [&](uint32_t sc, uint32_t id) {                 // does not rank before its predecessor
          wrong |= __uint_as_float(sc) > above || (__uint_as_float(sc) == above && id < above_id);
          above = __uint_as_float(sc); above_id = id;
        };
#pragma unroll 1
        for (int i = 1; i < M; ++i) {
          uint32_t s1, i1;
          lds64(half + (uint32_t)i * SLOT_PITCH, s1, i1);
          const bool ok = __uint_as_float(s0) > __uint_as_float(s1) || (s0 == s1 && i0 <= i1);
          const uint32_t fs = ok ? s0 : s1, fi = ok ? i0 : i1;         // goes to slot i - 1
          sts64(half + (uint32_t)(i - 1) * SLOT_PITCH, fs, fi);
          follows(fs, fi);
          s0 = ok ? s1 : s0; i0 = ok ? i1 : i0;
        }
        sts64(half + (uint32_t)(M - 1) * SLOT_PITCH, s0, i0);
        follows(s0, i0);
      }
      bad |= have && wrong;
    }
    // the bitmap of excluded chunks starts empty (the Kc ring is idle once the last tile of sweep 2
    // has been consumed)
    const bool sampling = p.r > 0 || p.n_global > 0;
    if (sampling)
      for (int w = j; w < ((v + 31) >> 5); w += TPR) sts32(bits + (uint32_t)w * WORD_PITCH, 0u);
    PH_LAP(4);
    quarter_sync(quarter);

    // ===== cuts: thread 0 rank k, thread 1 rank k + m ====================================================
    const int rank = j == 0 ? kk : p.m > 0 ? T : kk;         // m = 0: no near-miss sentinels
    {
      // entry a of the first half ranks before entry b of the second: higher score, or equal score and
      // smaller chunk id
      int lo = max(0, rank - M), hi = min(rank, M);
#pragma unroll 1
      for (int s = 1; s <= M; s *= 2) {
        const int mid = (lo + hi) >> 1;
        uint32_t sa, ia, sb, ib;
        lds64(col + (uint32_t)min(mid, M - 1) * SLOT_PITCH, sa, ia);
        lds64(col + (uint32_t)(M + min(max(rank - mid - 1, 0), M - 1)) * SLOT_PITCH, sb, ib);
        const float fa = __uint_as_float(sa), fb = __uint_as_float(sb);
        const bool more = fa > fb || (fa == fb && ia < ib), step_ = lo < hi;
        lo = step_ && more ? mid + 1 : lo;
        hi = step_ && !more ? mid : hi;
      }
      const int a = lo, b = rank - a;
      auto score = [&](int slot) -> float { return ldsf(col + (uint32_t)slot * SLOT_PITCH); };
      if (force_hard && have && g % 5 == 0) bad = true;      // test hook: exercise the slow path
      ctl->cut[j][r] = (uint8_t)(a | (bad ? 128 : 0));
      if (j == 0) {
        const float la = score(max(a - 1, 0)), lb = score(M + min(max(b - 1, 0), M - 1));
        const float xa = score(min(a, M - 1)), xb = score(M + min(max(b, 0), M - 1));
        const float last_in = fminf(a > 0 ? la : pinf, b > 0 ? lb : pinf);
        const float first_out = fmaxf(a < M ? xa : ninf, b < M ? xb : ninf);
        if (have && !bad) {                                  // (overwritten by the slow path if it takes the row)
          p.kth[g] = last_in;
          p.margin[g] = v > kk ? last_in - first_out : pinf;
        }
      }
    }
    quarter_sync(quarter);
    const int a_k = ctl->cut[0][r] & 127, a_d = ctl->cut[1][r] & 127;
    const bool hard = ((ctl->cut[0][r] | ctl->cut[1][r]) & 128) != 0;
    const bool go = have && !hard;
    if (j == 0 && hard) {
      const uint32_t idx = atomicAdd(&ctl->hard_n, 1u);
      ctl->hard_rows[idx] = (uint8_t)r;
      ctl->hard_slot[r] = (int8_t)idx;
    }
    PH_LAP(5);

    // ===== copy-out: thread 0 the route, thread 1 the near-miss sentinels ===============================
    const int n_excl = p.m > 0 ? T : kk;                     // route + near-miss ids of the row
    int32_t* const sent = p.sentinels + (size_t)g * p.sw;
    {
      const int e0 = j == 0 ? 0 : a_k, n0 = j == 0 ? a_k : a_d - a_k;
      const int e1 = M + (j == 0 ? 0 : kk - a_k), n1 = j == 0 ? kk - a_k : (n_excl - a_d) - (kk - a_k);
      const int width = j == 0 ? p.k : p.m;
      int32_t* const dst = j == 0 ? p.routes + (size_t)g * p.k : sent;
      const bool vec = j == 0 ? (p.k & 3) == 0 : ((p.m | p.sw) & 3) == 0;
      const int m0 = go ? n0 : 0, m1 = go ? n1 : 0;
      if (width > 0) {
        if (width <= 16) gather_ids<16>(col, e0, m0, e1, m1, bits, sampling, dst, width, vec, go);
        else gather_ids<32>(col, e0, m0, e1, m1, bits, sampling, dst, width, vec, go);
      }
    }
    PH_LAP(6);
    if (sampling) quarter_sync(quarter);                     // the bitmap is complete
    // ===== sentinels (Section 3.1 items 2, 3): the row's second thread ===================================
    if (j == 1 && sampling)
      draw_sentinels<WORD_PITCH, SLOT_PITCH, CAP>(p, bits, col, g, v, n_excl, layer, lane, go);
    PH_LAP(7);
  }

  // ===== slow path: rows the fast path could not settle ============================================
  // One more sweep per batch of hard_slots rows stores their complete score rows (as order keys)
  // over the column area; a warp per row then runs the exact radix select on them.
  fence_proxy_async_smem();                                // the ring was written by ordinary stores
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
      for (int t = j; t < n_tiles; t += TPR) {
        const int gt = next_gt + t;
        if (!tile_wait(gt)) break;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          const int col0 = t * BN + h * SLICE;
          uint32_t acc[SLICE];
          tmem_ld_32x32(acc_addr(gt, h), acc);
          if (mine) {
#pragma unroll
            for (int i = 0; i < SLICE; ++i)
              if (col0 + i < v) sts32(srow + (uint32_t)(col0 + i) * 4u, rr_order_key(__uint_as_float(acc[i])));
          }
          __syncwarp();
        }
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
        const int hg = row_list ? row_list[seg_lo + tm * BM + rr] : prob * p.n_q + tm * BM + rr;
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
  if (tid == 0) { PH_CNT(14, clock64() - cta_t0_); PH_CNT(15, 1); }
#endif
  if (warp == 1) {                                         // the warp that allocated
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
  if (tid == 0 && ctl->abort_flag) atomicOr(p.status, RR_STATUS_TIMEOUT);
  if (!row_list_arg) rr_pdl_wait();                        // complete only after the predecessor is
}

// ---- configuration -------------------------------------------------------------------------------
// 48 entries hold what passes the bound (keep 24: mean / largest of 10^5 random rows of 1024 chunks 27 / 40); a row that
// needs more takes the slow path, and the CTA that meets one runs 12 us longer.
struct Plan { int ctas, ring_bytes; size_t smem; };   // ctas: per SM
bool plan(const RRParams& p, Plan& out) {
  const int keep = p.k + (p.m > 0 ? p.m : 1);
  if (p.dtype != RR_BF16 || (p.d != 64 && p.d != 128) || p.n_k > RR_MAX_NK || keep > MAX_KEEP) return false;
  const int words = (p.n_k + 31) / 32;
  int ring = STAGES * BN * p.d * 2;
  if (ring < words * (int)WORD_PITCH) ring = words * (int)WORD_PITCH;
  out.ring_bytes = (ring + 1023) / 1024 * 1024;
  out.smem = (size_t)out.ring_bytes + CTL_BYTES + (size_t)CAP * SLOT_PITCH;
  out.ctas = 2 * (out.smem + 1024) <= 228 * 1024 ? 2 : 1;
  return out.smem <= 227 * 1024;
}

typedef void (*Kernel)(RRParams, const __nv_bfloat16*, const CUtensorMap, const int32_t*, uint32_t, int, int, int);
Kernel kernel_of(int d) { return d == 128 ? route_rows_kernel<128> : route_rows_kernel<64>; }

}  // namespace

#ifdef RR_PHASE_TIMING
extern "C" int rr_debug_rows_phase_counters(unsigned long long* out32, int reset) {
  cudaDeviceSynchronize();
  if (cudaMemcpyFromSymbol(out32, g_rows_phase, sizeof(unsigned long long) * 32) != cudaSuccess) return -1;
  if (reset) {
    unsigned long long z[32] = {};
    cudaMemcpyToSymbol(g_rows_phase, z, sizeof z);
  }
  return 0;
}
#endif

bool rr_route_rows_supported(const RRParams& p) { Plan pl; return plan(p, pl); }

cudaError_t rr_launch_route_rows(const RRParams& p, const void* qc, const void* kc, const int32_t* row_list,
                                 int layer, int hooks, cudaStream_t st) {
  Plan pl;
  if (!plan(p, pl)) return cudaErrorInvalidConfiguration;
  CUtensorMap tmap;
  cudaError_t e = rr_encode_tmap_bf16_tile(&tmap, kc, p.d, p.n_k, p.P, BN);
  if (e != cudaSuccess) return e;
  static unsigned long long attr_done = 0;      // devices on which the attributes are set
  e = rr_once_per_device(attr_done, [] {
    for (int d = 64; d <= 128; d += 64) {
      const cudaError_t a = cudaFuncSetAttribute((const void*)kernel_of(d), cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
      if (a != cudaSuccess) return a;
      cudaFuncSetAttribute((const void*)kernel_of(d), cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    }
    return cudaSuccess;
  });
  if (e != cudaSuccess) return e;
  e = rr_launch_pdl(kernel_of(p.d), p.n_tiles, NT, pl.smem, st, p, (const __nv_bfloat16*)qc, tmap, row_list,
                    (uint32_t)layer, hooks, pl.ring_bytes, pl.ctas * rr_sm_count());
  rr_count_launch();
  return e;
}
