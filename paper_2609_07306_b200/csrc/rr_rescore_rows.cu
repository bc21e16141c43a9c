// Candidate rescoring + challenge test (Section 3.2, Eq. 5) on the score strip of the tensor cores:
// the default for bf16 beyond one row tile per SM (smaller grids test inside the routing kernel, rr_route_quad.cuh).
//
// One CTA owns 128 query rows of one problem and walks the key chunks in tiles of 64: warp 0 loads Kc
// (TMA), warp 1 multiplies (tcgen05.mma, the Qc tile as the A operand in TMEM), warps 2-9 consume.
// Two threads share a row; thread j takes the tiles t with t % 2 == j.  The row's ledger entries are
// first turned into two bitmaps in shared memory, one of the route and one of the sentinels; per 32
// columns a thread reads its scores from TMEM and folds those whose bits are set into a minimum
// (route) and a maximum (sentinels).
//
// What bounds it: at 256 x 1024 x 1024, d = 128, k = 32, m + r = 32 it takes 91 us (31 us of bytes at
// the measured copy rate).  The ALU pipe is 55 % busy with bit tests and predicated min / max over
// every computed score and with the marks, the rest is the latency of a CTA's phases, which the two
// CTAs of an SM hide only in part.  The same tile loop took 111 us while every thread read its own
// ledger row and its own half of a Qc row (32 lanes on 32 rows: up to 32 cache lines per load), and the
// shared pipeline with Qc in shared memory took 105 us.  Hence, together 111 -> 91 us:
//   * the ledger rows of a quarter's 32 query rows are consecutive, so its two warps read them as one
//     array (16 bytes per lane where a row splits into them) and compute the row of what they hold;
//   * the Qc tile comes by TMA into the Kc ring, whose first tiles are not needed before the bitmaps
//     are built, and goes on to TMEM from there: it needs no shared memory of its own, so two CTAs
//     fit an SM up to n_k = 2048 (at 64 x 2048 x 2048, k = 64: 133 -> 79 us).
// Two tiles to a turn beat a split of every tile's columns between a row's threads (91 : 94 us: half
// the waits).  A third CTA per SM (tiles of 32, 64 registers: 94 us), a third ring stage (89 us, but
// one CTA per SM at n_k = 2048) and min / max of three operands with the selection on the FMA pipe
// (99 us: more instructions) were no better.
#include "rr_common.cuh"
#include "rr_sm100.cuh"
#include "rr_test_marks.cuh"

using namespace sm100;

namespace {

constexpr int BM = 128, BN = 64, STAGES = 2, ACC = 2;
constexpr int TPR = 2, COLS = 32;                    // threads per row, columns per step
constexpr int CONS_WARPS = TPR * (BM / 32), NT = (2 + CONS_WARPS) * 32;
constexpr int TMEM_COLS = 256, A_COL = ACC * BN;     // accumulators, then the Qc tile
constexpr unsigned FULL = 0xFFFFFFFFu;

struct Ctl {
  uint64_t full[STAGES], q_full;                    // Kc tiles, the Qc tile
  uint64_t acc_full[ACC], acc_empty[ACC];
  uint64_t drain;
  uint32_t tmem_base, abort_flag, flagged, cand;
  unsigned long long full_pairs;
};
constexpr int CTL_BYTES = 256;
static_assert(sizeof(Ctl) <= CTL_BYTES, "control block too large");

__device__ __forceinline__ void consumers_sync() {   // the consumer warps only
  asm volatile("bar.sync 1, %0;" ::"n"(CONS_WARPS * 32) : "memory");
}
template <int D>
__global__ void __launch_bounds__(NT, 2)
rescore_rows_kernel(RRParams p, const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                    int words, int force_timeout) {
  constexpr int KH = D / 64, TILE = BN * D * 2;
  rr_pdl_wait();
  if (p.force_threshold > 0 && p.force_in[0] > 0) return;   // forced anchor: nothing is tested
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  Ctl* ctl = (Ctl*)(smem + STAGES * TILE);
  const uint32_t pitch = 2u * words + 1u;                   // bitmap words per row (odd: no bank conflicts)
  const uint32_t ring = smem_u32(smem), parts = smem_u32(ctl) + CTL_BYTES, maps = parts + 2u * BM * 4u;

  const int tid = threadIdx.x, warp = __shfl_sync(FULL, tid >> 5, 0), lane = tid & 31;
  const int tiles_m = p.tiles_per_problem;
  const int prob = blockIdx.x % p.P, tm = tiles_m - 1 - blockIdx.x / p.P;   // heaviest first
  const int row_end = min(p.n_q, (tm + 1) * BM);
  const int n_tiles = (rr_valid_count(row_end - 1, p.n_k, p.causal, p.causal_offset) + BN - 1) / BN;
  const bool is_cons = warp >= 2;
  const int quarter = warp & 3, j = (warp - 2) >> 2;
  const int r = quarter * 32 + lane, row = tm * BM + r;
  const bool has = is_cons && row < p.n_q;
  const size_t g = (size_t)prob * p.n_q + row;

  constexpr int QT = D == 128 ? 2 : 1, QW = 32;             // threads per row, words per thread
  static_assert(STAGES * TILE >= BM * D * 2, "the Qc tile passes through the Kc ring");
  const bool q_loader = is_cons && j < QT;
  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) mbar_init(&ctl->full[s], 1);
    for (int s = 0; s < ACC; ++s) { mbar_init(&ctl->acc_full[s], 1); mbar_init(&ctl->acc_empty[s], CONS_WARPS / TPR); }
    mbar_init(&ctl->q_full, 1);
    mbar_init(&ctl->drain, 1);
    ctl->abort_flag = 0; ctl->flagged = 0; ctl->cand = 0; ctl->full_pairs = 0ull;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc(&ctl->tmem_base, TMEM_COLS);
    rr_pdl_trigger();                                       // (not before: the successor takes TMEM, too)
  }
  if (warp == 0) {
    __syncwarp();
    tma_load_tile_warp(ring, &tmap_q, tm * BM, prob, &ctl->q_full, BM * D * 2);
  }
  // The two warps of a quarter clear the bitmaps of its rows together.
  const uint32_t maps_q = maps + (uint32_t)(quarter * 32) * pitch * 4u;
  if (is_cons) {
#pragma unroll 4
    for (uint32_t o = (uint32_t)(j * 32 + lane) * 16u; o < 32u * pitch * 4u; o += TPR * 32 * 16)
      asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(maps_q + o), "r"(0u) : "memory");
  }
  const uint32_t mapA = maps + (uint32_t)r * pitch * 4u, mapB = mapA + (uint32_t)words * 4u;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  volatile uint32_t* abort_flag = &ctl->abort_flag;
  if (q_loader) {
    // (a wait that gives up raises the abort flag: no role enters its loop)
    __all_sync(FULL, mbar_wait(&ctl->q_full, 0, abort_flag));
    uint32_t qv[QW];
    const uint32_t src = ring + (uint32_t)(j * BM * 128 + r * 128);
#pragma unroll
    for (int i = 0; i < QW / 4; ++i)
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(qv[4 * i]), "=r"(qv[4 * i + 1]), "=r"(qv[4 * i + 2]),
                   "=r"(qv[4 * i + 3]) : "r"(src + (uint32_t)((i ^ (r & 7)) << 4)) : "memory");
    tmem_st_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + A_COL + j * QW, qv);
    tmem_st_wait();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) {
    // ===== TMA producer: a stage is free again when its tile's MMAs are done (acc_full) =====
    int t = 0;
#pragma unroll 1
    for (; t < n_tiles; ++t) {
      const int done = t - STAGES;
      if (done >= 0 && !__all_sync(FULL, mbar_wait_spin(&ctl->acc_full[done % ACC], (done / ACC) & 1, abort_flag))) break;
      tma_load_tile_warp(ring + (t % STAGES) * TILE, &tmap_k, t * BN, prob, &ctl->full[t % STAGES], TILE);
    }
    // no copies in flight beyond this point
#pragma unroll 1
    for (uint32_t it = 0; it < kSpinLimit && !mbar_try_wait(&ctl->q_full, 0); ++it) __nanosleep(64);
#pragma unroll 1
    for (int u = max(0, t - STAGES); u < t; ++u)
#pragma unroll 1
      for (uint32_t it = 0; it < kSpinLimit && !mbar_try_wait(&ctl->full[u % STAGES], (u / STAGES) & 1); ++it) __nanosleep(64);
    __syncwarp();
  } else if (warp == 1) {
    // ===== MMA issuer =====
    constexpr uint32_t idesc = umma_idesc_bf16(BM, BN);
    const uint32_t tmem_u = __shfl_sync(FULL, tmem_base, 0);
    const uint64_t desc0 = umma_desc_k_sw128(ring);
#pragma unroll 1
    for (int t = 0; t < n_tiles; ++t) {
      const int s = t % STAGES, as = t % ACC;
      if (!__all_sync(FULL, mbar_wait_spin(&ctl->acc_empty[as], ((t / ACC) & 1) ^ 1, abort_flag))) break;
      if (!__all_sync(FULL, mbar_wait_spin(&ctl->full[s], (t / STAGES) & 1, abort_flag))) break;
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < KH * 4; ++k)
        umma_bf16_ts_warp(tmem_u + as * BN, tmem_u + A_COL + k * 8,
                          desc0 + (uint64_t)(s * (TILE >> 4) + (k >> 2) * (BN * 128 >> 4) + (k & 3) * 2), idesc,
                          k > 0 ? 1u : 0u);
      umma_commit_warp(&ctl->acc_full[as]);
    }
    umma_commit_warp(&ctl->drain);                           // TMEM is not freed while an MMA may write to it
#pragma unroll 1
    for (uint32_t it = 0; it < kSpinLimit && !mbar_try_wait(&ctl->drain, 0); ++it) __nanosleep(64);
    __syncwarp();
  } else {
    // ===== consumers =====
    const float pinf = __int_as_float(0x7f800000);
    const int v = has ? rr_valid_count(row, p.n_k, p.causal, p.causal_offset) : 0;
    // ---- the quarter's ledger rows -> this warp's bitmap (j = 0: routes, 1: sentinels) ---------------
    const int row0 = tm * BM + quarter * 32, n_rows = max(0, min(32, p.n_q - row0));
    bool bad = false;
    int n_cand = rr_mark_rows<1, 4>(p, j == 0 ? p.routes : p.sentinels, j == 0 ? p.k : p.sw, prob, row0, n_rows,
                                    maps_q + (j == 0 ? 0u : (uint32_t)words * 4u), pitch * 4u, 0, lane, bad);
    if (p.debug && has && j == 0)
      for (int s = 0; s < p.c; ++s) p.cand_scores[g * p.c + s] = __int_as_float(0x7fc00000);
    consumers_sync();                                        // either thread reads both bitmaps

    float amin = pinf, bmax = -pinf;
    const uint32_t acc_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
    bool alive = true;
#pragma unroll 1
    for (int t = j; t < n_tiles; t += TPR) {
      // test hook: the first wait of CTA 0 counts as expired
      if (force_timeout && blockIdx.x == 0) { *abort_flag = 1u; alive = false; }
      if (alive) alive = __all_sync(FULL, mbar_wait(&ctl->acc_full[t % ACC], (t / ACC) & 1, abort_flag));
      if (!alive) break;
      tc_fence_after();
      constexpr int NC = BN / COLS;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int wi = t * NC + c;
        const bool in = wi < words;
        const uint32_t wa = in ? lds32(mapA + wi * 4u) : 0u, wb = in ? lds32(mapB + wi * 4u) : 0u;
        const bool work = __any_sync(FULL, (wa | wb) != 0u);
        uint32_t s[COLS];
        if (work) tmem_ld_32x32(acc_lane + (uint32_t)((t % ACC) * BN + c * COLS), s);
        if (c == NC - 1) {                                   // the accumulator goes back
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&ctl->acc_empty[t % ACC]);
        }
        if (!work) continue;
#pragma unroll
        for (int i = 0; i < COLS; ++i) {
          min_if(amin, __uint_as_float(s[i]), wa, 1u << i);
          max_if(bmax, __uint_as_float(s[i]), wb, 1u << i);
        }
        if (p.debug && has) {                                // tests: every candidate's score
          for (int q = 0; q < p.c; ++q) {
            const int id = q < p.k ? p.routes[g * p.k + q] : p.sentinels[g * p.sw + q - p.k];
            if (id < 0 || id >= v || (id >> 5) != wi) continue;
#pragma unroll
            for (int i = 0; i < COLS; ++i)
              if ((id & 31) == i) p.cand_scores[g * p.c + q] = __uint_as_float(s[i]);
          }
        }
      }
    }
    // ---- the second thread of each row hands its part to the first, which tests the row --------------
    const uint32_t part = parts + (uint32_t)r * 4u;
    if (j == 1) { sts32(part, __float_as_uint(amin)); sts32(part + BM * 4u, __float_as_uint(bmax)); }
    consumers_sync();
    if (j == 0) {
      amin = fminf(amin, __uint_as_float(lds32(part)));
      bmax = fmaxf(bmax, __uint_as_float(lds32(part + BM * 4u)));
      bool flag = false;
      if (has && *abort_flag == 0u) {                        // (a wait that gave up: the CTA's rows stay)
        flag = rr_challenge(p, (int)g, amin, bmax);
        p.flags[g] = flag ? 1 : 0;
        p.alpha[g] = amin;
        p.beta[g] = bmax;
      }
      const int n_flag = __popc(__ballot_sync(FULL, flag));
      const int v_sum = __reduce_add_sync(FULL, flag ? v : 0);
      if (lane == 0) {
        atomicAdd(&ctl->flagged, (uint32_t)n_flag);
        atomicAdd(&ctl->full_pairs, (unsigned long long)v_sum);
      }
    }
    n_cand = __reduce_add_sync(FULL, n_cand);
    if (lane == 0) atomicAdd(&ctl->cand, (uint32_t)n_cand);
    if (__any_sync(FULL, bad) && lane == 0) atomicOr(p.status, RR_STATUS_BAD_INDEX);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {                                           // the warp that allocated
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
  if (tid == 0) {
    if (ctl->abort_flag) atomicOr(p.status, RR_STATUS_TIMEOUT);
    p.tile_counts[prob * tiles_m + tm] = (uint32_t)ctl->flagged;
    atomicAdd(&p.counters[RR_CNT_FLAGGED_ROWS], (unsigned long long)ctl->flagged);
    atomicAdd(&p.counters[RR_CNT_CAND_PAIRS], (unsigned long long)ctl->cand);
    atomicAdd(&p.counters[RR_CNT_FULL_PAIRS], ctl->full_pairs);
  }
}

size_t smem_bytes(int d, int n_k) {
  const int words = (n_k + 31) / 32;
  return 1024 + (size_t)STAGES * BN * d * 2 + CTL_BYTES + (size_t)2 * BM * 4 + (size_t)BM * (2 * words + 1) * 4;
}

}  // namespace

bool rr_rescore_rows_supported(const RRParams& p) {
  return p.dtype == RR_BF16 && (p.d == 64 || p.d == 128) && smem_bytes(p.d, p.n_k) <= 227 * 1024;
}

cudaError_t rr_launch_rescore_rows(const RRParams& p, const void* qc, const void* kc, int force_timeout,
                                   cudaStream_t st) {
  if (!rr_rescore_rows_supported(p)) return cudaErrorInvalidConfiguration;
  CUtensorMap tmap, tmap_q;
  cudaError_t e = rr_encode_tmap_bf16_tile(&tmap, kc, p.d, p.n_k, p.P, BN);
  if (e != cudaSuccess) return e;
  e = rr_encode_tmap_bf16_tile(&tmap_q, qc, p.d, p.n_q, p.P, BM);
  if (e != cudaSuccess) return e;
  static unsigned long long attr_done = 0;      // devices on which the attributes are set
  e = rr_once_per_device(attr_done, [] {
    for (const void* fn : {(const void*)rescore_rows_kernel<64>, (const void*)rescore_rows_kernel<128>}) {
      const cudaError_t a = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
      if (a != cudaSuccess) return a;
      cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    }
    return cudaSuccess;
  });
  if (e != cudaSuccess) return e;
  const int words = (p.n_k + 31) / 32;
  e = rr_launch_pdl(p.d == 128 ? rescore_rows_kernel<128> : rescore_rows_kernel<64>, p.n_tiles, NT, smem_bytes(p.d, p.n_k),
                    st, p, tmap_q, tmap, words, force_timeout);
  rr_count_launch();
  return e;
}
