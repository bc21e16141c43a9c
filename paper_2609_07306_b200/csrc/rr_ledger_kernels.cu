// Row compaction (Section 4.2: "A prefix sum compacts unstable row IDs") together with the
// ledger's book-keeping (Section 4.1: stable rows keep their routes and their ages advance;
// refreshed rows restart at age 0; cumulative work counters), the anchor's fill of the same
// state, token-range expansion, and ledger reset.
#include "rr_common.cuh"

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

// ---- compaction -----------------------------------------------------------------------
// One CTA per row tile (RR_ROW_TILE rows of one problem).  The tile's base offset is the sum
// of the flagged counts of all earlier tiles (written by the kernel that tested the rows); inside the
// tile a ballot/popcount scan gives each flagged row its slot.  The list is therefore in
// ascending global row id -- exactly numpy.nonzero(flags) -- with no atomics and no waits
// (the price: n_tiles^2 / 2 count reads in total, nothing at the few thousand tiles of a layer).
// The same pass advances the ages (flagged -> 0, stable -> +1) and, once per launch, the
// per-layer counters: nothing later in the layer reads either.
template <int WORDS>                                         // p.count_words
__global__ void __launch_bounds__(RR_ROW_TILE)
compact_kernel(RRParams p, unsigned long long dense_pairs) {
  __shared__ int s_part[RR_ROW_TILE / 32], s_cnt[RR_ROW_TILE / 32];   // earlier tiles' counts, by warp; this tile's
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tile_id = blockIdx.x;
  const int prob = tile_id / p.tiles_per_problem, tile = tile_id % p.tiles_per_problem;
  rr_pdl_wait();
  rr_pdl_trigger();

  // Forced anchor (Section 3.2, policy of rr_config.force_permille): the previous tested relay
  // flagged so many rows that this call routes every row.  The tile does what the anchor's fill
  // does for its rows; the rescoring kernel has exited without writing anything.
  if (p.force_threshold > 0 && p.force_in[0] > 0) {
    const int i = tile * RR_ROW_TILE + tid;
    const int g = prob * p.n_q + i;
    if (i < p.n_q) {
      const float qnan = __int_as_float(0x7fc00000);
      p.flags[g] = 1; p.refresh_rows[g] = g; p.ages[g] = 0;
      p.alpha[g] = qnan; p.beta[g] = qnan; p.tau[g] = __int_as_float(0xff800000);
    }
    if (tid == 0) {
      if (tile == 0) p.problem_offsets[prob] = prob * p.n_q;
      if (tile_id == 0) {
        p.counters[RR_CNT_LAYER_CALLS] += 1;
        p.counters[RR_CNT_DENSE_PAIRS] += dense_pairs;
        p.counters[RR_CNT_ANCHOR_ROWS] += (unsigned long long)p.rows;
        p.counters[RR_CNT_FULL_PAIRS] += dense_pairs;
      }
      if (tile_id == p.n_tiles - 1) {
        p.problem_offsets[p.P] = p.rows;
        *p.refresh_count = p.rows;
        p.force_out[0] = p.force_in[0] - 1; p.force_out[1] = p.force_in[1];
        p.force_stats[4] += 1; p.force_stats[5] = 1;
      }
    }
    return;
  }

  // The row's flag and age are asked for together with the counts (one round trip to L2), and one barrier
  // serves the base and the places inside the tile: 256 x 256 rows, 24 layers 938 -> 925 us.
  const int i = tile * RR_ROW_TILE + tid;
  const int g = prob * p.n_q + i;
  const bool in = i < p.n_q;
  const int flag = in ? p.flags[g] : 0;
  const int age = in ? p.ages[g] : 0;
  unsigned part = 0;                                         // (bytes: see RRParams)
  if constexpr (WORDS == 1) {
    for (int t = tid; t < tile_id; t += RR_ROW_TILE) part = __dp4a(p.tile_counts[t], 0x01010101u, part);
  } else {
    for (int t = tid; t < tile_id; t += RR_ROW_TILE) {
      const uint4 c = reinterpret_cast<const uint4*>(p.tile_counts)[t];
      part = __dp4a(c.x, 0x01010101u, __dp4a(c.y, 0x01010101u, __dp4a(c.z, 0x01010101u, __dp4a(c.w, 0x01010101u, part))));
    }
  }
  part = __reduce_add_sync(FULL, part);
  const bool f = flag != 0;
  const unsigned bal = __ballot_sync(FULL, f);
  if (lane == 0) { s_part[warp] = (int)part; s_cnt[warp] = __popc(bal); }
  __syncthreads();
  int base = 0, before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < RR_ROW_TILE / 32; ++w) {
    base += s_part[w];
    if (w < warp) before += s_cnt[w];
    total += s_cnt[w];
  }
  if (f) p.refresh_rows[base + before + __popc(bal & ((1u << lane) - 1u))] = g;
  if (in) p.ages[g] = f ? 0 : age + 1;
  if (tid == 0) {
    if (tile_id == 0) {
      p.counters[RR_CNT_LAYER_CALLS] += 1;
      p.counters[RR_CNT_DENSE_PAIRS] += dense_pairs;
      p.counters[RR_CNT_RELAY_ROWS] += (unsigned long long)p.rows;
    }
    if (tile == 0) p.problem_offsets[prob] = base;
    if (tile_id == p.n_tiles - 1) {
      total += base;
      p.problem_offsets[p.P] = total;
      *p.refresh_count = total;
      if (p.force_threshold > 0) {    // this call was tested: decide about the next ones
        const int run = total >= p.force_threshold ? min(max(1, 2 * p.force_in[1]), p.force_max_run) : 0;
        p.force_out[0] = run; p.force_out[1] = run; p.force_stats[5] = 0;
      }
    }
  }
}

// ---- anchor: every row is (re)routed ----------------------------------------------------
// Flags, identity refresh list, offsets, ages and the anchor's counters.
__global__ void anchor_fill_kernel(RRParams p, unsigned long long dense_pairs) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  const float qnan = __int_as_float(0x7fc00000);
  rr_pdl_wait();
  rr_pdl_trigger();
  if (g < p.rows) {
    p.flags[g] = 1;
    p.refresh_rows[g] = g;
    p.alpha[g] = qnan;
    p.beta[g] = qnan;
    p.ages[g] = 0;
  }
  if (g <= p.P) p.problem_offsets[g] = g * p.n_q;
  if (g == 0) {
    *p.refresh_count = p.rows;
    p.counters[RR_CNT_LAYER_CALLS] += 1;
    p.counters[RR_CNT_DENSE_PAIRS] += dense_pairs;
    p.counters[RR_CNT_ANCHOR_ROWS] += (unsigned long long)p.rows;
    p.counters[RR_CNT_FULL_PAIRS] += dense_pairs;
    if (p.force_threshold > 0) {      // a scheduled anchor clears a pending forced run
      p.force_out[0] = 0; p.force_out[1] = p.force_in[1]; p.force_stats[5] = 0;
    }
  }
}

// ---- token ranges of the rows that were re-routed -------------------------------------------
// Chunk j -> [j*T, (j+1)*T), ascending chunk id, (-1,-1) for empty slots.  General form, one warp per
// row: ids that are out of order are ranked by counting (they are distinct).
__device__ void expand_row(const RRParams& p, int g, int lane, int32_t* srt) {
  const int32_t* route = p.routes + (size_t)g * p.k;
  int32_t* out = p.token_ranges + (size_t)g * p.k * 2;
  // rows written by the routing kernels are already in ascending chunk id with the empty
  // slots last: their ranges are a plain map of the row (8-byte stores)
  bool ordered = true;
  for (int s = lane; s < p.k; s += 32) {
    const int id = route[s];
    if (s > 0 && id >= 0) { const int prev = route[s - 1]; ordered &= prev >= 0 && prev < id; }
  }
  const bool all_ordered = __all_sync(FULL, ordered);
  if (p.coalesce) {
    // the row's ids in ascending order (empty slots last) into shared memory, then one range
    // per run of consecutive ids: a run's first id writes its start, its last id its end
    for (int s = lane; s < p.k; s += 32) srt[s] = all_ordered ? route[s] : -1;
    __syncwarp();
    if (!all_ordered) {
      for (int s = lane; s < p.k; s += 32) {
        const int id = route[s];
        if (id >= 0) {
          int rank = 0;
          for (int t = 0; t < p.k; ++t) { const int o = route[t]; rank += (o >= 0 && o < id); }
          srt[rank] = id;
        }
      }
      __syncwarp();
    }
    int base = 0;
    for (int s0 = 0; s0 < p.k; s0 += 32) {
      const int s = s0 + lane;
      const int id = s < p.k ? srt[s] : -1;
      const bool valid = id >= 0;
      const bool joins_prev = valid && s > 0 && srt[s - 1] == id - 1 && srt[s - 1] >= 0;
      const bool joins_next = valid && s + 1 < p.k && srt[s + 1] == id + 1;
      const unsigned starts = __ballot_sync(FULL, valid && !joins_prev);
      const int ri = base + __popc(starts & (0xFFFFFFFFu >> (31 - lane))) - 1;
      if (valid && !joins_prev) out[2 * ri] = id * p.chunk_tokens;
      if (valid && !joins_next) out[2 * ri + 1] = (id + 1) * p.chunk_tokens;
      base += __popc(starts);
    }
    for (int s = base + lane; s < p.k; s += 32) { out[2 * s] = -1; out[2 * s + 1] = -1; }
    __syncwarp();
    return;
  }
  if (all_ordered) {
    for (int s = lane; s < p.k; s += 32) {
      const int id = route[s];
      reinterpret_cast<int2*>(out)[s] =
          id >= 0 ? make_int2(id * p.chunk_tokens, (id + 1) * p.chunk_tokens) : make_int2(-1, -1);
    }
    return;
  }
  int n_valid = 0;
  for (int s = lane; s < p.k; s += 32) n_valid += route[s] >= 0;
#pragma unroll
  for (int off = 16; off; off >>= 1) n_valid += __shfl_xor_sync(FULL, n_valid, off);
  for (int s = lane; s < p.k; s += 32) {
    const int id = route[s];
    if (id >= 0) {
      int rank = 0;
      for (int t = 0; t < p.k; ++t) { const int o = route[t]; rank += (o >= 0 && o < id); }
      out[2 * rank] = id * p.chunk_tokens;
      out[2 * rank + 1] = (id + 1) * p.chunk_tokens;
    }
  }
  for (int s = n_valid + lane; s < p.k; s += 32) { out[2 * s] = -1; out[2 * s + 1] = -1; }
}

// A warp takes EXPAND_ROWS rows, so that several loads are in flight before the first store: a row of
// up to 64 ids is one 8-byte load per lane, checked for order with one shuffle, and one 16-byte store
// per lane (the plain map).  Bound by DRAM: 100 MB per layer of 131072 rows at k = 64.
constexpr int EXPAND_ROWS = 4, EXPAND_WARPS = 8;
__host__ __device__ __forceinline__ bool expand_by_row(const RRParams& p) { return p.coalesce || p.k > 64 || (p.k & 1); }
__global__ void __launch_bounds__(EXPAND_WARPS * 32)
expand_kernel(RRParams p, int is_anchor) {
  extern __shared__ int32_t s_sorted[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  rr_pdl_wait();
  rr_pdl_trigger();
  int32_t* const srt = s_sorted + warp * p.k;
  if (expand_by_row(p)) {
    const int g = blockIdx.x * EXPAND_WARPS + warp;
    if (g < p.rows && (is_anchor || p.flags[g] != 0)) expand_row(p, g, lane, srt);   // (stable row: ranges unchanged)
    return;
  }
  const int g0 = (blockIdx.x * EXPAND_WARPS + warp) * EXPAND_ROWS;
  const int s = 2 * lane, T = p.chunk_tokens;
  int2 id[EXPAND_ROWS];
  bool on[EXPAND_ROWS];
#pragma unroll
  for (int u = 0; u < EXPAND_ROWS; ++u) {
    on[u] = g0 + u < p.rows && (is_anchor || p.flags[g0 + u] != 0);
    id[u] = make_int2(-1, -1);
    if (on[u] && s < p.k) id[u] = *reinterpret_cast<const int2*>(p.routes + (size_t)(g0 + u) * p.k + s);
  }
#pragma unroll
  for (int u = 0; u < EXPAND_ROWS; ++u) {
    if (!on[u]) continue;                              // (uniform)
    const int prev = __shfl_up_sync(FULL, id[u].y, 1);
    const bool ok = (lane == 0 || id[u].x < 0 || (prev >= 0 && prev < id[u].x)) &&
                    (id[u].y < 0 || (id[u].x >= 0 && id[u].x < id[u].y));
    if (!__all_sync(FULL, ok)) { expand_row(p, g0 + u, lane, srt); continue; }
    if (s < p.k) {
      int4 o = make_int4(-1, -1, -1, -1);
      if (id[u].x >= 0) { o.x = id[u].x * T; o.y = o.x + T; }
      if (id[u].y >= 0) { o.z = id[u].y * T; o.w = o.z + T; }
      *reinterpret_cast<int4*>(p.token_ranges + ((size_t)(g0 + u) * p.k + s) * 2) = o;
    }
  }
}

__global__ void reset_kernel(RRParams p) {
  const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t e = tid; e < (size_t)p.rows * p.k; e += stride) p.routes[e] = -1;
  for (size_t e = tid; e < (size_t)p.rows * p.sw; e += stride) p.sentinels[e] = -1;
  for (size_t e = tid; e < (size_t)p.rows; e += stride) {
    p.ages[e] = -1; p.kth[e] = 0.f; p.margin[e] = 0.f;
    p.flags[e] = 0; p.alpha[e] = 0.f; p.beta[e] = 0.f; p.refresh_rows[e] = -1;
  }
  for (size_t e = tid; e <= (size_t)p.P; e += stride) p.problem_offsets[e] = 0;
  for (size_t e = tid; e < (size_t)p.n_tiles * p.count_words; e += stride) p.tile_counts[e] = 0;
  if (p.token_ranges)
    for (size_t e = tid; e < (size_t)p.rows * p.k * 2; e += stride) p.token_ranges[e] = -1;
  if (tid < RR_NUM_COUNTERS) p.counters[tid] = 0;
  if (tid < 8) p.force_stats[tid] = 0;
  if (tid == 0) { *p.status = 0; *p.refresh_count = 0; }
}

}  // namespace

cudaError_t rr_launch_compact(const RRParams& p, unsigned long long dense_pairs, cudaStream_t st) {
  const cudaError_t e = rr_launch_pdl(p.count_words == 1 ? compact_kernel<1> : compact_kernel<RR_COUNT_WORDS_F32>, p.n_tiles, RR_ROW_TILE, 0, st, p, dense_pairs);
  rr_count_launch();
  return e;
}

cudaError_t rr_launch_anchor_fill(const RRParams& p, unsigned long long dense_pairs,
                                  cudaStream_t st) {
  const int n = p.rows > p.P + 1 ? p.rows : p.P + 1;
  const cudaError_t e = rr_launch_pdl(anchor_fill_kernel, (n + 255) / 256, 256, 0, st, p, dense_pairs);
  rr_count_launch();
  return e;
}

cudaError_t rr_launch_expand(const RRParams& p, int is_anchor, cudaStream_t st) {
  const int rows_per_block = EXPAND_WARPS * (expand_by_row(p) ? 1 : EXPAND_ROWS);
  const size_t smem = p.coalesce ? (size_t)EXPAND_WARPS * p.k * sizeof(int32_t) : 0;
  const cudaError_t e = rr_launch_pdl(expand_kernel, (p.rows + rows_per_block - 1) / rows_per_block, EXPAND_WARPS * 32,
                                      smem, st, p, is_anchor);
  rr_count_launch();
  return e;
}

cudaError_t rr_launch_reset(const RRParams& p, cudaStream_t st) {
  reset_kernel<<<148 * 4, 256, 0, st>>>(p);
  rr_count_launch();
  return cudaPeekAtLastError();
}
