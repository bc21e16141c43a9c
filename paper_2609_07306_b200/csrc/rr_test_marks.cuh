// The candidates of the challenge test (Section 3.2) as bitmaps in shared memory: the ledger rows of 32
// consecutive query rows are one array in memory, which a quarter's warps read in order (16 bytes per lane where
// a row splits into them); the row of what they hold is computed.  (A lane per row would touch 32 cache
// lines per load.)
#pragma once
#include "rr_common.cuh"

// Marks the valid ids of rows row0 .. row0 + n_rows - 1 (of problem prob; ids: the whole array, w per row): the bit
// of id goes to plane + row * row_pitch + (id / 32) * WORD_PITCH.  The warp is one of PARTS that share the work.
// (Ordinary loads: the routing kernel writes the same arrays later on, which rules out the read-only path.)
// Returns how many ids this lane has marked; `bad`: it has met one that its row may not select.
template <int PARTS, uint32_t WORD_PITCH>
__device__ __forceinline__ int rr_mark_rows(const RRParams& p, const int32_t* all_ids, int w, int prob, int row0,
                                            int n_rows, uint32_t plane, uint32_t row_pitch,
                                            int part, int lane, bool& bad) {
  const int32_t* const ids = all_ids + ((size_t)prob * p.n_q + row0) * w;
  int n_cand = 0;
  auto mark = [&](int id, int vr, uint32_t map) {
    bad |= id >= vr;
    // a shared-memory reduction: marks do not wait for one another
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 a, b;\n\tsetp.lt.u32 p, %1, %2;\n\t"
                 "shr.u32 a, %1, 5;\n\tmad.lo.u32 a, a, %4, %3;\n\tshf.l.wrap.b32 b, 0, 1, %1;\n\t"
                 "@p red.shared.or.b32 [a], b;\n\t@p add.s32 %0, %0, 1;\n\t}"
                 : "+r"(n_cand) : "r"(id), "r"(vr), "r"(map), "n"(WORD_PITCH) : "memory");
  };
  const bool vec = (w & 3) == 0;
  const int per = vec ? w >> 2 : w, total = n_rows * per;    // loads per row, of all the rows
  const uint32_t inv = per > 1 ? 0xFFFFFFFFu / (uint32_t)per + 1u : 0u;
  auto row_of = [&](int f) { return per > 1 ? (int)__umulhi((uint32_t)f, inv) : f; };
  auto valid_of = [&](int rr) { return rr_valid_count(row0 + rr, p.n_k, p.causal, p.causal_offset); };
  constexpr int STEP = 32 * PARTS, U = 8 / PARTS;
  if (vec) {
#pragma unroll 1
    for (int f0 = part * 32 + lane; f0 < total; f0 += U * STEP) {
      int4 q[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        q[u] = f0 + u * STEP < total ? reinterpret_cast<const int4*>(ids)[f0 + u * STEP] : make_int4(-1, -1, -1, -1);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int rr = row_of(f0 + u * STEP), vr = valid_of(rr);
        const uint32_t map = plane + (uint32_t)rr * row_pitch;
        mark(q[u].x, vr, map); mark(q[u].y, vr, map); mark(q[u].z, vr, map); mark(q[u].w, vr, map);
      }
    }
  } else {
#pragma unroll 1
    for (int f0 = part * 32 + lane; f0 < total; f0 += U * STEP) {
      int q[U];
#pragma unroll
      for (int u = 0; u < U; ++u) q[u] = f0 + u * STEP < total ? ids[f0 + u * STEP] : -1;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int rr = row_of(f0 + u * STEP);
        mark(q[u], valid_of(rr), plane + (uint32_t)rr * row_pitch);
      }
    }
  }
  return n_cand;
}
