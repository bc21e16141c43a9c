// Pieces that the routing kernels with several threads per row share: packed compare-exchanges, the rank search,
// the fixed-point sort keys, the threshold filter and the sentinel draws.
#pragma once
#include "rr_common.cuh"
#include "rr_sm100.cuh"

namespace rr_select {

using namespace sm100;
constexpr unsigned FULL = 0xFFFFFFFFu;

// ---- packed compare-exchanges -----------------------------------------------------------------
struct DescBF2 {                     // two bf16 lists at a time
  static __device__ __forceinline__ void ce(uint32_t& a, uint32_t& b) {
    uint32_t hi, lo;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(hi) : "r"(a), "r"(b));
    asm("min.bf16x2 %0, %1, %2;" : "=r"(lo) : "r"(a), "r"(b));
    a = hi; b = lo;
  }
};
// Non-negative integers below the pattern of +inf, compared as floats: an FMNMX pair per
// compare-exchange, where unsigned min / max become a compare and two selects.
struct DescPos {
  static __device__ __forceinline__ void ce(uint32_t& a, uint32_t& b) {
    const float hi = fmaxf(__uint_as_float(a), __uint_as_float(b)), lo = fminf(__uint_as_float(a), __uint_as_float(b));
    a = __float_as_uint(hi); b = __float_as_uint(lo);
  }
};
struct AscPos {
  static __device__ __forceinline__ void ce(uint32_t& a, uint32_t& b) { DescPos::ce(b, a); }
};
struct AscU2 {                       // two lists of 16-bit values at a time
  static __device__ __forceinline__ void ce(uint32_t& a, uint32_t& b) {
    const uint32_t hi = __vmaxu2(a, b), lo = __vminu2(a, b);
    a = lo; b = hi;
  }
};
__host__ __device__ constexpr int pow2_at_least(int n) { int p = 1; while (p < n) p *= 2; return p; }

// ---- rank search over two descending lists ----------------------------------------------------
// How many entries of the first list belong to the T largest of both (0 <= T <= 2 M): A(i) / B(i)
// are the lists' values, M entries each.
template <int M, class FA, class FB>
__device__ __forceinline__ int rank_split(int T, FA&& A, FB&& B) {
  int lo = max(0, T - M), hi = min(T, M);
#pragma unroll 1
  for (int s = 1; s <= M; s *= 2) {
    const int mid = (lo + hi) >> 1;
    const bool more = A(min(mid, M - 1)) > B(min(max(T - mid - 1, 0), M - 1));
    const bool go = lo < hi;
    lo = go && more ? mid + 1 : lo;
    hi = go && !more ? mid : hi;
  }
  return lo;
}

// ---- fixed-point image of a survivor ------------------------------------------------------------
// Bits of 2^23 + q, q = round(8355000 * sat((s - tau) * scale + 2^-22)): monotone in s, q >= 1 for
// s >= tau, 0 for an empty slot (-inf); 256 q + slot stays below the pattern of +inf.
__device__ __forceinline__ uint32_t fixed_bits(float s, float tau, float scale) {
  float t;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(t) : "f"(s - tau), "f"(scale), "f"(1.0f / 4194304.0f));
  return __float_as_uint(fmaf(t, 8355000.0f, 8388608.0f));
}

// ---- threshold filter of sweep 2 ------------------------------------------------------------
// One score: if it passes, {score, chunk id} goes to [w] and w moves on by one entry (a compare,
// an id add and three predicated instructions; EDGE: ids >= v never pass, one compare more).  Two
// 4-byte stores: an 8-byte store wants its operands in a register pair, which the scores of a TMEM
// load are not, and the moves cost more than the second store.
template <int I, bool EDGE>
__device__ __forceinline__ void filter_one(uint32_t& w, uint32_t sbits, float tau, uint32_t col0, uint32_t step, int v) {
  if constexpr (!EDGE) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 c;\n\t"
                 "setp.ge.f32 p, %1, %2;\n\t"
                 "add.u32 c, %3, %4;\n\t"
                 "@p st.shared.b32 [%0], %1;\n\t"
                 "@p st.shared.b32 [%0+4], c;\n\t"
                 "@p add.u32 %0, %0, %5;\n\t}"
                 : "+r"(w) : "f"(__uint_as_float(sbits)), "f"(tau), "r"(col0), "n"(I), "r"(step) : "memory");
  } else {
    asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b32 c;\n\t"
                 "add.u32 c, %3, %4;\n\t"
                 "setp.lt.s32 q, c, %6;\n\t"
                 "setp.ge.and.f32 p, %1, %2, q;\n\t"
                 "@p st.shared.b32 [%0], %1;\n\t"
                 "@p st.shared.b32 [%0+4], c;\n\t"
                 "@p add.u32 %0, %0, %5;\n\t}"
                 : "+r"(w) : "f"(__uint_as_float(sbits)), "f"(tau), "r"(col0), "n"(I), "r"(step), "r"(v) : "memory");
  }
}
// ---- sentinels (Section 3.1 items 2, 3) -------------------------------------------------------
// Mandatory global and random sentinels of a warp's 32 rows, a row per lane (lanes without `go` only help).
// bits: the row's bitmap of excluded chunks (word w at bits + w * WORD_PITCH), updated here; col: the row's column of
// CAP places (place e at col + e * SLOT_PITCH), where the ids are collected before they go out with 16-byte
// stores; v: valid chunks, n_excl: excluded ones.
// Sequential definition: pool <= r -> the whole pool in ascending order; else for t = 0, 1, ...:
// j = floor(u_t v / 2^32), accepted iff j is not excluded and not drawn yet; after 64 r draws the smallest free chunks.
// Bound by the latency of hash, look and acceptance, and by rows with few free chunks, which need many draws: they made
// the first row tiles of a causal problem the last to end.  32 x 1024 x 1024, 16 layers: every lane draws to the end
// 1117 us; hands over to the warp after 2, 3, 4, 8 r draws 1112, 1045, 999, 1000; with nothing but the last comparison
// left on the chain between the four draws of a step 983.
template <uint32_t WORD_PITCH, uint32_t SLOT_PITCH, int CAP>
__device__ __forceinline__ void draw_sentinels(const RRParams& p, uint32_t bits, uint32_t col, int g, int v, int n_excl,
                                               uint32_t layer, int lane, bool go) {
  int pool = v - n_excl;
  int32_t* const rnd = p.sentinels + (size_t)g * p.sw + p.m;
  auto word = [&](int id) -> uint32_t { return bits + (uint32_t)(id >> 5) * WORD_PITCH; };
  if (go && p.n_global) {     // mandatory global sentinels: a slot each after the random ones
    int32_t* glob = rnd + p.r;
    int gi = 0;
    for (int b = 0; b < 2; ++b) {
      if (!((p.global_mask >> b) & 1)) continue;
      const int id = b == 0 ? 0 : v - 1;
      const uint32_t w = lds32(word(id)), bit = 1u << (id & 31);
      const bool free_ = !(w & bit);
      if (free_) { sts32(word(id), w | bit); --pool; }
      glob[gi++] = free_ ? id : -1;
    }
  }
  const uint32_t end = col + (uint32_t)min(p.r, CAP) * SLOT_PITCH;
  uint32_t dst = col;                                      // the next id's place, `end` = complete
  if (p.r <= CAP) {
    const bool drawing = go && pool > p.r;
    const unsigned long long rk = rr_row_key(p.seed, (uint32_t)g);
    const int limit = 64 * p.r, alone = 4 * p.r;
    int t0 = 0;
    if (!drawing) dst = end;
    // Four draws at a time, so that their looks into the bitmap overlap; they are accepted in draw order,
    // one that repeats an earlier draw of the four is as good as excluded.
    auto accept = [&](const uint32_t (&id)[4]) {
      uint32_t a[4], hit[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = bits + (id[i] >> 5) * WORD_PITCH;
#pragma unroll
      for (int i = 0; i < 4; ++i) hit[i] = lds32(a[i]) & (1u << (id[i] & 31));
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        bool fresh = hit[i] == 0u;
#pragma unroll
        for (int q = 0; q < i; ++q) fresh = fresh && id[q] != id[i];
        // (what hangs on the draw before comes last)
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "setp.ne.u32 p, %1, 0;\n\t"
                     "setp.lt.and.u32 p, %0, %2, p;\n\t"
                     "@p red.shared.or.b32 [%4], %5;\n\t"
                     "@p st.shared.b32 [%0], %3;\n\t"
                     "@p add.u32 %0, %0, %6;\n\t}"
                     : "+r"(dst) : "r"((uint32_t)fresh), "r"(end), "r"(id[i]), "r"(a[i]), "r"(1u << (id[i] & 31)), "n"(SLOT_PITCH) : "memory");
      }
    };
#pragma unroll 1
    for (; t0 < alone && dst < end; t0 += 4) {
      uint32_t id[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) id[i] = __umulhi(rr_draw_u32(rk, layer, (uint32_t)(t0 + i)), (uint32_t)v);
      accept(id);
    }
    // A row with few free chunks needs many draws (65 chunks, 48 of them excluded, 16 to draw: 150):
    // what is left after 4 r draws is drawn by the warp, 32 at a time, a row after the other.
    // (All lanes read the marks of the row's lane: they are visible before the vote, which waits for every lane.  A
    // __syncwarp() here made whole passes 1-4 % longer, the fence costs nothing.)
    __threadfence_block();
    unsigned left = __ballot_sync(FULL, dst < end);
#pragma unroll 1
    while (left) {
      const int src = __ffs(left) - 1;
      left &= left - 1;
      const uint32_t o_bits = __shfl_sync(FULL, bits, src), o_end = __shfl_sync(FULL, end, src);
      const uint32_t o_v = (uint32_t)__shfl_sync(FULL, v, src);
      const unsigned long long o_rk = __shfl_sync(FULL, rk, src);
      uint32_t o_dst = __shfl_sync(FULL, dst, src);
      int t = __shfl_sync(FULL, t0, src);
#pragma unroll 1
      for (; t < limit && o_dst < o_end; t += 32) {
        const uint32_t id = __umulhi(rr_draw_u32(o_rk, layer, (uint32_t)(t + lane)), o_v);
        const uint32_t a = o_bits + (id >> 5) * WORD_PITCH, bit = 1u << (id & 31);
        const unsigned lt = (1u << lane) - 1u, same = __match_any_sync(FULL, id);
        const bool ok = t + lane < limit && (lds32(a) & bit) == 0u && (same & lt) == 0u;
        const unsigned oks = __ballot_sync(FULL, ok);
        const uint32_t at = o_dst + (uint32_t)__popc(oks & lt) * SLOT_PITCH;
        if (ok && at < o_end) {
          asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(a), "r"(bit) : "memory");
          sts32(at, id);
        }
        o_dst = min(o_end, o_dst + (uint32_t)__popc(oks) * SLOT_PITCH);
        __syncwarp();
      }
      if (lane == src) dst = o_dst;
    }
    if (go && !drawing) dst = col;
    // the whole pool, or the bounded-work fill: smallest free chunks first
    if (go && pool > 0) {
      for (int w = 0; w * 32 < v && dst < end; ++w) {
        uint32_t fr = ~lds32(bits + (uint32_t)w * WORD_PITCH);
        if (v - w * 32 < 32) fr &= (1u << (v - w * 32)) - 1u;
        for (; fr != 0u && dst < end; fr &= fr - 1u) {
          sts32(dst, (uint32_t)(w * 32 + __ffs(fr) - 1));
          dst += SLOT_PITCH;
        }
      }
    }
    if (go) {
      for (; dst < end; dst += SLOT_PITCH) sts32(dst, 0xFFFFFFFFu);
      if (((p.m | p.r | p.sw) & 3) == 0) {
        for (int e = 0; e < p.r; e += 4)
          *reinterpret_cast<int4*>(rnd + e) =
              make_int4((int)lds32(col + (uint32_t)e * SLOT_PITCH), (int)lds32(col + (uint32_t)(e + 1) * SLOT_PITCH),
                        (int)lds32(col + (uint32_t)(e + 2) * SLOT_PITCH), (int)lds32(col + (uint32_t)(e + 3) * SLOT_PITCH));
      } else {
        for (int e = 0; e < p.r; ++e) rnd[e] = (int)lds32(col + (uint32_t)e * SLOT_PITCH);
      }
    }
  } else if (go) {            // more sentinels than the column has places: straight to memory
    int taken = 0;
    auto put = [&](int id) { sts32(word(id), lds32(word(id)) | (1u << (id & 31))); rnd[taken++] = id; };
    auto is_free = [&](int id) { return !((lds32(word(id)) >> (id & 31)) & 1u); };
    const unsigned long long rk = rr_row_key(p.seed, (uint32_t)g);
    for (int t = 0; t < 64 * p.r && taken < p.r && pool > p.r; ++t) {
      const int id = (int)__umulhi(rr_draw_u32(rk, layer, (uint32_t)t), (uint32_t)v);
      if (is_free(id)) put(id);
    }
    for (int id = 0; id < v && taken < p.r && pool > 0; ++id)
      if (is_free(id)) put(id);
    for (; taken < p.r; ++taken) rnd[taken] = -1;
  }
}

}  // namespace rr_select
