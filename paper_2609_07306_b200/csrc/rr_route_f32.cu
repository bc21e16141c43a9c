// fp32 inputs: scores, challenge test and routing of a row tile in ONE kernel (Eq. 1, 2, 5; Sections
// 3.1-3.4, 4.2).  The tensor cores take no fp32 operands, so the scores are fused multiply-adds on
// the FP32 pipe, in ascending k like a plain dot product.
//
// One CTA owns R consecutive query rows of one problem (R = 16, or 8 where 16 would leave SMs idle)
// and keeps their complete score rows in shared memory as order-preserving keys:
//   1. scores: a thread takes two key chunks at a time and all R rows, two rows to a packed
//      fma.rn.f32x2; Kc comes straight from L2 in whole 32-byte sectors, Qc is transposed in shared
//      memory so that a 16-byte broadcast read feeds two packed operands (16 packed FMAs per four
//      such reads at R = 16);
//   2. a relay's test: a warp per row picks its candidates' scores out of the row (alpha, beta,
//      Eq. 5) -- the row is there anyway, so nothing is gathered from Kc;
//   3. rows that fail it (an anchor: all rows) are routed on the spot by the warp-level radix
//      select (rr_warp_topk.cuh), sentinels included.  The compaction kernel then only builds the list.
// Scoring the whole strip costs n_k / c times the multiply-adds of the candidates alone, but reuses
// every Kc row R times; the gathered form (rr_rescore.cu) moves c Kc rows per query row and needs a
// second GEMM and a second kernel for the refresh (10 x 384 x 192, c = 48: 135 + 7 + 9 us a relay layer,
// this kernel 21).  At that size (480 CTAs of 8 rows) it is bound by latency, not by the FP32 pipe, which
// needs 1.3 us: Kc loads with nothing loaded ahead, warps without a chunk at the barrier, and where
// rows are routed the select's shared-memory round trips (two thirds of an anchor's instructions).
#include "rr_warp_topk.cuh"

namespace {

constexpr int WARPS = 8, NT = WARPS * 32, COLS = 2 * NT;       // key chunks per pass over the strip
constexpr unsigned FULL = 0xFFFFFFFFu;

__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pair(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}

template <int D, int R>
__global__ void __launch_bounds__(NT)
route_f32_kernel(RRParams p, const float* __restrict__ qc, const float* __restrict__ kc, int anchor, uint32_t layer) {
  extern __shared__ __align__(16) uint32_t smem[];
  const int nk_pad = (p.n_k + 31) & ~31, words = nk_pad / 32;
  float* const qt = reinterpret_cast<float*>(smem);            // [D][R]
  uint32_t* const keys = smem + D * R;                         // [R][nk_pad]
  uint32_t* const scratch = keys + (size_t)R * nk_pad;         // per warp: histogram, bitmap
  __shared__ unsigned int s_flagged, s_cand;
  __shared__ unsigned long long s_full;

  rr_pdl_wait();
  rr_pdl_trigger();
  const int tiles = (p.n_q + R - 1) / R;
  const int prob = blockIdx.x / tiles, row0 = (tiles - 1 - blockIdx.x % tiles) * R;   // heaviest first
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool all = anchor || (p.force_threshold > 0 && p.force_in[0] > 0);   // (a forced call routes every row)
  if (tid == 0) { s_flagged = 0; s_cand = 0; s_full = 0; }
  for (int e = tid; e < D * R; e += NT) {
    const int r = e / D, k = e % D;
    qt[k * R + r] = row0 + r < p.n_q ? __ldg(qc + ((size_t)prob * p.n_q + row0 + r) * D + k) : 0.f;
  }
  __syncthreads();

  // ---- 1. score rows ---------------------------------------------------------------------------
  const int last = min(p.n_q, row0 + R) - 1;
  const int vmax = rr_valid_count(last, p.n_k, p.causal, p.causal_offset);
  const float* const kbase = kc + (size_t)prob * p.n_k * D;
  for (int c0 = 0; c0 < vmax; c0 += COLS) {
    if (c0 + (tid & ~31) >= vmax) break;                       // (whole warps)
    const int ca = c0 + tid, cb = ca + NT;
    const float4* const ka = reinterpret_cast<const float4*>(kbase + (size_t)min(ca, p.n_k - 1) * D);
    const float4* const kb = reinterpret_cast<const float4*>(kbase + (size_t)min(cb, p.n_k - 1) * D);
    const bool two = c0 + NT + (tid & ~31) < vmax;             // (warp-uniform)
    unsigned long long acc[2][R / 2];
#pragma unroll
    for (int i = 0; i < R / 2; ++i) { acc[0][i] = 0ull; acc[1][i] = 0ull; }
#pragma unroll 1
    for (int k0 = 0; k0 < D; k0 += 8) {
      float va[8], vb[8];
      *reinterpret_cast<float4*>(va) = __ldg(ka + k0 / 4); *reinterpret_cast<float4*>(va + 4) = __ldg(ka + k0 / 4 + 1);
      if (two) { *reinterpret_cast<float4*>(vb) = __ldg(kb + k0 / 4); *reinterpret_cast<float4*>(vb + 4) = __ldg(kb + k0 / 4 + 1); }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const ulonglong2* const q2 = reinterpret_cast<const ulonglong2*>(qt + (k0 + k) * R);
        const unsigned long long pa = pair(va[k], va[k]), pb = pair(vb[k], vb[k]);
#pragma unroll
        for (int i = 0; i < R / 4; ++i) {
          const ulonglong2 q = q2[i];
          fma2(acc[0][2 * i], q.x, pa); fma2(acc[0][2 * i + 1], q.y, pa);
          if (two) { fma2(acc[1][2 * i], q.x, pb); fma2(acc[1][2 * i + 1], q.y, pb); }
        }
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = h == 0 ? ca : cb;
      if (c < vmax) {
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
          keys[(size_t)(2 * i) * nk_pad + c] = rr_order_key(__uint_as_float((uint32_t)acc[h][i]));
          keys[(size_t)(2 * i + 1) * nk_pad + c] = rr_order_key(__uint_as_float((uint32_t)(acc[h][i] >> 32)));
        }
      }
    }
  }
  __syncthreads();

  // ---- 2., 3. a warp per row: challenge test, routing --------------------------------------------
  const float pinf = __int_as_float(0x7f800000), ninf = __int_as_float(0xff800000);
  for (int r = warp; r < R && row0 + r < p.n_q; r += WARPS) {
    const int i = row0 + r, g = prob * p.n_q + i;
    const int v = rr_valid_count(i, p.n_k, p.causal, p.causal_offset);
    const uint32_t* const krow = keys + (size_t)r * nk_pad;
    bool flag = true;
    if (!all) {
      float amin = pinf, bmax = ninf;
      int n = 0; bool bad = false;
      for (int s = lane; s < p.c; s += 32) {
        const int id = s < p.k ? p.routes[(size_t)g * p.k + s] : p.sentinels[(size_t)g * p.sw + s - p.k];
        bad |= id >= v;
        const bool ok = id >= 0 && id < v;
        const float sc = ok ? rr_key_to_float(krow[id]) : 0.f;
        if (ok) { ++n; if (s < p.k) amin = fminf(amin, sc); else bmax = fmaxf(bmax, sc); }
        if (p.debug) p.cand_scores[(size_t)g * p.c + s] = ok ? sc : __int_as_float(0x7fc00000);
      }
#pragma unroll
      for (int off = 16; off; off >>= 1) {
        amin = fminf(amin, __shfl_xor_sync(FULL, amin, off));
        bmax = fmaxf(bmax, __shfl_xor_sync(FULL, bmax, off));
      }
      n = __reduce_add_sync(FULL, n);
      if (__any_sync(FULL, bad) && lane == 0) atomicOr(p.status, RR_STATUS_BAD_INDEX);
      flag = rr_challenge(p, g, amin, bmax);
      if (lane == 0) {
        p.flags[g] = flag ? 1 : 0; p.alpha[g] = amin; p.beta[g] = bmax;
        atomicAdd(&s_cand, (unsigned)n);
        if (flag) { atomicAdd(&s_flagged, 1u); atomicAdd(&s_full, (unsigned long long)v); }
      }
      __syncwarp();
    }
    if (flag) {
      uint32_t* const hist = scratch + warp * (256 + words);
      warptopk::route_row(p, krow, hist, hist + 256, g, v, layer, lane);
      __syncwarp();
    }
  }
  if (!all) {
    __syncthreads();
    if (tid == 0) {
      rr_store_count<RR_COUNT_WORDS_F32>(p, prob, row0, R, (int)s_flagged);
      atomicAdd(&p.counters[RR_CNT_FLAGGED_ROWS], (unsigned long long)s_flagged);
      atomicAdd(&p.counters[RR_CNT_CAND_PAIRS], (unsigned long long)s_cand);
      atomicAdd(&p.counters[RR_CNT_FULL_PAIRS], s_full);
    }
  }
}

size_t smem_bytes(const RRParams& p, int R) {
  const size_t nk_pad = (p.n_k + 31) & ~31;
  return ((size_t)p.d * R + (size_t)R * nk_pad + (size_t)WARPS * (256 + nk_pad / 32)) * 4;
}
constexpr int MAX_SMEM = 200 * 1024;

typedef void (*Kernel)(RRParams, const float*, const float*, int, uint32_t);
Kernel kernel_of(int d, int R) {
  return d == 128 ? (R == 16 ? route_f32_kernel<128, 16> : route_f32_kernel<128, 8>)
                  : (R == 16 ? route_f32_kernel<64, 16> : route_f32_kernel<64, 8>);
}

}  // namespace

bool rr_route_f32_supported(const RRParams& p) {
  return p.dtype == RR_F32 && (p.d == 64 || p.d == 128) && smem_bytes(p, 8) <= MAX_SMEM;
}

cudaError_t rr_launch_route_f32(const RRParams& p, const void* qc, const void* kc, int anchor, int layer,
                                cudaStream_t st) {
  if (!rr_route_f32_supported(p)) return cudaErrorInvalidConfiguration;
  static unsigned long long attr_done = 0;      // devices on which the attributes are set
  const cudaError_t e = rr_once_per_device(attr_done, [] {
    for (int d = 64; d <= 128; d += 64)
      for (int R = 8; R <= 16; R += 8) {
        const cudaError_t a = cudaFuncSetAttribute((const void*)kernel_of(d, R), cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM);
        if (a != cudaSuccess) return a;
      }
    return cudaSuccess;
  });
  if (e != cudaSuccess) return e;
  // 16 rows per CTA reuse Kc twice as often; 8 where 16 would not give every SM two CTAs, or would
  // not fit the score rows
  const int R = p.P * ((p.n_q + 15) / 16) >= 2 * rr_sm_count() && smem_bytes(p, 16) <= MAX_SMEM ? 16 : 8;
  const int grid = p.P * ((p.n_q + R - 1) / R);
  const cudaError_t l = rr_launch_pdl(kernel_of(p.d, R), grid, NT, smem_bytes(p, R), st, p, (const float*)qc,
                                      (const float*)kc, anchor, (uint32_t)layer);
  rr_count_launch();
  return l;
}
