// A minimal consumer of the routes (Eq. 3): o_i = softmax(q_i K_R^T * scale) V_R over the tokens
// R that row i's token ranges cover -- the ranges rr_route_* writes when chunk_tokens > 0, one per
// route slot or, with coalesce_ranges, one per run of consecutive chunks.  It shows that the
// range layout is directly consumable and gives the tests an end-to-end check; it is FP32 arithmetic
// on the ordinary pipes, not a tuned attention backend: the paper leaves the sparse-attention
// backend unchanged (Section 4.3).
//
// Every query row has its own tokens, so the work is a matrix-vector product per row and the floor is
// the traffic of its K and V rows through L2.  A CTA of four warps takes one row.  The row's
// tokens are numbered in ascending order through its ranges (a prefix sum over the slots, a binary
// search per token); block b of 32 tokens goes to warp b % 4, which keeps a running maximum, sum and
// output (online softmax), and the four parts are merged in warp order.  The split depends on a
// token's number only, never on how tokens are grouped into ranges, so coalesced and per-slot ranges
// give bit-identical outputs.
//   K: dh / 8 lanes (bf16) read one token's row with a 16-byte load each, 32 / lanes tokens at a time;
//      the partial dot products of a block are reduced together (each exchange step halves the number
//      of values a lane holds: 15 shuffles for 32 tokens at dh = 128), leaving a lane one logit;
//   V: the same loads; a lane accumulates the 8 output dimensions it loads.
// A first version (one warp per row, a lane per token for K, two passes) read K with 32 separate
// cache lines per load and computed every logit twice: 2400 us for 2048 rows of 1024 tokens, dh = 128,
// bf16; this one: 101 us (1.07 GB of K and V rows, 10.6 TB/s from L2).  Widths that do not split into 16-byte lanes keep it.
#include <type_traits>
#include "rr_common.cuh"

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int WARPS = 4, MAX_DH = 256;

template <typename T> __device__ __forceinline__ float to_f32(T x);
template <> __device__ __forceinline__ float to_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }

template <typename T>
__global__ void __launch_bounds__(WARPS * 32)
attend_ranges_kernel(const int32_t* __restrict__ ranges, int rows, int slots, int n_q,
                     const T* __restrict__ q, const T* __restrict__ keys, const T* __restrict__ values,
                     int tokens, int dh, float scale, float* __restrict__ out) {
  __shared__ float s_q[WARPS][MAX_DH];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * WARPS + warp;
  if (row >= rows) return;
  const int prob = row / n_q;
  for (int e = lane; e < dh; e += 32) s_q[warp][e] = to_f32(q[(size_t)row * dh + e]);
  __syncwarp();
  const T* kp = keys + (size_t)prob * tokens * dh;
  const T* vp = values + (size_t)prob * tokens * dh;
  const int32_t* rg = ranges + (size_t)row * slots * 2;
  const float ninf = __int_as_float(0xff800000);

  auto logit = [&](int t) -> float {
    const T* kr = kp + (size_t)t * dh;
    float acc = 0.f;
    for (int e = 0; e < dh; ++e) acc = fmaf(s_q[warp][e], to_f32(kr[e]), acc);
    return acc * scale;
  };
  // pass 1: the maximum logit
  float mx = ninf;
  for (int s = 0; s < slots; ++s) {
    const int lo = rg[2 * s], hi = min(rg[2 * s + 1], tokens);
    if (lo < 0) continue;
    for (int t0 = lo; t0 < hi; t0 += 32) {
      const int t = t0 + lane;
      if (t < hi) mx = fmaxf(mx, logit(t));
    }
  }
#pragma unroll
  for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, off));
  // pass 2: sums in token order; lane owns output dimensions lane, lane + 32, ...
  float acc[MAX_DH / 32];
#pragma unroll
  for (int i = 0; i < MAX_DH / 32; ++i) acc[i] = 0.f;
  float denom = 0.f;
  for (int s = 0; s < slots; ++s) {
    const int lo = rg[2 * s], hi = min(rg[2 * s + 1], tokens);
    if (lo < 0) continue;
    for (int t0 = lo; t0 < hi; t0 += 32) {
      const int t = t0 + lane;
      const float w = t < hi ? expf(logit(t) - mx) : 0.f;
      const int n = min(32, hi - t0);
      for (int u = 0; u < n; ++u) {
        const float wu = __shfl_sync(FULL, w, u);
        denom += wu;
        const T* vr = vp + (size_t)(t0 + u) * dh;
#pragma unroll
        for (int i = 0; i < MAX_DH / 32; ++i)
          if (lane + 32 * i < dh) acc[i] = fmaf(wu, to_f32(vr[lane + 32 * i]), acc[i]);
      }
    }
  }
  const float inv = denom > 0.f ? 1.f / denom : 0.f;
#pragma unroll
  for (int i = 0; i < MAX_DH / 32; ++i)
    if (lane + 32 * i < dh) out[(size_t)row * dh + lane + 32 * i] = acc[i] * inv;
}

// ---- 16-byte lanes -----------------------------------------------------------------------------
template <typename T> struct Lane;
template <> struct Lane<__nv_bfloat16> {
  static constexpr int N = 8;
  static __device__ __forceinline__ void load(const __nv_bfloat16* ptr, float (&x)[8]) {
    const uint4 t = __ldg(reinterpret_cast<const uint4*>(ptr));
    const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { x[2 * i] = __uint_as_float(w[i] << 16); x[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u); }
  }
};
template <> struct Lane<float> {
  static constexpr int N = 4;
  static __device__ __forceinline__ void load(const float* ptr, float (&x)[4]) {
    *reinterpret_cast<float4*>(x) = __ldg(reinterpret_cast<const float4*>(ptr));
  }
};

// LPT: lanes per token (dh = LPT * Lane<T>::N)
template <typename T, int LPT>
__global__ void __launch_bounds__(WARPS * 32)
attend_row_kernel(const int32_t* __restrict__ ranges, int slots, int n_q, const T* __restrict__ q,
                  const T* __restrict__ keys, const T* __restrict__ values, int tokens, float scale,
                  float* __restrict__ out) {
  constexpr int E = Lane<T>::N, DH = LPT * E, TP = 32 / LPT;   // elements per lane, tokens per load
  extern __shared__ int32_t s_slots[];                         // [slots + 1] first token number, [slots] start - first
  __shared__ float s_acc[WARPS][DH], s_m[WARPS], s_l[WARPS];
  int32_t* const s_first = s_slots;
  int32_t* const s_base = s_slots + slots + 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x;
  const int32_t* const rg = ranges + (size_t)row * slots * 2;
  if (warp == 0) {                                             // number the row's tokens
    int run = 0;
    for (int s0 = 0; s0 < slots; s0 += 32) {
      const int s = s0 + lane;
      int lo = 0, len = 0;
      if (s < slots) { lo = rg[2 * s]; len = lo < 0 ? 0 : max(0, min(rg[2 * s + 1], tokens) - lo); }
      int incl = len;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) { const int t = __shfl_up_sync(FULL, incl, off); if (lane >= off) incl += t; }
      if (s < slots) { s_first[s] = run + incl - len; s_base[s] = lo - (run + incl - len); }
      run += __shfl_sync(FULL, incl, 31);
    }
    if (lane == 0) s_first[slots] = run;
  }
  __syncthreads();
  const int n_tok = s_first[slots];
  const int sub = lane % LPT, grp = lane / LPT;
  const size_t prob = (size_t)(row / n_q) * tokens;
  const T* const kp = keys + prob * DH + sub * E;
  const T* const vp = values + prob * DH + sub * E;
  float qv[E], acc[E];
  Lane<T>::load(q + (size_t)row * DH + sub * E, qv);
#pragma unroll
  for (int e = 0; e < E; ++e) acc[e] = 0.f;
  const float ninf = __int_as_float(0xff800000);
  float m = ninf, l = 0.f;
  // One block of 32 tokens, or the row's last one with n_last: its empty places repeat the last token with
  // weight 0 -- and a value of 0, as its row may hold an infinity.
  auto block = [&](int b0, int n_last, auto whole) {
    const int n = decltype(whole)::value ? 32 : n_last;
    // token of number b0 + lane: the last slot that starts at or before it (empty slots start where
    // the next one does and are passed over)
    const int num = b0 + min(lane, n - 1);
    int s = 0, hi = slots;
    while (hi - s > 1) { const int mid = (s + hi) >> 1; if (s_first[mid] <= num) s = mid; else hi = mid; }
    const int tok = s_base[s] + num;
    float part[LPT];                                           // step i: token i * TP + grp of the block
#pragma unroll
    for (int i = 0; i < LPT; ++i) {
      float kv[E];
      Lane<T>::load(kp + (size_t)__shfl_sync(FULL, tok, i * TP + grp) * DH, kv);
      float d = 0.f;
#pragma unroll
      for (int e = 0; e < E; ++e) d = fmaf(qv[e], kv[e], d);
      part[i] = d;
    }
    // sum over a token's lanes; lane `sub` is left with step `sub`
#pragma unroll
    for (int off = LPT / 2; off >= 1; off >>= 1) {
      const bool up = (sub & off) != 0;
#pragma unroll
      for (int i = 0; i < off; ++i) {
        const float mine = up ? part[i + off] : part[i], give = up ? part[i] : part[i + off];
        part[i] = mine + __shfl_xor_sync(FULL, give, off);
      }
    }
    const int my = sub * TP + grp;                             // this lane's token of the block
    const float logit = my < n ? part[0] * scale : ninf;
    float bm = logit;
#pragma unroll
    for (int off = 16; off; off >>= 1) bm = fmaxf(bm, __shfl_xor_sync(FULL, bm, off));
    // while the warp has met nothing but -inf, 0 stands for the maximum (-inf - -inf would be NaN)
    const float m_new = fmaxf(m, bm), m_ref = m_new == ninf ? 0.f : m_new;
    const float f = expf(m - m_ref), w = expf(logit - m_ref);
    l = l * f + w;
    m = m_new;
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] *= f;
#pragma unroll
    for (int i = 0; i < LPT; ++i) {
      float vv[E];
      Lane<T>::load(vp + (size_t)__shfl_sync(FULL, tok, i * TP + grp) * DH, vv);
      const float wi = __shfl_sync(FULL, w, grp * LPT + i);
#pragma unroll
      for (int e = 0; e < E; ++e) acc[e] = fmaf(wi, i * TP + grp < n ? vv[e] : 0.f, acc[e]);
    }
  };
  int b0 = warp * 32;
  for (; b0 + 32 <= n_tok; b0 += WARPS * 32) block(b0, 32, std::true_type());
  if (b0 < n_tok) block(b0, n_tok - b0, std::false_type());
#pragma unroll
  for (int off = LPT; off < 32; off <<= 1)                     // the token groups of the warp
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] += __shfl_xor_sync(FULL, acc[e], off);
#pragma unroll
  for (int off = 16; off; off >>= 1) l += __shfl_xor_sync(FULL, l, off);
  if (grp == 0) {
#pragma unroll
    for (int e = 0; e < E; ++e) s_acc[warp][sub * E + e] = acc[e];
  }
  if (lane == 0) { s_m[warp] = m; s_l[warp] = l; }
  __syncthreads();
  float mx = ninf;
#pragma unroll
  for (int w = 0; w < WARPS; ++w) mx = fmaxf(mx, s_m[w]);
  float fw[WARPS], den = 0.f;
#pragma unroll
  for (int w = 0; w < WARPS; ++w) { fw[w] = s_m[w] == ninf ? 0.f : expf(s_m[w] - mx); den = fmaf(s_l[w], fw[w], den); }
  // (tokens that all score -inf have no softmax: NaN, as without the split; a row without tokens gives 0)
  const float inv = den > 0.f ? 1.f / den : n_tok > 0 ? __int_as_float(0x7fc00000) : 0.f;
  for (int e = threadIdx.x; e < DH; e += WARPS * 32) {
    float o = 0.f;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) o = fmaf(s_acc[w][e], fw[w], o);
    out[(size_t)row * DH + e] = o * inv;
  }
}

template <typename T>
bool launch_rows(const int32_t* ranges, int rows, int slots, int n_q, const void* q, const void* keys,
                 const void* values, int tokens, int dh, float scale, float* out, cudaStream_t st) {
  const size_t smem = (size_t)(2 * slots + 1) * sizeof(int32_t);
  if (smem > 40 * 1024 || dh % Lane<T>::N != 0 || (((uintptr_t)q | (uintptr_t)keys | (uintptr_t)values) & 15u) != 0) return false;
  auto go = [&](auto kernel) {
    kernel<<<rows, WARPS * 32, smem, st>>>(ranges, slots, n_q, (const T*)q, (const T*)keys, (const T*)values, tokens, scale, out);
    return true;
  };
  switch (dh / Lane<T>::N) {
    case 8: return go(attend_row_kernel<T, 8>);
    case 16: return go(attend_row_kernel<T, 16>);
    case 32: return go(attend_row_kernel<T, 32>);
    default: return false;
  }
}

}  // namespace

extern "C" int rr_attend_token_ranges(const int32_t* ranges, int32_t rows, int32_t slots, int32_t n_q,
                                      const void* q, const void* keys, const void* values,
                                      int32_t tokens, int32_t dh, int32_t dtype, float scale,
                                      float* out, void* stream) {
  if (!ranges || !q || !keys || !values || !out) return RR_ERR_INVALID_ARG;
  if (rows <= 0 || slots <= 0 || n_q <= 0 || rows % n_q != 0 || tokens <= 0) return RR_ERR_INVALID_ARG;
  if (dh <= 0 || dh > MAX_DH) return RR_ERR_UNSUPPORTED;
  if (dtype != RR_BF16 && dtype != RR_F32) return RR_ERR_UNSUPPORTED;
  cudaStream_t st = (cudaStream_t)stream;
  const int grid = (rows + WARPS - 1) / WARPS;
  const bool done = dtype == RR_BF16
      ? launch_rows<__nv_bfloat16>(ranges, rows, slots, n_q, q, keys, values, tokens, dh, scale, out, st)
      : launch_rows<float>(ranges, rows, slots, n_q, q, keys, values, tokens, dh, scale, out, st);
  if (done) {
  } else if (dtype == RR_BF16)
    attend_ranges_kernel<__nv_bfloat16><<<grid, WARPS * 32, 0, st>>>(
        ranges, rows, slots, n_q, (const __nv_bfloat16*)q, (const __nv_bfloat16*)keys,
        (const __nv_bfloat16*)values, tokens, dh, scale, out);
  else
    attend_ranges_kernel<float><<<grid, WARPS * 32, 0, st>>>(
        ranges, rows, slots, n_q, (const float*)q, (const float*)keys, (const float*)values, tokens,
        dh, scale, out);
  rr_count_launch();
  return cudaPeekAtLastError() == cudaSuccess ? RR_OK : RR_ERR_CUDA;
}
