// Configurations and launch of the routing kernel with four threads per row (rr_route_quad.cuh).
#include "rr_route_quad.cuh"

namespace {

// keep = k + max(m, 1) and the number of key chunks decide how many entries a row's column needs: the bound lets
// 1.05-1.25 keep scores pass, and a pair of threads has half of what the column holds beyond keep to itself.  A row
// that needs more takes the slow path, and its CTA runs 12 us longer.
//   keep <= 40: 128 groups, 48 / 64 / 80 entries (fewer than 1 row in 10^4 overflows, up to 2048 chunks);
//   beyond:     256 groups.  80 entries (88 at d = 64) are the longest column that lets two CTAs share an SM; longer
//               ones run with one, with registers to spare.
// MOST: most kept chunks for a column of 80, 88 (d = 64), 104 or 128 entries, by the number of key chunks; 160 entries for
// the rest.  Among the columns with one CTA per SM the lines lie where 1 row in 10^4 to 3 x 10^3 overflows, over random
// rows of every length up to n_k (keep 96 of 2048 chunks: 144 entries overflow in 1 row of 200, which cost 418 -> 372
// us per launch what four threads had gained; 160 entries: 301).  Two CTAs per SM are worth more overflows: six layers
// at rho = 0.2, 80 entries against 104, 256 x 256 x 256, keep 65: 717 and 860 us, keep 70: 765 and 888; 64 x 2048 x
// 2048, keep 56: 1534 and 1783; 200 x 140 x 1024, keep 58: 396 and 505; 88 entries against 104 (d = 64): 100 x 300 x
// 300, keep 72: 455 and 478; 256 x 192 x 192, keep 72: 597 and 779.
struct Plan { int variant, ring_bytes; size_t smem; };
constexpr struct { int n_k, cap80, cap88, cap104, cap128; } MOST[] = {
    {256, 70, 76, 76, 88}, {320, 66, 72, 74, 86}, {512, 62, 68, 76, 88}, {1024, 58, 64, 70, 84},
    {1536, 56, 62, 70, 82}, {2048, 56, 0, 68, 82}, {RR_MAX_NK, 0, 0, 66, 80}};   // (0: the bitmaps leave no room for two)

bool plan(const RRParams& p, Plan& out) {
  const int keep = p.k + (p.m > 0 ? p.m : 1);
  if (p.dtype != RR_BF16 || (p.d != 64 && p.d != 128) || p.n_k > RR_MAX_NK || keep > 96) return false;
  if (keep <= 40) {
    out.variant = keep <= 28 ? 0 : keep <= 36 ? 1 : 2;
  } else {
    int i = 0;
    while (p.n_k > MOST[i].n_k) ++i;
    const auto& most = MOST[i];
    const bool narrow = p.k <= 64 && p.m <= 64;      // (with 56 registers a thread orders 64 ids at most)
    out.variant = (narrow && keep <= most.cap80) || keep <= 48 ? 3 : narrow && p.d == 64 && keep <= most.cap88 ? 4
                  : keep <= most.cap104 ? 5 : keep <= most.cap128 ? 6 : 7;
  }
  const int words = (p.n_k + 31) / 32;
  int ring = stages_of(p.d, CTAS_OF[out.variant]) * BN * p.d * 2;
  if (ring < words * (int)WORD_PITCH) ring = words * (int)WORD_PITCH;
  out.ring_bytes = (ring + 1023) / 1024 * 1024;
  out.smem = (size_t)out.ring_bytes + CTL_BYTES + (size_t)std::max(CAPS[out.variant], LIST_SLOTS) * SLOT_PITCH;
  return out.smem <= 227 * 1024;
}

rr_quad_kernel kernel_of(int d, int variant, bool test) { return d == 128 ? rr_quad_kernel_d128(variant, test) : rr_quad_kernel_d64(variant, test); }

// Rows of a CTA that tests its rows itself: as few as leave the grid one CTA per SM.  Every phase of a CTA is as
// long as its pipes need for all of its rows, an idle SM takes rows for nothing: 1 x 1024 x 1024, 16 layers 657 -> 558 us
// (32 rows instead of 128), 4 x 512 x 512 215 -> 201, 15 x 389 x 777 404 -> 387 (64 rows), 8 x 256 x 256 260 -> 251.
int rows_per_test_cta(const RRParams& p) {
  const int sms = rr_sm_count();
  for (int rows = 32; rows < BM; rows *= 2)
    if ((long long)p.P * ((p.n_q + rows - 1) / rows) <= sms) return rows;
  return BM;
}

int ctas_per_sm(const Plan& pl) { return CTAS_OF[pl.variant] == 2 && 2 * (pl.smem + 1024) <= 228 * 1024 ? 2 : 1; }

}  // namespace

bool rr_route_quad_supported(const RRParams& p) { Plan pl; return plan(p, pl); }

// A relay's test inside the routing kernel: every row goes through sweep 1 there, and the test, the list and the launch
// of the routing kernel no longer wait for one another.  Taken where every CTA has an SM to itself, so that the
// rows that pass keep nobody from working: 8 x 256 x 256, twelve layers 371 -> 260 us (without it 361), 15 x 389 x 777
// 485 -> 404 (440).  (A relay without any failing row is the exception: sweep 1 keeps and sorts its maxima for nothing,
// 7 x 1345 x 1915, six layers 181 us where the list has 139.)  With two CTAs to an SM the list is better, dense or not:
// 32 x 1024 x 1024, 97 % flagged 1000 us against 1090, 17 % flagged 820 against 1005.  (Buckets that run side by side
// have a line of their own, rr_buckets.cu.)  The candidates' bitmaps have to fit the column.
bool rr_route_quad_tests(const RRParams& p) {
  Plan pl;
  if (!plan(p, pl) || (p.n_k + 31) / 32 > std::max(CAPS[pl.variant], LIST_SLOTS)) return false;
  return p.n_tiles <= rr_sm_count();
}

cudaError_t rr_launch_route_quad(const RRParams& p, const void* qc, const void* kc, const int32_t* row_list, bool test,
                                 int layer, int hooks, cudaStream_t st) {
  Plan pl;
  if (!plan(p, pl)) return cudaErrorInvalidConfiguration;
  CUtensorMap tmap;
  cudaError_t e = rr_encode_tmap_bf16_tile(&tmap, kc, p.d, p.n_k, p.P, BN);
  if (e != cudaSuccess) return e;
  static unsigned long long attr_done = 0;      // devices on which the attributes are set
  e = rr_once_per_device(attr_done, [] {
    for (int d = 64; d <= 128; d += 64)
      for (int v = 0; v < 2 * VARIANTS; ++v) {
        const void* fn = (const void*)kernel_of(d, v >> 1, v & 1);
        const cudaError_t a = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (a != cudaSuccess) return a;
        cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
      }
    return cudaSuccess;
  });
  if (e != cudaSuccess) return e;
  const int rows = test ? rows_per_test_cta(p) : BM;
  e = rr_launch_pdl(kernel_of(p.d, pl.variant, test), p.P * ((p.n_q + rows - 1) / rows), NT, pl.smem, st, p, (const __nv_bfloat16*)qc, tmap, row_list,
                    (uint32_t)layer, hooks, pl.ring_bytes, ctas_per_sm(pl) * rr_sm_count(), rows);
  rr_count_launch();
  return e;
}
