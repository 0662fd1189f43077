// Step 2 as its own kernel (avtp_allocate): one warp per request runs the budget
// rule of avtp_alloc.cuh (paper §3.3.3 adaptive keep ratio, App. A.2 clamps) and
// writes the request's budgets: a lane per image for requests of up to 32 images,
// four or eight images a lane up to 256, shared memory beyond. avtp_prune of more than kFusedImages images
// runs it between the scores and k_select.
// Latency and instruction fetches bound it: right behind the scoring stream, which sweeps L2,
// a cold run of the rule takes 15-25 us, most of it fetching code. The first warm_ctas CTAs,
// which start beside the scoring on an SM left free for them, run the rule once on made-up sums
// before they wait: the stage of 64 images of one request 72 -> 67 us, of eight requests of five
// images 68 -> 61 us. The CTAs that start behind the scoring have nothing to hide it behind.
#include "avtp_alloc.cuh"

namespace avtp {
namespace {

constexpr int kMaxWarpsPerCta = 4;
constexpr size_t kSmemBudget = 200 * 1024;
static_assert(warp_alloc_smem_bytes(kMaxImagesPerRequest) <= kSmemBudget, "one warp's scratch fits at any size");

__global__ void __launch_bounds__(kMaxWarpsPerCta * 32, 1)
k_allocate(const int32_t* __restrict__ img_cu, const int32_t* __restrict__ img_len,
           const int64_t* __restrict__ img_sums, const float* __restrict__ keep_ratio, float alpha, float r_min,
           float r_max, int relative, const int32_t* __restrict__ vis_cu, int32_t* req_budget,
           int32_t* __restrict__ budgets, int R, int NI, int m_cap, int warm_ctas, DevStatus* st) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = blockIdx.x * (blockDim.x >> 5) + warp;
  if (r >= R) return;
  // ---- from the call's inputs, beside the kernel before this one; the layout may not be
  // validated yet, so the spans are clamped
  const int i0 = min(max(img_cu[r], 0), NI);
  const int m = min(min(max(img_cu[r + 1], i0), NI) - i0, m_cap);
  const WarpAllocSmem sm = carve_warp_alloc(smem + static_cast<size_t>(warp) * warp_alloc_smem_bytes(m_cap), m_cap);
  int32_t n = 0;
  for (int j = lane; j < m; j += 32) {
    n = min(max(img_len[i0 + j], 0), kMaxVisualPerRequest);
    sm.n[j] = n;
  }
  const float kr = keep_ratio[r];
  const RatioRule rule = make_ratio_rule(kr, alpha, relative);
  const int64_t inv_n = recip62(n);
  int32_t K = 0;
  int err = AVTP_OK;
  // one copy of the code for the warm-up and the real run
#pragma unroll 1
  for (int pass = static_cast<int>(blockIdx.x) < warm_ctas && m <= kMultiImages ? 0 : 1; pass < 2; ++pass) {
    int64_t S = 0, B;
    int32_t N;
    if (pass == 1) {
      pdl_wait();
      pdl_trigger();
      // ---- one round of loads
      const int ok = st->layout_ok;
      const int32_t v0 = vis_cu[i0], v1 = vis_cu[i0 + m];
      B = req_budget[r];
      for (int j = lane; j < m; j += 32) {
        S = img_sums[i0 + j];
        if (m > 32) sm.S[j] = S;
      }
      if (!ok || m == 0) return;
      N = v1 - v0;
    } else {
      // made-up sums. A lane per image: one image far above the others, so that clamps bind and
      // the grid's shift is fetched too (eight requests of eight images 82.4 -> 79.5 us).
      // Several images a lane: means that differ by a little from image to image, so that no
      // clamp binds, and by odd numbers, so that no remainders of images of one size tie at the
      // cut. What these forms leave to the general stage is left out here (dry), as are requests
      // that only that stage serves: it takes longer than most scorings. (With equal means all
      // odd sizes tie: the stage of one request of 40 images of 729 tokens took 163 us, without
      // ties 108; of 128 of 65 tokens, hidden 256, 182 and 25.)
      int64_t nn = 0;
      for (int j = lane; j < m; j += 32) {
        nn += sm.n[j];
        S = m <= 32 ? static_cast<int64_t>(sm.n[j]) << (j == 0 ? 40 : 30)
                    : sm.n[j] * ((int64_t(1) << 30) + j * ((int64_t(1) << 18) - 1));
        if (m > 32) sm.S[j] = S;
      }
      nn = warp_sum(nn);
      if (nn <= 0 || nn > kMaxVisualPerRequest) continue;
      N = static_cast<int32_t>(nn);
      B = N / 2;
    }
    if (m <= 32) {
      err = warp_allocate32(sm, m, S, n, inv_n, B, N, recip62(N), rule, alpha, r_min, r_max, &K, pass == 0);
    } else {
      __syncwarp();
      err = warp_allocate(sm, m, B, N, kr, alpha, r_min, r_max, relative, pass == 0);
    }
  }
  if (err != AVTP_OK) {
    if (lane == 0) {
      record_error(st, err, r);
      req_budget[r] = -1;  // the selection behind this kernel leaves the request alone
    }
    return;
  }
  for (int j = lane; j < m; j += 32) budgets[i0 + j] = m <= 32 ? K : sm.K[j];
}

}  // namespace

cudaError_t launch_allocate(const avtp_layout_t& L, const int64_t* img_sums, const avtp_alloc_args_t& aa,
                            int32_t* budgets, void* ws, const WsPlan& p, cudaStream_t s, int warm_ctas) {
  if (L.n_images == 0) return cudaSuccess;
  const int m_cap = L.n_images < kMaxImagesPerRequest ? L.n_images : kMaxImagesPerRequest;
  const size_t per_warp = warp_alloc_smem_bytes(m_cap);
  int wpc = static_cast<int>(kSmemBudget / per_warp);
  wpc = wpc < 1 ? 1 : (wpc > kMaxWarpsPerCta ? kMaxWarpsPerCta : wpc);
  const size_t smem = wpc * per_warp;
  // the attribute belongs to the device and not to the call, and other threads may launch: set
  // once, to the most that any call asks for
  static PerDevice attrs;
  const cudaError_t ae = once_per_device(attrs, [](int, int*) {
    return cudaFuncSetAttribute(k_allocate, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(kSmemBudget));
  });
  if (ae != cudaSuccess) return ae;
  const int grid = (L.n_requests + wpc - 1) / wpc;
  return launch_kernel(k_allocate, dim3(grid), dim3(32 * wpc), smem, s, /*pdl=*/true, L.img_cu, L.img_len, img_sums,
                       aa.keep_ratio, aa.alpha, aa.r_min, aa.r_max, aa.relative, ws_at<int32_t>(ws, p.vis_cu),
                       ws_at<int32_t>(ws, p.req_budget), budgets, L.n_requests, L.n_images, m_cap, warm_ctas,
                       ws_at<DevStatus>(ws, p.status));
}

}  // namespace avtp
