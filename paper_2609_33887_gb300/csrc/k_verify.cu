// Merge of the verification partials and the acceptance rules of speculative
// decoding (typical-acceptance and lossless-reference appendices), for a whole
// grid of eps settings in one pass.
//
// One CTA per request, a warp per row (up to 16). A warp merges the partial slots
// of its row (lanes split the slots, a lane's loads issued together, then a
// shuffle tree) into the row's softmax state
// (max M, sum S, argmax A, first moment T in log2 units) and draft logit; lane
// 0 then derives
//   p(x) = exp(l_x - M) / S,   H = ln S - T / (S log2 e)
// and sets bit k when p(x) > min(eps_k, sqrt(eps_k) exp(-H)) and bit 31 when
// the draft equals the argmax. The CTA finally counts, per setting, the
// accepted prefix of the request's draft rows.
#include "kernels.h"

namespace bd {

namespace {
constexpr int MAX_WARPS = 16;
constexpr int MAX_ROWS = 33;  // n_draft <= 32 drafts + the bonus row
// Partial slots a lane loads at once. A verification of 40 rows (d = 4096,
// V = 128256) takes 163 us, 166.5 us with four warps that took two rows each in
// turn and one slot at a time.
constexpr int BATCH = 3;
}  // namespace

__global__ void __launch_bounds__(32 * MAX_WARPS) merge_verify_kernel(VerifyArgs a) {
  __shared__ uint32_t bits_s[MAX_ROWS];
  const int q = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int D = a.n_draft, Rq = D + 1;
  griddep_launch_dependents();  // a kernel behind this one waits for it before touching memory
  griddep_wait();               // the partials come from the LM-head kernel
  // partial slots per row over the plan's launches (header word)
  const int ns = a.n_rows[HDR_SLOTS];

  for (int i = warp; i < Rq; i += static_cast<int>(blockDim.x >> 5)) {
    const int r = q * Rq + i;
    float m = -INFINITY, s = 0.f, t = 0.f, lx = -INFINITY;
    int arg = 0x7fffffff;
#pragma unroll 1
    for (int slot = lane; slot < ns; slot += 32 * BATCH) {
      float pm[BATCH], ps[BATCH], pt[BATCH], px[BATCH];
      int pa[BATCH];
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int64_t o = static_cast<int64_t>(slot + 32 * u) * a.P + r;
        const bool in = slot + 32 * u < ns;
        pm[u] = in ? a.part_m[o] : -INFINITY;
        ps[u] = in ? a.part_s[o] : 0.f;
        pa[u] = in ? a.part_a[o] : 0x7fffffff;
        pt[u] = in ? a.part_t[o] : 0.f;
        px[u] = in ? a.part_x[o] : -INFINITY;
      }
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        softmax_combine_t(m, s, arg, t, pm[u], ps[u], pa[u], pt[u]);
        lx = fmaxf(lx, px[u]);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
      const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
      const int a2 = __shfl_xor_sync(0xffffffffu, arg, o);
      const float t2 = __shfl_xor_sync(0xffffffffu, t, o);
      softmax_combine_t(m, s, arg, t, m2, s2, a2, t2);
      lx = fmaxf(lx, __shfl_xor_sync(0xffffffffu, lx, o));
    }
    if (lane == 0) {
      const int x = a.draft_row[r];
      const float H = logf(s) - t / (s * LOG2E);
      const float px = (x >= 0 && lx != -INFINITY) ? ex2_approx((lx - m) * LOG2E) / s : 0.f;
      uint32_t bits = 0;
      if (x >= 0) {
        const float eh = expf(-H);
        for (int k = 0; k < a.E; ++k)
          if (px > fminf(a.eps[k], a.sqrt_eps[k] * eh)) bits |= 1u << k;
        if (x == arg) bits |= 1u << 31;
      }
      a.out_tokens[r] = arg;
      a.out_p_draft[r] = px;
      a.out_entropy[r] = H;
      a.out_accept[r] = bits;
      bits_s[i] = bits;
    }
  }
  __syncthreads();
  if (threadIdx.x <= a.E) {
    const int k = threadIdx.x;
    const int bit = k == a.E ? 31 : k;
    int n = 0;
    while (n < D && ((bits_s[n] >> bit) & 1u)) ++n;
    a.out_accepted[static_cast<int64_t>(q) * (a.E + 1) + k] = n;
  }
}

cudaError_t launch_merge_verify(const VerifyArgs& a, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(a.n_req), 1, 1);
  const int rows = a.n_draft + 1;
  cfg.blockDim = dim3(32 * (rows < MAX_WARPS ? rows : MAX_WARPS), 1, 1);  // at least two warps: E + 1 <= 32 settings
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, merge_verify_kernel, a);
}

}  // namespace bd
