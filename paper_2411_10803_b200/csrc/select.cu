// Dual criteria, key set and selection: one CTA per request (Eq. 9, Eq. 10; Sec. 3.3 key set).
//
// The work of a request is in select_body.cuh; this file is the stand-alone kernel around it.
#include "select_body.cuh"

namespace mustdrop {
namespace {

__global__ void __launch_bounds__(kSelThreads) select_kernel(SelectParams p) {
  __shared__ SelectShared s;
  __shared__ SelectScratch x;
  extern __shared__ uint32_t val[];   // G and I of the request, M rounded up to 256 words each
  const int tid = threadIdx.x, b = blockIdx.x;
  // Work that touches no global data, then let the next kernel start its prologue and wait for
  // the kernel that produced g / i.
  MD_PIPE(p.workspace, 1, false, false);
  select_clear(s, tid, kSelThreads);
  __syncthreads();
  pdl_launch_dependents();
  pdl_wait();
  const int M = p.vis_cnt ? clamp_vis_cnt(p.vis_cnt[b], p.M) : p.M;
  uint32_t* const val_i = val + select_pad(p.M);
  const float* const g = p.g + static_cast<size_t>(b) * p.M;
  const float* const i = p.i + static_cast<size_t>(b) * p.M;
  // the key set's loads and the first strips' are under way together
  float gv[4], iv[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int j = tid + e * kSelThreads;
    gv[e] = j < M ? g[j] : 0.0f;
    iv[e] = j < M ? i[j] : 0.0f;
  }
  select_mark_keys(p, s, b, tid, kSelThreads, true);
#pragma unroll 1
  for (int j0 = tid; j0 < M; j0 += 4 * kSelThreads) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int j = j0 + e * kSelThreads, next = j + 4 * kSelThreads;
      if (j < M) {
        val[j] = __float_as_uint(gv[e]);
        val_i[j] = __float_as_uint(iv[e]);
      }
      gv[e] = next < M ? g[next] : 0.0f;
      iv[e] = next < M ? i[next] : 0.0f;
    }
  }
  __syncthreads();
  if (p.M <= kFewTokens) select_request<1, SelectSyncCta>(p, s, x, val, val_i, b, tid, true, nullptr, nullptr);
  else select_request<4, SelectSyncCta>(p, s, x, val, val_i, b, tid, true, nullptr, nullptr);
  MD_PIPE(p.workspace, 1, true, false);
}

}  // namespace

cudaError_t launch_select(const mustdrop_plan& plan, const float* g, const float* i, const int32_t* key_idx,
                          const int32_t* key_cnt, int32_t* kept_idx, int32_t* kept_cnt, float* s_out,
                          void* workspace, cudaStream_t stream, const LayerArgs& la) {
  const Resolved& r = plan.r;
  SelectParams p;
  p.g = g; p.i = i; p.key_idx = key_idx; p.key_cnt = key_cnt; p.kept_idx = kept_idx; p.kept_cnt = kept_cnt;
  p.s_out = s_out; p.workspace = workspace;
  p.M = r.M; p.key_max = r.key_max; p.mode = r.mode; p.criteria = r.criteria; p.budget = r.budget; p.cap = r.cap;
  p.gamma = r.gamma; p.alpha = r.alpha;
  p.vis_cnt = la.vis_cnt; p.orig_in = la.orig_in; p.orig_out = la.orig_out;
  p.key_idx_out = la.key_idx_out; p.key_cnt_out = la.key_cnt_out;
  p.vis_start = r.vis_start; p.N = r.N; p.gamma_default = r.gamma_default; p.alpha_default = r.alpha_default;
  static_assert(sizeof(SelectShared) + sizeof(SelectScratch) + 8 * select_pad(kMaxVis) <= 48 * 1024, "no opt-in needed");
  return launch_pdl(select_kernel, dim3(r.B), dim3(kSelThreads), static_cast<size_t>(8) * select_pad(r.M), stream, p);
}

}  // namespace mustdrop
