// The fused BF16 kernel for launches too small to fill its tiles (soft
// visibility): 32 or 64 samples per 128-row tile, each by four or two replica
// rows that share its serial chain (REP in render_bf16_kernel.cuh).  Such a
// launch is one chain of evaluations long: 256 points x 32 directions took
// 40.9 us with 32 valid rows per tile, 20.5 us with four replicas.  Adding the
// directions' terms in their order in replica 0 (for the bits of a full tile)
// instead of the replicas' partial sums costs nothing there (cold, 34.0 us both)
// and up to 7 % elsewhere: 256 x 64 under 8 lights 45.0 -> 47.2 us, 256 x 32
// with 64 secondary directions 41.1 -> 43.8 us.  One light's terms added a step
// later, behind the next round trip's barrier: 34.4 us, left out.
#include "render_bf16_kernel.cuh"

namespace rtk {

// Two warpgroups per CTA, so that few warpgroups still spread over many SMs.
constexpr int kSmallWG = 2;

cudaError_t prepare_render_bf16_small() {
  const cudaError_t e = prepare_wg<kSmallWG, false, false, 2>();
  return e != cudaSuccess ? e : prepare_wg<kSmallWG, false, false, 4>();
}

// Replicas per sample.  Warpgroups own whole pixels, two or four of them per
// resident CTA; with one warpgroup per pixel (or the pixels dealt out over all
// of them) each has `rows` samples.  Up to 64 leave half of a 128-row tile
// idle, up to 32 three quarters.
int small_replicas(int P, int N, int num_sms) {
  const long long workers = 4LL * num_sms;
  const long long rows = ((long long)P + workers - 1) / workers * N;
  return rows <= 32 ? 4 : rows <= 64 ? 2 : 1;
}

cudaError_t launch_render_bf16_small(int rep, int nl, const ModelDesc& m, const HeadParams& hp, const rt_gbuffer& gb,
                                     int P, long long offset, const float4* envs, float4* out, int num_sms,
                                     cudaStream_t s) {
  return rep == 4 ? launch_lights<kSmallWG, false, false, 4>(nl, m, hp, gb, P, offset, envs, out, num_sms, s)
                  : launch_lights<kSmallWG, false, false, 2>(nl, m, hp, gb, P, offset, envs, out, num_sms, s);
}

}  // namespace rtk
