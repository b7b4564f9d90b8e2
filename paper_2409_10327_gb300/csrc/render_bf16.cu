// The consecutive-sample and hard-visibility instantiations of the fused BF16
// kernel (render_bf16_kernel.cuh) and the light dispatch of rt_render_frame /
// rt_render_frame_multi on RT_BF16.
#include "render_bf16_kernel.cuh"

namespace rtk {

cudaError_t prepare_render_bf16() {
  cudaError_t e = prepare_wg<2, false, false>();
  e = e != cudaSuccess ? e : prepare_wg<3, false, false>();
  e = e != cudaSuccess ? e : prepare_wg<4, false, false>();
  e = e != cudaSuccess ? e : prepare_wg<4, true, false>();
  e = e != cudaSuccess ? e : prepare_render_bf16_chunked();
  e = e != cudaSuccess ? e : prepare_render_bf16_small();
  return e;
}

// E lights in launches of up to `max_nl` (1, 2, 4 or 8) lights each; light e
// reads envs + e * env_h * env_w and writes out + e * P.  Every launch
// recomputes the geometry, so fewer, wider launches share more work.  Hard
// visibility always runs 4 warpgroups per CTA.
cudaError_t launch_render_bf16_lights(const ModelDesc& m, const HeadParams& hp, const rt_gbuffer& gb, int P,
                                      long long offset, const float4* envs, int E, float4* out, int num_sms,
                                      int max_nl, int wg, cudaStream_t s) {
  const long long hw = (long long)m.env_h * m.env_w;
  for (int e0 = 0; e0 < E;) {
    int nl = 1;
    while (nl * 2 <= max_nl && nl * 2 <= E - e0) nl *= 2;
    ModelDesc mm = m;
    mm.env = envs + e0 * hw;
    const float4* ee = envs + e0 * hw;
    float4* oo = out + (long long)e0 * P;
    const bool chunk = !m.hard && (m.dpt == 32 || m.dpt == 64) && m.N % m.dpt == 0 && m.N > m.dpt;
    const int rep = m.hard ? 1 : small_replicas(P, m.N, num_sms);
    const cudaError_t err =
        rep > 1     ? launch_render_bf16_small(rep, nl, mm, hp, gb, P, offset, ee, oo, num_sms, s)
        : chunk       ? launch_render_bf16_chunked(nl, wg, mm, hp, gb, P, offset, ee, oo, num_sms, s)
        : m.hard    ? launch_lights<4, true, false>(nl, mm, hp, gb, P, offset, ee, oo, num_sms, s)
        : wg == 2   ? launch_lights<2, false, false>(nl, mm, hp, gb, P, offset, ee, oo, num_sms, s)
        : wg == 3   ? launch_lights<3, false, false>(nl, mm, hp, gb, P, offset, ee, oo, num_sms, s)
                    : launch_lights<4, false, false>(nl, mm, hp, gb, P, offset, ee, oo, num_sms, s);
    if (err != cudaSuccess) return err;
    e0 += nl;
  }
  return cudaSuccess;
}

}  // namespace rtk
