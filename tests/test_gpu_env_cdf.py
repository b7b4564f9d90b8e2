"""The texel CDFs that rt_set_params builds, at map sizes around the edges of their kernels' loops (16-texel
blocks of the running sum, rows shorter and longer than a CTA, one row, one texel), through the MIS render
that inverts them, against the FP64 oracle."""
import dataclasses

import numpy as np
import pytest
import torch

import scenegen
from oracle import render as orender
from tests import helpers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,w", [(1, 1), (2, 15), (5, 16), (33, 47), (129, 3), (3, 1025)])
def test_mis_frame_over_map_sizes(h, w):
    from paper_2409_10327_gb300 import build
    build.build()
    cfg = dataclasses.replace(scenegen.CONFIGS["tiny64"], env_h=h, env_w=w)
    sc, gb = helpers.scene_arrays(cfg, 4, bias=0.1, n_pixels=96)
    r = helpers.renderer_for(cfg, sc, sampling=1)
    out = r.render_frame(helpers.to_cuda(gb)).cpu().numpy()
    torch.cuda.synchronize()
    prm = helpers.oracle_params(sc)
    opt = helpers.oracle_options(cfg, sampling="mis")
    ref, allow = orender.render(gb, prm, dataclasses.replace(opt, mis_margin=helpers.MIS_MARGIN))
    sens = orender.float32_sensitivity(gb, prm, opt, draws=4)
    ok, stats = helpers.fp32_parity(out[:, :3], ref, sens, extra=allow)
    assert np.isfinite(out).all() and ok, stats


# a context made while the default stream is busy, in memory that another context (of another map height) has used, and
# bound several times on a stream that does not wait for the default one: the marginal CDF is complete every time
@pytest.mark.parametrize("h", [5, 300])
def test_mis_frame_of_a_context_made_on_a_busy_stream(h):
    cfg = dataclasses.replace(scenegen.CONFIGS["tiny64"], env_h=h, env_w=24)
    sc, gb = helpers.scene_arrays(cfg, 4, bias=0.1, n_pixels=64)
    dgb = helpers.to_cuda(gb)
    want = helpers.renderer_for(cfg, sc, sampling=1).render_frame(dgb).cpu().numpy()
    from paper_2409_10327_gb300 import binding
    model = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (sc.table, sc.brdf_blob, sc.irt_blob, sc.env)]
    other = torch.rand_like(model[3])
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for k in range(4):
        used = dataclasses.replace(cfg, env_h=h + 1 + k)
        helpers.renderer_for(used, scenegen.make_scene(used, k), sampling=1).close()
        torch.cuda._sleep(20_000_000)
        r = binding.Renderer(binding.make_config(cfg, sampling=1))
        with torch.cuda.stream(side):
            for env in [other] * k + [model[3]]:
                r.set_params(*model[:3], env)
            got = r.render_frame(dgb).cpu().numpy()
        assert r.check() == 0
        np.testing.assert_array_equal(got, want)
        r.close()
