"""BF16 launches too small to fill 128-row tiles share a sample over replica rows: the same frame as in one large launch.

A row computes the same values either way; for a count of directions that is no multiple of 32 the grouping of the sum
over them differs.  All terms are non-negative, so each sum is within its term count times 2^-23 of the other.
"""
import numpy as np
import pytest
import torch

from tests import helpers

pytestmark = pytest.mark.gpu


# 4, 20, 32: four replicas (many pixels in a tile, a ragged tile, a full one); 33, 50, 64: two; M below, off and at a
# multiple of the replicas; one light and several
@pytest.mark.parametrize("n_dirs, m_dirs, sizes, lights", [(4, 8, (1, 9, 600), 1), (20, 3, (7, 608), 1), (32, 8, (256,), 3),
                                                           (32, 1, (33,), 1), (33, 5, (50,), 1), (64, 8, (2, 301), 2),
                                                           (50, 7, (607,), 1)])
def test_small_launch_equals_large(n_dirs, m_dirs, sizes, lights):
    # more than 64 samples for each of the chip's warpgroups: full tiles
    P = 4 * torch.cuda.get_device_properties(0).multi_processor_count * -(-72 // n_dirs)
    cfg = helpers.small_cfg(n_dirs=n_dirs, m_dirs=m_dirs, levels=14, max_res=512, precision="bf16")
    sc, gb = helpers.scene_arrays(cfg, 3, bias=0.2, n_pixels=P)
    r = helpers.renderer_for(cfg, sc)
    dgb = helpers.to_cuda(gb)
    envs = torch.from_numpy(np.stack([np.roll(sc.env, 3 * e, axis=1) for e in range(lights)])).cuda()
    whole = r.render_frame_multi(dgb, envs).cpu().numpy()
    lo = 0
    for n in sizes:
        part = {k: v[lo:lo + n].contiguous() for k, v in dgb.items()}
        got = r.render_frame_multi(part, envs, pixel_offset=lo).cpu().numpy()
        np.testing.assert_allclose(got, whole[:, lo:lo + n], rtol=(n_dirs + m_dirs) * 2.0 ** -23, atol=0)
        lo += n
    assert r.check() == 0


# a frame above the small-launch rule against shards on both sides of it, one of them by two replicas at 32 directions:
# with a multiple of 32 directions the pixel sums group alike too, so every bit is the frame's
@pytest.mark.parametrize("n_dirs, m_dirs, lights, kw", [(32, 8, 1, {}), (32, 5, 8, {}), (32, 1, 3, {}), (64, 8, 2, {}),
                                                        (64, 3, 1, {"sampling": 1}), (32, 6, 5, {"force_vis2": 0.25})])
def test_shards_have_the_frames_bits(n_dirs, m_dirs, lights, kw):
    workers = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    per = -(-72 // n_dirs)                       # pixels per warpgroup that make more than 64 samples
    P = 2 * workers * per + 11
    cfg = helpers.small_cfg(n_dirs=n_dirs, m_dirs=m_dirs, precision="bf16")
    sc, gb = helpers.scene_arrays(cfg, 7, bias=0.2, n_pixels=P)
    r = helpers.renderer_for(cfg, sc, **kw)
    dgb = helpers.to_cuda(gb)
    envs = torch.from_numpy(np.stack([np.roll(sc.env, 3 * e, axis=1) for e in range(lights)])).cuda()
    whole = r.render_frame_multi(dgb, envs, pixel_offset=3).cpu().numpy()
    cuts = [0, 1, 8, 8 + workers // 2, 8 + workers // 2 + (64 // n_dirs) * workers, P]
    assert cuts[-1] - cuts[-2] > workers * (per - 1)   # the last shard is above the rule, the others below
    for lo, hi in zip(cuts, cuts[1:]):
        part = {k: v[lo:hi].contiguous() for k, v in dgb.items()}
        got = r.render_frame_multi(part, envs, pixel_offset=3 + lo).cpu().numpy()
        np.testing.assert_array_equal(got, whole[:, lo:hi])
    assert r.check() == 0
