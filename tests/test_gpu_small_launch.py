"""BF16 launches too small to fill 128-row tiles share a sample over replica rows: the same frame as in one large launch.

A row computes the same values either way; only the order of the sums over the M secondary and the N primary
directions differs.  All terms are non-negative, so each sum is within its term count times 2^-23 of the other.
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
