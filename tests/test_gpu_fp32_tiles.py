"""The FP32 kernels where their tiles can go wrong: rows that fill no tile, tiles of many points, several work units.

Tolerances are those the same quantities have elsewhere (test_gpu_render, test_gpu_stages, test_gpu_distill,
test_gpu_denoise); the sizes put the edges of the 128-row tiles, of the per-pixel slots and of the direction units
inside the data.
"""
import numpy as np
import pytest
import torch

import scenegen
from oracle import denoise as oden
from oracle import mlp
from oracle import render as orender
from tests import helpers, test_gpu_denoise, test_gpu_distill

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2409_10327_gb300 import build
    build.build()
    from paper_2409_10327_gb300 import binding
    return binding


# 1 .. 14: more pixels in a tile than shared feature slots; 15: as many, or one more, by where the tile starts; 16, 33,
# 130: fewer, with pixels that start and end anywhere in a tile or span several
@pytest.mark.parametrize("n_dirs, P", [(1, 300), (2, 131), (3, 700), (4, 129), (14, 40), (15, 61), (16, 33), (33, 11),
                                       (130, 5)])
def test_frame_tiles(lib, n_dirs, P):
    cfg = helpers.small_cfg(n_dirs=n_dirs, m_dirs=3)
    sc, gb = helpers.scene_arrays(cfg, 4, bias=0.2, n_pixels=P)
    r = helpers.renderer_for(cfg, sc)
    out = r.render_frame(helpers.to_cuda(gb), pixel_offset=17).cpu().numpy()
    assert r.check() == 0
    prm, opt = helpers.oracle_params(sc), helpers.oracle_options(cfg)
    ref = orender.render(gb, prm, opt, pixel_offset=17)
    sens = orender.float32_sensitivity(gb, prm, opt, pixel_offset=17, draws=4)
    ok, stats = helpers.fp32_parity(out[:, :3], ref, sens)
    assert ok, stats


# rows = 1, 127, 128, 129 and one tile over the number of warpgroups; K = 1 and 3: more points in a tile than slots
@pytest.mark.parametrize("P, K", [(1, 1), (127, 1), (43, 3), (32, 4), (129, 1), (7, 17), (2600, 15)])
def test_mlp_rows(lib, P, K):
    cfg = helpers.small_cfg(levels=5)
    sc = scenegen.make_scene(cfg, 6, bias_scale=0.3)
    r = helpers.renderer_for(cfg, sc)
    rng = np.random.default_rng(P + K)
    feat = rng.normal(0, 0.2, (P, 10)).astype(np.float32)
    d = rng.normal(size=(P, K, 3))
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    dirs = np.zeros((P, K, 4), np.float32)
    dirs[..., :3] = d
    f = torch.from_numpy(feat).cuda()
    vis, depth = r.trace(f, torch.from_numpy(dirs).cuda())
    out = r.decode(f).cpu().numpy()
    f64 = torch.from_numpy(np.repeat(feat.astype(np.float64), K, axis=0))
    v_ref, t_ref = mlp.implicit_ray_tracer(f64, torch.from_numpy(dirs[..., :3].reshape(-1, 3).astype(np.float64)),
                                           mlp.as_layers(sc.irt), cfg.near, cfg.far)
    np.testing.assert_allclose(vis.cpu().numpy().ravel(), v_ref.numpy(), atol=3e-6)
    np.testing.assert_allclose(depth.cpu().numpy().ravel(), t_ref.numpy(), atol=3e-6)
    a, rr, n = mlp.brdf_decoder(torch.from_numpy(feat.astype(np.float64)), mlp.as_layers(sc.brdf))
    np.testing.assert_allclose(out[:, 0:3], n.numpy(), atol=2e-6)
    np.testing.assert_allclose(out[:, 3:6], a.numpy(), atol=2e-6)
    np.testing.assert_allclose(out[:, 6], rr.numpy(), atol=2e-6)
    assert np.all(out[:, 7] == 0) and r.check() == 0


# K = 1: points without a front-facing direction; K = 289, 576: two and three direction units, ragged
@pytest.mark.parametrize("P, K", [(50, 1), (5, 289), (2, 576)])
def test_distill_units(lib, P, K):
    test_gpu_distill.test_distill_gradient_matches_oracle(lib, P, K)


# images with and without blocks whose window lies inside, and every exponent's route
@pytest.mark.parametrize("h, w, iters, sigma_n", [(26, 70, 2, 128.0), (17, 130, 1, 0.0), (40, 66, 1, 1.0), (33, 97, 2, 300.0)])
def test_denoise_blocks(lib, h, w, iters, sigma_n):
    c, z, n = test_gpu_denoise._image(h, w, h + w)
    got = test_gpu_denoise._run(lib, c, z, n, iterations=iters, sigma_n=sigma_n)
    ref_c, ref_v = oden.svgf(c, z, n, iterations=iters, sigma_n=sigma_n)
    test_gpu_denoise._check(got, ref_c, ref_v)


# 16-byte accesses where every buffer allows them, 4-byte ones otherwise; sizes off four
@pytest.mark.parametrize("n", [1, 3, 4, 1003, 300001])
@pytest.mark.parametrize("shift", [0, 1])
def test_adam_alignment(lib, n, shift):
    g = torch.Generator(device="cuda").manual_seed(n)
    base = [torch.rand(n + 1, generator=g, device="cuda") for _ in range(4)]
    one = [b[:n].clone() for b in base]                       # aligned
    two = [torch.cat([b.new_zeros(shift), b[:n]])[shift:] for b in base]
    lib.adam_step(*one, step=3, lr=0.01, weight_decay=1e-2)
    lib.adam_step(*two, step=3, lr=0.01, weight_decay=1e-2)
    for a, b in zip(one, two):
        assert torch.equal(a, b)
    # the update from its definition, in 64 bits; each of the few operations rounds once
    p, d, m, v = (b[:n].double() for b in base)
    d = d + 1e-2 * p
    m, v = 0.9 * m + 0.1 * d, 0.999 * v + 0.001 * d * d
    p = p - 0.01 * (m / (1 - 0.9 ** 3)) / ((v / (1 - 0.999 ** 3)).sqrt() + 1e-8)
    torch.testing.assert_close(one[0].double(), p, rtol=1e-5, atol=1e-6)


# features go out as pairs where the buffer allows 8-byte stores
def test_encode_alignment(lib):
    cfg = helpers.small_cfg(levels=5)
    r = helpers.renderer_for(cfg, scenegen.make_scene(cfg, 0))
    pos = torch.rand(77, 4, device="cuda") * 2.4 - 1.2
    want = r.encode(pos)
    buf = torch.full((77 * 10 + 1,), float("nan"), device="cuda")
    assert lib.LIB.rt_encode(r.ctx, lib._ptr(pos), 77, lib._ptr(buf[1:]), None, None, None) == lib.RT_OK
    torch.cuda.synchronize()
    assert torch.equal(buf[1:].view(77, 10), want)


# the distillation's targets are rt_trace's values at the front-facing directions (within the rounding both are allowed
# above), and zero visibility at the near depth elsewhere; one and several direction units, a point without any
@pytest.mark.parametrize("P, K", [(1, 1), (7, 31), (3, 256), (2, 700)])
def test_distill_targets(lib, P, K):
    cfg = helpers.small_cfg(levels=5)
    r = helpers.renderer_for(cfg, scenegen.make_scene(cfg, 6, bias_scale=0.3))
    rng = np.random.default_rng(P + K)
    unit = lambda a: a / np.linalg.norm(a, axis=-1, keepdims=True)
    plane = lambda a: torch.from_numpy(np.concatenate([a, np.zeros(a.shape[:-1] + (1,))], -1).astype(np.float32)).cuda()
    feat = torch.from_numpy(rng.normal(0, 0.2, (P, 10)).astype(np.float32)).cuda()
    d, n = unit(rng.normal(size=(P, K, 3))), unit(rng.normal(size=(P, 3)))
    d[0] = unit(d[0] - 3.0 * n[0])                           # all behind point 0
    dirs, normal = plane(d), plane(n)
    vis, depth = r.distill_targets(feat, dirs, normal)
    tv, td = r.trace(feat, dirs)
    front = (dirs[..., :3].double() * normal[:, None, :3].double()).sum(-1) > 0
    assert not front[0].any()
    assert (vis[~front] == 0).all() and (depth[~front] == cfg.near).all()
    torch.testing.assert_close(vis[front], tv[front], rtol=0, atol=6e-6)
    torch.testing.assert_close(depth[front], td[front], rtol=0, atol=6e-6)


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


# Two warpgroups per SM share the points, so tiles of several pixels need frames sized from the chip: 41 pixels per
# warpgroup below 16 directions (more in a tile than shared feature slots; at 14 and 15 some tiles have more and some
# have not, by where they start), 6 above (pixels that start and end anywhere in a tile, or span several).  Against the
# oracle on rows of the first, a middle and the last warpgroup, and bit for bit in shards, whose tiles fall elsewhere
@pytest.mark.parametrize("n_dirs, per", [(1, 40), (3, 40), (7, 40), (14, 40), (15, 40), (16, 40), (33, 5), (40, 5),
                                         (130, 5)])
def test_frame_tiles_of_several_pixels(lib, n_dirs, per):
    P = 2 * _sms() * per + 7
    cfg = helpers.small_cfg(n_dirs=n_dirs, m_dirs=2)
    sc, gb = helpers.scene_arrays(cfg, 4, bias=0.2, n_pixels=P)
    r = helpers.renderer_for(cfg, sc)
    dgb = helpers.to_cuda(gb)
    out = r.render_frame(dgb, pixel_offset=17).cpu().numpy()
    lo = 0
    for hi in (1, P // 3, P // 3 + 2 * _sms() + 1, P):
        part = {k: v[lo:hi].contiguous() for k, v in dgb.items()}
        np.testing.assert_array_equal(r.render_frame(part, pixel_offset=17 + lo).cpu().numpy(), out[lo:hi])
        lo = hi
    assert r.check() == 0
    rows = np.r_[0:per + 2, P // 2:P // 2 + per, P - per - 2:P]
    prm, opt = helpers.oracle_params(sc), helpers.oracle_options(cfg)
    ref = orender.render(gb, prm, opt, pixel_offset=17, rows=rows)
    sens = orender.float32_sensitivity(gb, prm, opt, pixel_offset=17, rows=rows, draws=4)
    ok, stats = helpers.fp32_parity(out[rows, :3], ref, sens)
    assert ok, stats


# three warpgroups per SM: a second and a third tile for some of them, the next tile made while a layer of this one runs;
# one point's directions (K = 500), tiles of few points, and more points in a tile than slots (K = 1, 3)
@pytest.mark.parametrize("K, tiles", [(1, 1.01), (3, 2.3), (16, 1.5), (500, 1.01)])
def test_mlp_rows_second_tiles(lib, K, tiles):
    test_mlp_rows(lib, int(3 * _sms() * 128 * tiles) // K + 5, K)


def test_decode_second_tiles(lib):
    test_mlp_rows(lib, 2 * 3 * _sms() * 128 + 130, 1)
