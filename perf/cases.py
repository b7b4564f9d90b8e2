"""The work that users of the hash-grid renderer have it do, as measurable cases.

A case is one call (or one training step) through the package's public entry
points.  The inputs stand for a trained model on a visible surface: the surface
is a bumpy star-shaped body seen by a camera, so frames are coherent along
their rows and every point faces its viewer, and training batches are random
points of the same kind of surface.  Tables, weights and environment maps have
the distributions of the repository's own scene generator (uniform tables,
Xavier weights with the bias scale of its training benchmark, lognormal maps).

``exact`` restates the renderer from its definitions (include/rt.h) in 64-bit
torch, without the package's code.
"""
from __future__ import annotations

import math

import torch

from paper_2409_10327_gb300 import autograd, binding, distill

PI = math.pi
NEAR, FAR, F0 = 0.05, 1.5, 0.04
SEED = 0x5EED


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


# ---- the cases --------------------------------------------------------------

def _case(name, kind, **kw):
    base = {"name": name, "kind": kind, "width": 64, "height": 64, "n_dirs": 64, "m_dirs": 8, "levels": 16,
            "log2_T": 19, "max_res": 2048, "env_h": 64, "env_w": 128, "bf16": True, "hard": False, "mis": False}
    base.update(kw)
    return base


def listed():
    return [
        # one 16 x 16 tile of an interactive viewport, the paper's grid (14 levels, T = 2^17) and 32 directions:
        # launches and latency
        _case("tile_bf16", "frame", width=16, height=16, n_dirs=32, levels=14, log2_T=17),
        # the headline frame: 800 x 800, 128 directions, the tensor-core path
        _case("frame_bf16", "frame", width=800, height=800, n_dirs=128),
        # the paper's inference: MIS directions, the hard hit test, 64 directions, its grid; a ragged window
        _case("inference_bf16", "frame", width=601, height=399, levels=14, log2_T=17, hard=True, mis=True),
        # serving: one view lit by several environment maps on one geometry pass, the serving table
        _case("relight_bf16", "multi", width=480, height=270, log2_T=20, lights=8),
        # interactive relighting: bind a new, larger map, then a small MIS preview under it
        _case("bind_preview_bf16", "bind", width=160, height=90, n_dirs=16, env_h=256, env_w=512, mis=True),
        # the full-precision frame
        _case("frame_fp32", "frame", width=800, height=800, n_dirs=128, bf16=False),
        # a full-precision crop of odd size, a direction count that fills no tile, MIS
        _case("crop_fp32", "frame", width=97, height=61, n_dirs=40, levels=12, log2_T=16, bf16=False, mis=True),
        # one step of radiance training on the tensor cores: forward, loss gradient, adjoint
        _case("train_bf16", "train", width=65536, height=1),
        # the same in full precision through torch.autograd (rebinding the parameters as training does)
        _case("train_fp32", "train", width=16384, height=1, bf16=False),
        # one online distillation step, 2,048 points x 1,024 stratified directions, Adam in mid-training
        _case("distill_step", "distill", width=2048, height=1, n_dirs=1024, bf16=False),
        # the model's heads at given points (the stage calls: encode, decode, trace): data for a teacher or a viewer
        _case("heads_fp32", "heads", width=100003, height=1, n_dirs=16, bf16=False),
        # the spatial denoiser on the headline frame's size, the default five passes
        _case("denoise", "denoise", width=800, height=800, passes=5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame_bf16", "frame_bf16", "frame_fp32", "frame_fp32", "multi", "bind", "train_bf16",
                       "train_fp32", "distill", "heads", "denoise"])
    levels = rng.choice([8, 12, 14, 16, 16])
    grid = {"levels": levels, "log2_T": rng.choice([14, 17, 19]), "max_res": 2048 if levels >= 12 else 256,
            "m_dirs": rng.choice([4, 8, 8, 8])}
    small_env = rng.choice([(64, 128), (64, 128), (32, 64), (100, 200)])
    env = {"env_h": small_env[0], "env_w": small_env[1]}
    if kind in ("frame_bf16", "frame_fp32"):
        n = rng.choice([16, 32, 64, 128, rng.randint(8, 130)])
        w = _log(rng, 8, 500)
        h = max(1, min(_log(rng, 8, 500), (12_000_000 if kind == "frame_bf16" else 6_000_000) // (n * w)))
        return dict(_case("", "frame", width=w, height=h, n_dirs=n, bf16=kind == "frame_bf16",
                          mis=rng.random() < 0.4, hard=kind == "frame_bf16" and rng.random() < 0.35, **grid, **env))
    if kind == "multi":
        n = rng.choice([32, 64, 96])
        w = _log(rng, 16, 320)
        h = max(1, min(_log(rng, 16, 180), 3_000_000 // (n * w)))
        return dict(_case("", "multi", width=w, height=h, n_dirs=n, lights=rng.randint(2, 9), **grid, **env))
    if kind == "bind":
        eh = _log(rng, 32, 512)
        return dict(_case("", "bind", width=_log(rng, 16, 320), height=_log(rng, 9, 180), n_dirs=rng.choice([8, 16, 32]),
                          env_h=eh, env_w=2 * eh + rng.randint(0, 1), mis=True, **grid))
    if kind in ("train_bf16", "train_fp32"):
        n = rng.choice([16, 32, 64, rng.randint(8, 96)])
        p = max(1, min(_log(rng, 256, 65536), (3_000_000 if kind == "train_bf16" else 700_000) // n))
        return dict(_case("", "train", width=p, height=1, n_dirs=n, bf16=kind == "train_bf16",
                          mis=rng.random() < 0.3, **grid, **env))
    if kind == "distill":
        s = rng.choice([8, 12, 16, 32])
        return dict(_case("", "distill", width=_log(rng, 128, 3000), height=1, n_dirs=s * s, bf16=False, **grid, **env))
    if kind == "heads":
        k = rng.choice([1, 8, 16, rng.randint(2, 70)])
        return dict(_case("", "heads", width=min(_log(rng, 500, 200000), 3_000_000 // k), height=1, n_dirs=k, bf16=False,
                          **grid, **env))
    return dict(_case("", "denoise", width=_log(rng, 48, 1280), height=_log(rng, 48, 720), passes=rng.choice([3, 4, 5, 5])))


# ---- inputs -----------------------------------------------------------------

def _gen(seed, stream):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed) * 64 + stream)
    return g


def _uniform(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device=_dev()) * (hi - lo) + lo


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=_dev())


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _plane(v):
    out = torch.zeros(v.shape[0], 4, device=v.device)
    out[:, : v.shape[1]] = v
    return out


def _surface(case, seed):
    """Primary surface points: four float32 [P, 4] planes and the camera depth.  Frames take the pixels of a
    width x height window in row order, batches (height 1) random points of the surface."""
    g = _gen(seed, 1)
    W, H = case["width"], case["height"]
    if H > 1:
        v, u = torch.meshgrid((torch.arange(H, device=_dev()) + 0.5) / H * 2 - 1,
                              (torch.arange(W, device=_dev()) + 0.5) / W * 2 - 1, indexing="ij")
        u, v = u.reshape(-1), v.reshape(-1)
    else:
        u, v = _uniform(g, -1, 1, W), _uniform(g, -1, 1, W)
    # the square window onto the front hemisphere of directions, then the body's radius and its bumps
    rho = torch.maximum(u.abs(), v.abs()) * 0.97
    ang = torch.atan2(v, u)
    d = torch.stack([rho * torch.cos(ang), rho * torch.sin(ang), -torch.sqrt(1 - rho * rho)], -1)
    k = _normal(g, 3, 4) * 2.5
    ph = _uniform(g, 0, 2 * PI, 4)
    amp = torch.tensor([0.08, 0.05, 0.04, 0.03], device=_dev())
    wave = d @ k + ph
    r = 0.72 + (amp * torch.sin(wave)).sum(-1, keepdim=True)
    grad = (amp * torch.cos(wave)) @ k.t()
    tang = grad - (grad * d).sum(-1, keepdim=True) * d
    x = r * d
    n = _unit(d - tang / r)
    cam = torch.tensor([0.0, 0.0, -3.0], device=_dev())
    to = cam - x
    depth = to.norm(dim=-1)
    wo = to / depth[:, None]
    facing = (n * wo).sum(-1, keepdim=True)
    n = _unit(torch.where(facing < 0.1, n + (0.1 - facing) * wo, n))   # what the camera sees faces it
    k2 = _normal(g, 3, 4) * 3.0
    tex = torch.sin(x @ k2 + _uniform(g, 0, 2 * PI, 4))
    ar = 0.5 + 0.4 * tex + 0.05 * _normal(g, x.shape[0], 4)
    ar[:, :3].clamp_(0.02, 0.98)
    ar[:, 3].clamp_(0.09, 1.0)
    gb = {"pos": _plane(x), "normal": _plane(n), "view": _plane(wo), "albedo_rough": ar.contiguous()}
    return gb, depth.contiguous()


def _mlp(g, dims, last_bias=None):
    parts = []
    for a, b in zip(dims[:-1], dims[1:]):
        lim = math.sqrt(6.0 / (a + b))
        w, bias = _uniform(g, -lim, lim, b, a), _uniform(g, -0.1, 0.1, b)
        if b == dims[-1] and last_bias is not None:
            bias = bias + torch.tensor(last_bias, device=_dev())
        parts += [w.reshape(-1), bias]
    return torch.cat(parts)


def _model(case, seed):
    """(table, B, I, env): float32, the table's precision as the case has it.  B's outputs have the scale of a
    trained normal (about 1 along the mean direction); most of I's directions are unoccluded."""
    L, lf = case["levels"], 2 * case["levels"]
    table = _uniform(_gen(seed, 2), -0.1, 0.1, L, 1 << case["log2_T"], 2)
    brdf = _mlp(_gen(seed, 3), [lf, 64, 64, 7], [0.3, -0.2, -0.5, 0.0, 0.0, 0.0, 0.0])
    irt = _mlp(_gen(seed, 4), [lf + 27, 64, 64, 2], [0.2, -0.4])
    return (table.half() if case["bf16"] else table), brdf, irt, _env(case, seed, 1)[0]


def _env(case, seed, count):
    e = torch.zeros(count, case["env_h"], case["env_w"], 4, device=_dev())
    e[..., :3] = torch.exp(_normal(_gen(seed, 5), count, case["env_h"], case["env_w"], 3))
    return e


def _config(case):
    return binding.make_config(levels=case["levels"], log2_T=case["log2_T"], base_res=16, max_res=case["max_res"],
                               n_dirs=case["n_dirs"] if case["kind"] in ("frame", "multi", "bind", "train") else 64,
                               m_dirs=case["m_dirs"], env_h=case["env_h"], env_w=case["env_w"],
                               precision=binding.RT_BF16 if case["bf16"] else binding.RT_FP32,
                               visibility=binding.RT_VIS_HARD if case["hard"] else binding.RT_VIS_SOFT,
                               sampling=binding.RT_SAMPLE_MIS if case["mis"] else binding.RT_SAMPLE_COSINE)


def _renderer(case, model):
    r = binding.Renderer(_config(case))
    r.set_params(*model)
    return r


def _noisy_frame(case, seed):
    """A Monte Carlo frame of the surface: smooth shading times per-pixel noise."""
    gb, depth = _surface(case, seed)
    g = _gen(seed, 6)
    light = _unit(torch.tensor([0.4, 0.6, -0.7], device=_dev()))
    shade = 0.3 + (gb["normal"][:, :3] @ light).clamp_min(0)[:, None]
    rad = gb["albedo_rough"][:, :3] * shade * torch.exp(0.4 * _normal(g, depth.shape[0], 3))
    return _plane(rad), depth, gb["normal"]


def _moments(params, seed):
    """Adam's moments in mid-training."""
    g = _gen(seed, 7)
    m1 = [_normal(g, *p.shape) * 1e-5 for p in params]
    return m1, [(_uniform(g, 0.5, 2.0, *p.shape) * 1e-5) ** 2 for p in params]


ADAM_T = 1000


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "denoise":
        s["radiance"], s["depth"], s["normal"] = _noisy_frame(case, seed)
        return s
    s["gb"], _ = _surface(case, seed)
    s["model"] = _model(case, seed)
    s["r"] = _renderer(case, s["model"])
    if kind == "multi":
        s["envs"] = _env(case, seed, case["lights"])
    elif kind == "train":
        s["target"] = _target(case, seed)
        table, brdf, irt, _ = s["model"]
        if case["bf16"]:
            s["grads"] = [torch.zeros(t.shape, device=_dev()) for t in (table, brdf, irt)]
        else:
            s["leaves"] = [t.clone().requires_grad_(True) for t in (table, brdf, irt)]
    elif kind == "distill":
        s["teacher"] = _renderer(case, _model(case, seed + 1))
        s["d"] = distill.Distiller(s["r"], s["teacher"], *s["model"], K=case["n_dirs"])
        s["d"].m1, s["d"].m2 = _moments(s["d"].params, seed)
        s["d"].t = ADAM_T
    elif kind == "heads":
        g = _gen(seed, 8)
        s["dirs"] = _unit(_normal(g, case["width"], case["n_dirs"], 3))
        s["dirs"] = _plane(s["dirs"].reshape(-1, 3)).reshape(case["width"], case["n_dirs"], 4)
    return s


def _target(case, seed):
    return _uniform(_gen(seed, 9), 0.0, 2.0, case["width"] * case["height"], 3)


# ---- one pass ---------------------------------------------------------------

def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "denoise":
        return binding.denoise(s["radiance"], s["depth"], s["normal"], case["width"], case["height"],
                               iterations=case["passes"])
    r = s["r"]
    if kind == "frame":
        return r.render_frame(s["gb"])
    if kind == "multi":
        return r.render_frame_multi(s["gb"], s["envs"])
    if kind == "bind":
        r.set_params(*s["model"])
        return r.render_frame(s["gb"])
    if kind == "train":
        P = s["target"].shape[0]
        if not case["bf16"]:
            out = autograd.render(r, s["gb"], *s["leaves"], s["model"][3])
            loss = 0.5 * ((out - s["target"]) ** 2).mean()
            return [out.detach()] + list(torch.autograd.grad(loss, s["leaves"]))
        out = r.render_frame(s["gb"])
        d = torch.zeros_like(out)
        d[:, :3] = (out[:, :3] - s["target"]) / (3.0 * P)
        for g in s["grads"]:
            g.zero_()
        r.backward(s["gb"], d, *s["grads"])
        return [out[:, :3]] + s["grads"]
    if kind == "distill":
        loss = s["d"].step(s["gb"]["pos"], s["gb"]["normal"])
        return [loss] + s["d"].params + s["d"].grads
    feat = r.encode(s["gb"]["pos"])
    return [feat, r.decode(feat)] + list(r.trace(feat, s["dirs"]))


# ---- what a pass cannot do without ------------------------------------------

def _mlp_flops(case):
    lf = 2 * case["levels"]
    return 2 * ((lf + 27) * 64 + 4096 + 128), 2 * (lf * 64 + 4096 + 448)


def work(case):
    P, N, M, kind = case["width"] * case["height"], case["n_dirs"], case["m_dirs"], case["kind"]
    if kind == "denoise":
        # per pixel: radiance, depth and normal in, colour and variance out; the 7 x 7 moments and 25 taps per pass
        # of about 25 operations each
        return {"bytes": P * (16 + 4 + 16 + 16), "flops": P * 25 * (49 + 25 * case["passes"])}
    fi, fb = _mlp_flops(case)
    entry = 4 if case["bf16"] else 8
    lookups = P * (N + 1) if kind in ("frame", "multi", "bind", "train") else P
    table = min(case["levels"] * (entry << case["log2_T"]), lookups * case["levels"] * 8 * entry)
    env = 16 * case["env_h"] * case["env_w"]
    full = P * N * ((1 + M) * fi + fb)
    if kind in ("frame", "multi", "bind"):
        E = case.get("lights", 1)
        # hard visibility: the bounce is due only for shadowed directions, taken as a quarter
        flops = P * N * (fi + 0.25 * (M * fi + fb)) if case["hard"] else full
        return {"bytes": P * (64 + 16 * E) + table + env * E, "flops": flops}
    if kind == "train":
        grads = 4 * (case["levels"] * (2 << case["log2_T"]) + 2 * 10000)
        return {"bytes": P * (64 + 12 + 12) + table + env + grads, "flops": 4 * full}
    if kind == "distill":
        # teacher forward, student forward and adjoint; Adam reads 4 and writes 3 floats per parameter
        n = case["levels"] * (2 << case["log2_T"])
        return {"bytes": P * 32 + 2 * table + 4 * 8 * n, "flops": P * (N * 4 * fi + 4 * fb)}
    return {"bytes": P * (16 + 8 * case["levels"] + 32 + N * 24) + table, "flops": P * (N * fi + fb)}


# ---- the same in 64 bits ----------------------------------------------------

def _s64(x):
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >> 63 else x


def _shr(z, n):
    return (z >> n) & ((1 << (64 - n)) - 1)


def _splitmix(k, seed=SEED):
    z = k * _s64(0x9E3779B97F4A7C15) + _s64(seed)
    z = (z ^ _shr(z, 30)) * _s64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _s64(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _u12(ctr):
    return tuple(_shr(_splitmix(2 * ctr + j), 40).double() * 2.0 ** -24 for j in (1, 2))


def _sphere(u1, u2):
    rho = 2 * torch.sqrt((u1 * (1 - u1)).clamp_min(0))
    return torch.stack([rho * torch.cos(2 * PI * u2), rho * torch.sin(2 * PI * u2), 1 - 2 * u1], -1)


def _dot(a, b):
    return (a * b).sum(-1)


def _x_encode(case, table, x):
    L, T = case["levels"], 1 << case["log2_T"]
    b = math.exp((math.log(case["max_res"]) - math.log(16)) / max(L - 1, 1))
    u = (x * 0.5 + 0.5).clamp(0, 1)
    out = []
    for l in range(L):
        res = int(math.floor(16 * b ** l + 1e-9))
        g = u * res
        i0 = g.detach().floor().clamp_max(res - 1)
        w, i = g - i0, i0.long()
        f = 0
        for c in range(8):
            o = [(c >> a) & 1 for a in range(3)]
            j = [i[:, a] + o[a] for a in range(3)]
            if (res + 1) ** 3 <= T:
                row = j[0] + (res + 1) * (j[1] + (res + 1) * j[2])
            else:
                row = (j[0] ^ (j[1] * 2654435761) ^ (j[2] * 805459861)) & (T - 1)
            wt = 1
            for a in range(3):
                wt = wt * (w[:, a] if o[a] else 1 - w[:, a])
            f = f + wt[:, None] * table[l][row]
        out.append(f)
    return torch.cat(out, -1)


def _x_layers(blob, i, o):
    dims, at, out = [i, 64, 64, o], 0, []
    for a, b in zip(dims[:-1], dims[1:]):
        out.append((blob[at: at + a * b].reshape(b, a), blob[at + a * b: at + a * b + b]))
        at += a * b + b
    return out


def _x_mlp(layers, h):
    for k, (w, b) in enumerate(layers):
        h = h @ w.t() + b
        h = torch.relu(h) if k < 2 else h
    return h


def _x_trace(irt, f, w):
    pe = [w]
    for k in range(4):
        pe += [torch.sin(2 ** k * PI * w), torch.cos(2 ** k * PI * w)]
    z = _x_mlp(irt, torch.cat([f] + pe, -1))
    return z[..., 0], z[..., 1]


def _x_depth(z):
    return NEAR + (FAR - NEAR) * torch.nn.functional.softplus(z).clamp_max(1)


def _x_brdf(albedo, rough, n, wi, wo, with_d=False):
    a2 = rough ** 4
    nol, nov = _dot(n, wi).clamp_min(0), _dot(n, wo).clamp_min(1e-4)
    h = wi + wo
    hl = h.norm(dim=-1)
    h = h / hl.clamp_min(1e-10)[..., None]
    noh, voh = _dot(n, h), 0.5 * hl
    sin2 = torch.linalg.cross(n, h).square().sum(-1)
    dd = torch.where(noh > 0, sin2 + noh * noh * a2, torch.ones_like(noh))
    D = a2 / (PI * dd * dd)
    F = F0 + (1 - F0) * (1 - voh) ** 5
    vis = 0.5 / (nol * torch.sqrt(nov * nov * (1 - a2) + a2) + nov * torch.sqrt(nol * nol * (1 - a2) + a2))
    fr = albedo / PI + (D * F * vis)[..., None]
    return (fr, D, noh, voh) if with_d else fr


def _x_env_coords(env, w):
    H, W = env.shape[-3:-1]
    phi = torch.atan2(w[..., 1], w[..., 0])
    theta = torch.atan2(torch.sqrt(w[..., 0] ** 2 + w[..., 1] ** 2), w[..., 2])
    return (phi + PI) / (2 * PI) * W, theta / PI * H


def _x_env(env, w):
    H, W = env.shape[-3:-1]
    s, q = _x_env_coords(env, w)
    s, q = s - 0.5, q - 0.5
    s0, q0 = s.floor(), q.floor()
    fs, fq = (s - s0)[..., None], (q - q0)[..., None]
    c0 = s0.long() % W
    c1 = (c0 + 1) % W
    r0, r1 = q0.long().clamp(0, H - 1), (q0.long() + 1).clamp(0, H - 1)
    e = env[..., :3]
    return (1 - fq) * ((1 - fs) * e[r0, c0] + fs * e[r0, c1]) + fq * ((1 - fs) * e[r1, c0] + fs * e[r1, c1])


def _x_mis_tables(env):
    lum = (env[..., :3].double() @ torch.tensor([0.2126, 0.7152, 0.0722], dtype=torch.float64, device=env.device))
    p = lum.clamp_min(0) + 1e-6
    rows = p.sum(-1)
    return torch.cumsum(rows, 0) / rows.sum(), torch.cumsum(p, 1) / rows[:, None]


def _x_mis(case, tabs, n, wo, ar, i, u1, u2):
    """Primary MIS directions and their BRDF times the balance weight."""
    cm, cc = tabs
    H, W = cc.shape
    pm = torch.cat([torch.zeros_like(cm[:1]), cm])
    pc = torch.cat([torch.zeros_like(cc[:, :1]), cc], 1)
    r = torch.searchsorted(cm, u1.contiguous(), right=True).clamp_max(H - 1)
    ur = (u1 - pm[r]) / (pm[r + 1] - pm[r])
    # row by row inversion of the conditional CDFs: rows offset by their index are one increasing sequence
    flat = (cc + torch.arange(H, device=cc.device, dtype=cc.dtype)[:, None]).reshape(-1)
    c = (torch.searchsorted(flat, u2 + r, right=True) - r * W).clamp(0, W - 1)
    uc = (u2 - pc[r, c]) / (pc[r, c + 1] - pc[r, c])
    th, ph = PI * (r + ur) / H, 2 * PI * (c + uc) / W - PI
    light = torch.stack([torch.sin(th) * torch.cos(ph), torch.sin(th) * torch.sin(ph), torch.cos(th)], -1)
    # visible-normal GGX sampling (Heitz 2018) in the frame of Duff et al. 2017
    rough = ar[:, 3]
    alpha = rough ** 2
    sign = torch.where(n[:, 2] >= 0, 1.0, -1.0)
    a = -1 / (sign + n[:, 2])
    bb = n[:, 0] * n[:, 1] * a
    t = torch.stack([1 + sign * n[:, 0] ** 2 * a, sign * bb, -sign * n[:, 0]], -1)
    b = torch.stack([bb, sign + n[:, 1] ** 2 * a, -n[:, 1]], -1)
    vh = _unit(torch.stack([alpha * _dot(wo, t), alpha * _dot(wo, b), _dot(wo, n)], -1))
    inv = 1 / torch.sqrt(vh[:, 0] ** 2 + vh[:, 1] ** 2).clamp_min(1e-300)
    t1 = torch.stack([-vh[:, 1] * inv, vh[:, 0] * inv, torch.zeros_like(inv)], -1)
    t2 = torch.linalg.cross(vh, t1)
    p1, p2 = torch.sqrt(u1) * torch.cos(2 * PI * u2), torch.sqrt(u1) * torch.sin(2 * PI * u2)
    s = 0.5 * (1 + vh[:, 2])
    p2 = (1 - s) * torch.sqrt((1 - p1 * p1).clamp_min(0)) + s * p2
    nh = t1 * p1[:, None] + t2 * p2[:, None] + vh * torch.sqrt((1 - p1 * p1 - p2 * p2).clamp_min(0))[:, None]
    ne = _unit(torch.stack([alpha * nh[:, 0], alpha * nh[:, 1], nh[:, 2].clamp_min(0)], -1))
    h = t * ne[:, :1] + b * ne[:, 1:2] + n * ne[:, 2:]
    ggx = h * (2 * _dot(wo, h))[:, None] - wo
    seen = _dot(n, wo) > 1e-4
    w = torch.where(((i % 2 == 1) & seen)[:, None], ggx, light)
    # f_r (n . w)+ / (n_L p_L + n_G p_G) N / pi
    N = case["n_dirs"]
    fr, D, noh, voh = _x_brdf(ar[:, :3], rough, n, w, wo, with_d=True)
    sc, qc = _x_env_coords(torch.empty(H, W, 4), w)
    rr, c2 = qc.floor().long().clamp(0, H - 1), sc.floor().long().clamp(0, W - 1)
    pt = (pm[rr + 1] - pm[rr]) * (pc[rr, c2 + 1] - pc[rr, c2])
    pl = pt / ((2 * PI / W) * (PI / H) * torch.sqrt(w[:, 0] ** 2 + w[:, 1] ** 2))
    nov, a2 = _dot(n, wo), rough ** 4
    g1 = 2 * nov / (nov + torch.sqrt(a2 + (1 - a2) * nov * nov))
    ng = torch.where(seen, float(N // 2), 0.0)
    pg = torch.where(seen & (noh > 0) & (voh > 0), g1 * D / (4 * nov), torch.zeros_like(nov))
    pdf = (N - ng) * pl + ng * pg
    return w, fr * (_dot(n, w).clamp_min(0) / pdf * (N / PI))[:, None]


def _x_rows(case, m, gb, p):
    """Radiance [len(p), lights, 3] of the pixels p."""
    N, M = case["n_dirs"], case["m_dirs"]
    table, brdf, irt, envs, tabs = m
    pp, i = p.repeat_interleave(N), torch.arange(N, device=p.device).repeat(p.shape[0])
    x, n, wo = gb["pos"][pp, :3], _unit(gb["normal"][pp, :3]), _unit(gb["view"][pp, :3])
    ar = gb["albedo_rough"][pp]
    q = (pp * N + i) * (M + 1)
    u1, u2 = _u12(q)
    if case["mis"]:
        w, fr1 = _x_mis(case, tabs, n, wo, ar, i, u1, u2)
    else:
        w = _unit(n + _sphere(u1, u2))
        fr1 = _x_brdf(ar[:, :3], ar[:, 3], n, w, wo)
    f = _x_encode(case, table, gb["pos"][p, :3]).repeat_interleave(N, 0)
    z0, z1 = _x_trace(irt, f, w)
    v = torch.sigmoid(z0)
    f2 = _x_encode(case, table, x + w * _x_depth(z1)[:, None])
    y = _x_mlp(brdf, f2)
    n2, a2, r2 = _unit(y[:, :3]), torch.sigmoid(y[:, 3:6]), 0.09 + 0.91 * torch.sigmoid(y[:, 6])
    lo = [0.0] * len(envs)
    for j in range(M):
        wj = _unit(n2.detach() + _sphere(*_u12(q + 1 + j)))   # sampled directions are constants
        v2 = torch.sigmoid(_x_trace(irt, f2, wj)[0])
        c = v2[:, None] * _x_brdf(a2, r2, n2, wj, -w)
        lo = [s + c * _x_env(e, wj) for s, e in zip(lo, envs)]
    out = [((v[:, None] * _x_env(e, w) + (1 - v)[:, None] * s * (PI / M)) * fr1).reshape(-1, N, 3).sum(1) * (PI / N)
           for e, s in zip(envs, lo)]
    return torch.stack(out, 1)


def _x_model(case, model, envs):
    table, brdf, irt, env = model
    lf = 2 * case["levels"]
    t, b, r = table.double(), brdf.double(), irt.double()
    return (t, _x_layers(b, lf, 7), _x_layers(r, lf + 27, 2), [e.double() for e in envs],
            _x_mis_tables(env) if case["mis"] else None), (t, b, r)


def _chunks(n, rows):
    step = max(1, (1 << 16) // rows)
    return [torch.arange(a, min(n, a + step), device=_dev()) for a in range(0, n, step)]


def _x_frame(case, seed):
    gb = {k: v.double() for k, v in _surface(case, seed)[0].items()}
    model = _model(case, seed)
    envs = _env(case, seed, case["lights"]) if case["kind"] == "multi" else model[3][None]
    with torch.no_grad():
        m, _ = _x_model(case, model, envs)
        P = gb["pos"].shape[0]
        out = torch.zeros(len(envs), P, 4, dtype=torch.float64, device=_dev())
        for p in _chunks(P, case["n_dirs"]):
            out[:, p, :3] = _x_rows(case, m, gb, p).transpose(0, 1)
    return out if case["kind"] == "multi" else out[0]


def _x_train(case, seed):
    gb = {k: v.double() for k, v in _surface(case, seed)[0].items()}
    model = _model(case, seed)
    target = _target(case, seed).double()
    leaves = [t.double().requires_grad_(True) for t in model[:3]]
    m, _ = _x_model(case, leaves + [model[3]], model[3][None])
    P, outs = gb["pos"].shape[0], []
    for p in _chunks(P, case["n_dirs"]):
        table, brdf, irt = leaves
        lf = 2 * case["levels"]
        mm = (table, _x_layers(brdf, lf, 7), _x_layers(irt, lf + 27, 2), m[3], m[4])
        o = _x_rows(case, mm, gb, p)[:, 0]
        (0.5 * ((o - target[p]) ** 2).sum() / (3 * P)).backward()
        outs.append(o.detach())
    return [torch.cat(outs)] + [t.grad for t in leaves]


def _x_heads_of(case, m, feat, dirs):
    y = _x_mlp(m[1], feat)
    brdf = torch.cat([_unit(y[:, :3]), torch.sigmoid(y[:, 3:6]), 0.09 + 0.91 * torch.sigmoid(y[:, 6:7]),
                      torch.zeros_like(y[:, :1])], -1)
    z0, z1 = _x_trace(m[2], feat[:, None, :].expand(-1, dirs.shape[1], -1), dirs)
    return brdf, z0, z1


def _x_heads(case, seed):
    pos = _surface(case, seed)[0]["pos"].double()
    g = _gen(seed, 8)
    dirs = _unit(_normal(g, case["width"], case["n_dirs"], 3)).double()
    out = []
    with torch.no_grad():
        model = _model(case, seed)
        m, _ = _x_model(case, model, model[3][None])
        for p in _chunks(pos.shape[0], case["n_dirs"]):
            f = _x_encode(case, m[0], pos[p, :3])
            brdf, z0, z1 = _x_heads_of(case, m, f, dirs[p])
            out.append((f, brdf, torch.sigmoid(z0), _x_depth(z1)))
    return [torch.cat(v) for v in zip(*out)]


def _x_distill(case, seed):
    gb = {k: v.double() for k, v in _surface(case, seed)[0].items()}
    P, K = case["width"], case["n_dirs"]
    S = math.isqrt(K)
    model, teach = _model(case, seed), _model(case, seed + 1)
    leaves = [t.double().requires_grad_(True) for t in model[:3]]
    with torch.no_grad():
        tm, _ = _x_model(case, teach, teach[3][None])
    loss = torch.zeros(3, dtype=torch.float64, device=_dev())
    k = torch.arange(K, device=_dev())
    lf = 2 * case["levels"]
    for p in _chunks(P, K):
        sm = (leaves[0], _x_layers(leaves[1], lf, 7), _x_layers(leaves[2], lf + 27, 2))
        x1, x2 = _u12(p[:, None] * K + k)
        # the directions are float32 data that every head reads
        w = _sphere((k // S + x1) / S, (k % S + x2) / S)
        n = gb["normal"][p, :3]
        front = (_dot(w, n[:, None, :]) > 0).double()
        with torch.no_grad():
            bt, z0t, z1t = _x_heads_of(case, tm, _x_encode(case, tm[0], gb["pos"][p, :3]), w)
        bs, z0, z1 = _x_heads_of(case, sm, _x_encode(case, sm[0], gb["pos"][p, :3]), w)
        wt = front / front.sum(-1, keepdim=True).clamp_min(1) / P
        vt = (z0t > 0).double()
        bce = torch.nn.functional.binary_cross_entropy_with_logits(z0, vt, reduction="none")
        dl = (torch.nn.functional.softplus(z1).clamp_max(1) - torch.nn.functional.softplus(z1t).clamp_max(1)).abs()
        terms = torch.stack([(bs[:, :7] - bt[:, :7]).abs().sum() / (7 * P), (wt * bce).sum(), (wt * dl).sum()])
        terms.sum().backward()
        loss += terms.detach()
    grads = [t.grad for t in leaves]
    m1, m2 = _moments(model[:3], seed)
    params = []
    for t, g, a, b, wd in zip(leaves, grads, m1, m2, [0.0, 1e-6, 1e-6]):
        x = t.detach()
        gg = g + wd * x
        a, b = 0.9 * a.double() + 0.1 * gg, 0.999 * b.double() + 0.001 * gg * gg
        step = ADAM_T + 1
        params.append(x - 2e-3 * (a / (1 - 0.9 ** step)) / (torch.sqrt(b / (1 - 0.999 ** step)) + 1e-8))
    return [loss] + params + grads


def _shifted(img, dy, dx):
    """img at (y + dy, x + dx) and whether that lies inside."""
    H, W = img.shape[:2]
    y, x = torch.arange(H, device=img.device) + dy, torch.arange(W, device=img.device) + dx
    ok = ((y >= 0) & (y < H))[:, None] & ((x >= 0) & (x < W))[None, :]
    return img[y.clamp(0, H - 1)][:, x.clamp(0, W - 1)], ok.double()


def _x_denoise(case, seed):
    W, H = case["width"], case["height"]
    rad, z, n = _noisy_frame(case, seed)
    c, z, n = rad[:, :3].double().reshape(H, W, 3), z.double().reshape(H, W), n[:, :3].double().reshape(H, W, 3)
    lw = torch.tensor([0.2126, 0.7152, 0.0722], dtype=torch.float64, device=_dev())
    gx, gy = torch.zeros_like(z), torch.zeros_like(z)
    if W > 1:
        gx[:, :-1] = z[:, 1:] - z[:, :-1]
        gx[:, -1] = z[:, -1] - z[:, -2]
    if H > 1:
        gy[:-1] = z[1:] - z[:-1]
        gy[-1] = z[-1] - z[-2]

    def geom(dy, dx):
        zq, ok = _shifted(z, dy, dx)
        nq, _ = _shifted(n, dy, dx)
        return ok * torch.exp(-(z - zq).abs() / ((gx * dx + gy * dy).abs() + 1e-10)) * _dot(n, nq).clamp_min(0) ** 128

    s0 = s1 = s2 = 0
    for dy in range(-3, 4):
        for dx in range(-3, 4):
            w, l = geom(dy, dx), _shifted(c, dy, dx)[0] @ lw
            s0, s1, s2 = s0 + w, s1 + w * l, s2 + w * l * l
    var = (s2 / s0 - (s1 / s0) ** 2).clamp_min(0)
    h = [1 / 16, 1 / 4, 3 / 8, 1 / 4, 1 / 16]
    for it in range(case["passes"]):
        gs = gw = 0
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                v, ok = _shifted(var, dy, dx)
                k = (2 - abs(dx)) * (2 - abs(dy)) * ok
                gs, gw = gs + k * v, gw + k
        den, lum = 4.0 * torch.sqrt((gs / gw).clamp_min(0)) + 1e-10, c @ lw
        ws, ac, av = 0, 0, 0
        for dy in range(-2, 3):
            for dx in range(-2, 3):
                oy, ox = dy << it, dx << it
                cq, vq = _shifted(c, oy, ox)[0], _shifted(var, oy, ox)[0]
                w = h[dy + 2] * h[dx + 2] * geom(oy, ox) * torch.exp(-(lum - cq @ lw).abs() / den)
                ws, ac, av = ws + w, ac + w[..., None] * cq, av + w * w * vq
        c, var = ac / ws[..., None], av / ws ** 2
    return torch.cat([c, var[..., None]], -1).reshape(H * W, 4)


def exact(case, seed):
    kind, rows = case["kind"], case["width"] * case["height"] * case["n_dirs"]
    if kind == "denoise":
        return _x_denoise(case, seed)
    if kind == "heads":
        return _x_heads(case, seed)
    if kind == "distill":
        return _x_distill(case, seed)
    if case["hard"] or rows > 4_000_000:
        # the hit test decides an integer from floating point (bf16 logits); the largest frames take too long
        return None
    if kind == "train":
        if case["bf16"]:
            # the gradient's derivative of the finest levels jumps at cell faces, so bf16 points give another one
            return None
        return _x_train(case, seed) if rows <= 1_200_000 else None
    return _x_frame(case, seed)
