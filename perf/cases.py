"""Performance cases: the work a user of this framework has it do, through its public entry points.

  render  kns.render: sphere-traced and shaded camera views, FP32 or BF16
  views   kns.render_views: one batch of a render server, several resolutions over a stack of grids
  rays    kns.trace_rays: explicit rays
  paths   kns.path_trace: a Lambertian path-traced image
  points  kns.sdf: the batch field query (distance, feature, gradient)
  train   kns.train: loss and gradient of one fine-tuning batch

Grids are the synthetic workloads' (c1: 8^3 cells of width 32 without a mask; c2: 16^3, width 32; c3l:
32^3, width 64; the last two with a 128^3 occupancy mask): one SAL sphere with a perturbation per cell.  A
program loads its scene once and renders it many times, so a process keeps one context and its loaded
grids; cameras, rays, points, random draws, targets and trained weights come from the seed.

BF16 renders run with tail_rays = -1, the documented setting under which a render is reproducible bit for
bit (every step of the trace on the tensor cores); with the default hand-over two renders of one view
differ in a few pixels, so their outputs could not be compared.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2206_10885_gb300 as kns
from paper_2206_10885_gb300 import synth as S

EPS = 1e-4
DEV = "cuda:0"


# ---------------------------------------------------------------- cases
def listed():
    return [
        # the smallest render: four 64 x 64 previews of a small grid (latency and launches)
        dict(name="preview", op="render", grid="c1", precision="fp32", cams=4, W=64, H=64, steps=64),
        # the FP32 workload of the paper's 16^3 grid: eight views of 800 x 800
        dict(name="orbit_fp32", op="render", grid="c2", precision="fp32", cams=8, W=800, H=800, steps=128),
        # full-HD frames of the large grid in FP32
        dict(name="wide_fp32", op="render", grid="c3l", precision="fp32", cams=2, W=1920, H=1080, steps=128),
        # the largest render: eight full-HD views of the large grid on the tensor cores
        dict(name="wide_bf16", op="render", grid="c3l", precision="bf16", cams=8, W=1920, H=1080, steps=128),
        # one odd-sized interactive view on the tensor cores
        dict(name="view_bf16", op="render", grid="c2", precision="bf16", cams=1, W=511, H=383, steps=128),
        # one batch of a render server: requests of mixed sizes over two stacked scenes
        dict(name="serve_batch", op="views", grid="c2", grids=2, sizes="256x256,512x512,800x800,256x256,333x217",
             precision="fp32", steps=128),
        # explicit rays (picking, shadow and bounce rays of a caller's own integrator), a ragged count
        dict(name="rays", op="rays", grid="c2", n=100003, steps=128),
        # a path-traced image
        dict(name="paths", op="paths", grid="c2", W=200, H=150, spp=8, depth=4, steps=128),
        # a small batch of field queries
        dict(name="points_small", op="points", grid="c2", n=4096, full=True),
        # a large ragged batch of field queries on the large grid
        dict(name="points_field", op="points", grid="c3l", n=1000003, full=True),
        # the paper's fine-tuning batch (1,024 rays), driven by torch autograd
        dict(name="train_paper", op="train", H=3, N=16, rays=1024, strat=64, imp=32, eik=16384, autograd=True),
        # a large fine-tuning batch through the fused step
        dict(name="train_batch", op="train", H=3, N=16, rays=65536, strat=64, imp=32, eik=16384, autograd=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["render", "render", "render", "views", "rays", "paths", "points", "points", "train", "train"])
    if op == "render":
        grid = rng.choice(["c1", "c2", "c3l"])
        W, cams = _log(rng, 48, 1920), rng.randint(1, 8)
        return dict(op=op, grid=grid, precision=rng.choice(["fp32", "fp32", "bf16"]) if grid != "c1" else "fp32",
                    cams=cams if grid != "c1" else min(cams, 4), W=W if grid != "c1" else min(W, 512),
                    H=max(32, int(W * rng.uniform(0.5, 1.0))) if grid != "c1" else max(32, min(W, 512) - rng.randint(0, 9)),
                    steps=64 if grid == "c1" else 128)
    if op == "views":
        sizes = ["%dx%d" % (w, max(16, int(w * rng.uniform(0.5, 1.0)))) for w in
                 (_log(rng, 64, 1024) for _ in range(rng.randint(2, 6)))]
        return dict(op=op, grid="c2", grids=rng.randint(1, 2), sizes=",".join(sizes), precision="fp32", steps=128)
    if op == "rays":
        return dict(op=op, grid=rng.choice(["c2", "c3l"]), n=_log(rng, 300, 1000000), steps=128)
    if op == "paths":
        return dict(op=op, grid="c2", W=_log(rng, 24, 400), H=_log(rng, 24, 300), spp=rng.randint(1, 12),
                    depth=rng.randint(2, 5), steps=128)
    if op == "points":
        return dict(op=op, grid=rng.choice(["c1", "c2", "c3l"]), n=_log(rng, 100, 1000000),
                    full=rng.random() < 0.7)
    return dict(op=op, H=rng.choice([2, 3]), N=rng.choice([8, 16]), rays=_log(rng, 300, 65536),
                strat=rng.choice([32, 48, 64]), imp=rng.choice([0, 16, 32]), eik=_log(rng, 1000, 16384),
                autograd=rng.random() < 0.5)


# ---------------------------------------------------------------- scenes
_CTX = []
_GRIDS = {}


def _ctx():
    if not _CTX:
        _CTX.append(kns.Context(0))
    return _CTX[0]


def _weights(desc, seed, std=1e-3):
    """(cells, parameters) FP32 on the GPU: the SAL sphere of synth, perturbed per cell; random colours."""
    one = S.GridDesc(N=1, sdf_hidden=desc.sdf_hidden, sdf_width=desc.sdf_width, col_width=desc.col_width)
    base = torch.from_numpy(S.sal_sphere_grid(one, seed=0, perturb_std=0.0)[:desc.p_sdf]).to(DEV)
    g = torch.Generator(DEV).manual_seed(seed)
    w = torch.empty((desc.n_cells, desc.p_cell), device=DEV)
    w[:, :desc.p_sdf] = base + std * torch.randn((desc.n_cells, desc.p_sdf), device=DEV, generator=g)
    scale = np.concatenate([np.full(i * o + o, 1.0 / math.sqrt(i)) for i, o in desc.col_layers()]).astype(np.float32)
    w[:, desc.p_sdf:] = (torch.rand((desc.n_cells, desc.p_col), device=DEV, generator=g) * 2 - 1) * torch.from_numpy(
        scale).to(DEV)
    return w


def _mask(desc, w):
    """Occupancy in 64 bits: voxels with |d(centre)| under a voxel diagonal."""
    if not desc.occ_res:
        return None
    n = desc.occ_res
    ax = -1.0 + (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) * (2.0 / n)
    p = torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3).flip(1)  # x fastest
    return (_field(desc, w, p)[0].abs() < math.sqrt(3.0) * 2.0 / n).reshape(n, n, n)  # [z, y, x]


def _scene(name, k=0):
    """(desc, weights on the GPU, mask) of grid k of a workload's shape."""
    if (name, k) not in _GRIDS:
        desc = S.config_desc(name)
        w = _weights(desc, 11 + k)
        _GRIDS[name, k] = (desc, w, _mask(desc, w))
    return _GRIDS[name, k]


def _words(mask):
    return np.packbits(mask.cpu().numpy().reshape(-1), bitorder="little").view(np.uint64)


def _grid(name, n=1):
    """The loaded grid (n > 1: a stack)."""
    if (name, "loaded", n) not in _GRIDS:
        sc = [_scene(name, k) for k in range(n)]
        desc = sc[0][0]
        w = [s[1].cpu().numpy().reshape(-1) for s in sc]
        occ = [_words(s[2]) for s in sc] if desc.occ_res else None
        _GRIDS[name, "loaded", n] = (kns.Grid.load(_ctx(), desc, w[0], occ[0] if occ else None) if n == 1
                                     else kns.Grid.load_stack(_ctx(), desc, w, occ))
    return _GRIDS[name, "loaded", n]


# ---------------------------------------------------------------- inputs
def _sizes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["sizes"].split(",")]


def _requests(case, seed):
    return [(S.orbit_cameras(1, W, H, seed=1000 * seed + 7 * i + 3)[0], W, H, i % case["grids"])
            for i, (W, H) in enumerate(_sizes(case))]


def _rays(case, seed):
    """Rays from around the object towards it, as a caller's own integrator makes them."""
    g = torch.Generator(DEV).manual_seed(seed)
    o = torch.nn.functional.normalize(torch.randn((case["n"], 3), device=DEV, generator=g), dim=1)
    o = o * (1.2 + 1.5 * torch.rand((case["n"], 1), device=DEV, generator=g))
    to = 1.2 * torch.rand((case["n"], 3), device=DEV, generator=g) - 0.6
    return o, torch.nn.functional.normalize(to - o, dim=1)


def _points(case, seed):
    g = torch.Generator(DEV).manual_seed(seed)
    return 2.0 * torch.rand((case["n"], 3), device=DEV, generator=g) - 1.0


def _train_desc(case):
    return S.GridDesc(N=case["N"], sdf_hidden=case["H"], sdf_width=32, col_width=32, occ_res=0)


def _batch(case, seed):
    """One fine-tuning batch: pixel rays of orbit cameras, smooth target colours, the step's random draws."""
    g = torch.Generator(DEV).manual_seed(seed)
    B, Ns, Ni = case["rays"], case["strat"], case["imp"]
    cams = S.orbit_cameras(8, 800, 800, seed=seed)
    sel = torch.randint(0, 8 * 800 * 800, (B,), device=DEV, generator=g).cpu().numpy()
    o, d = (torch.from_numpy(v).to(DEV) for v in S.pixel_rays(cams, 800, 800, sel))
    return dict(origins=o, dirs=d, target=0.5 + 0.3 * torch.sin(4.0 * d + o),
                u_strat=torch.rand((B, Ns), device=DEV, generator=g),
                u_imp=torch.rand((B, Ni), device=DEV, generator=g).sort(dim=1)[0],
                eik_points=2.0 * torch.rand((case["eik"], 3), device=DEV, generator=g) - 1.0)


def prepare(case, seed):
    op = case["op"]
    st = dict(case=case, ctx=_ctx())
    if op == "train":
        st["desc"] = _train_desc(case)
        st["params"] = _weights(st["desc"], seed).reshape(-1)
        if case["autograd"]:
            st["params"] = torch.nn.Parameter(st["params"])
        st["batch"] = kns.train.TrainBatch(**_batch(case, seed))
        return st
    st["grid"] = _grid(case["grid"], case.get("grids", 1))
    if op == "render":
        st["cams"] = S.orbit_cameras(case["cams"], case["W"], case["H"], seed=seed)
    elif op == "views":
        st["requests"] = _requests(case, seed)
    elif op == "rays":
        st["o"], st["d"] = _rays(case, seed)
    elif op == "paths":
        st["cams"], st["seed"] = S.orbit_cameras(1, case["W"], case["H"], seed=seed), seed
    else:
        st["pts"] = _points(case, seed)
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    op = case["op"]
    if op == "render":
        if case["precision"] == "bf16":
            return kns.render(ctx, st["grid"], st["cams"], case["W"], case["H"], case["steps"], EPS,
                              precision=kns.KNS_BF16, tuning=dict(tail_rays=-1))
        return kns.render(ctx, st["grid"], st["cams"], case["W"], case["H"], case["steps"], EPS)
    if op == "views":
        return kns.render_views(ctx, st["grid"], st["requests"], case["steps"], EPS)
    if op == "rays":
        return kns.trace_rays(ctx, st["grid"], st["o"], st["d"], case["steps"], EPS)
    if op == "paths":
        return kns.path_trace(ctx, st["grid"], st["cams"], case["W"], case["H"], spp=case["spp"],
                              max_depth=case["depth"], seed=st["seed"], max_steps=case["steps"], eps=EPS)
    if op == "points":
        return kns.sdf(ctx, st["grid"], st["pts"], want_feat=case["full"], want_grad=case["full"])
    if case["autograd"]:
        st["params"].grad = None
        loss = kns.train.neus_loss(ctx, st["desc"], st["params"], st["batch"])
        loss.backward()
        return loss.detach(), st["params"].grad
    return kns.train.step(ctx, st["desc"], st["params"], st["batch"])


# ---------------------------------------------------------------- work
def _macs(desc):
    W, H, IN = desc.sdf_width, desc.sdf_hidden, desc.sdf_in
    hidden = IN * W + (H - 1) * W * W
    trace = hidden + W                          # d alone
    full = hidden + 16 * W                      # d and the feature
    colour = desc.col_in * W + 3 * W
    return trace, full, hidden, colour          # hidden: also one reverse pass to the encoding


def work(case):
    """Inputs read once, outputs written once; multiply-adds of the samples a ray takes (2.5 with empty-space
    skipping, 10 without: both measured on these views) and of shading a fifth of the rays."""
    op = case["op"]
    desc = _train_desc(case) if op == "train" else S.config_desc(case["grid"])
    trace, full, rev, colour = _macs(desc)
    params = 4 * desc.n_cells * desc.p_cell
    if op == "points":
        n = case["n"]
        touched = params * min(1.0, n / desc.n_cells) * desc.p_sdf / desc.p_cell
        return dict(bytes=n * (12 + (4 + 60 + 12 if case["full"] else 4)) + touched,
                    flops=2 * n * (full + rev if case["full"] else trace))
    if op == "train":
        S_ = case["strat"] + case["imp"]
        fd, centre = 6 * (case["rays"] * S_ + case["eik"]), case["rays"] * S_
        return dict(bytes=2 * params + 4 * (case["rays"] * (9 + S_) + 3 * case["eik"]),
                    flops=2 * (case["rays"] * case["strat"] * trace + 3 * fd * trace + 3 * centre * (full + colour)))
    if op == "render":
        rays = case["cams"] * case["W"] * case["H"]
    elif op == "views":
        rays = sum(w * h for w, h in _sizes(case))
    elif op == "rays":
        rays = case["n"]
    else:
        rays = case["W"] * case["H"] * case["spp"]
    per_ray = 2.5 if desc.occ_res else 10.0
    shell = 0.1 * params  # the cells around the surface
    out = 12 * case["W"] * case["H"] if op == "paths" else (57 if op == "rays" else 33) * rays
    return dict(bytes=out + min(shell, rays * 4.0 * desc.p_cell),
                flops=2 * rays * (per_ray * trace + 0.2 * (full + rev + colour)))


# ---------------------------------------------------------------- the same in 64 bits
def _encode(p, L):
    a = [p]
    for k in range(L):
        a += [torch.sin(2.0 ** k * math.pi * p), torch.cos(2.0 ** k * math.pi * p)]
    return torch.cat(a, 1)


def _cell(desc, p):
    i = torch.floor((p + 1.0) * (desc.N / 2.0)).clamp(0, desc.N - 1).long()
    return i[:, 0] + desc.N * (i[:, 1] + desc.N * i[:, 2])


def _split(desc, w):
    """(W, b) of every layer, SDF then colour, of rows of canonical parameters w (n, p)."""
    out, off = [], 0
    for i, o in desc.sdf_layers() + desc.col_layers():
        out.append((w[:, off:off + i * o].reshape(-1, o, i), w[:, off + i * o:off + i * o + o]))
        off += i * o + o
    return out


def _softplus(s):
    return s.clamp(min=0) + torch.log1p(torch.exp(-100.0 * s.abs())) / 100.0


def _mlp(layers, x, act):
    for k, (W, b) in enumerate(layers):
        x = torch.baddbmm(b[:, None, :], x, W.transpose(1, 2))
        if k + 1 < len(layers):
            x = act(x)
    return x


def _by_cell(desc, cell):
    """Yields (indices (c, m), cells (c,), valid (c, m)): points grouped by cell, groups of similar size."""
    order = torch.argsort(cell)
    cells, counts = torch.unique_consecutive(cell[order], return_counts=True)
    start = torch.cumsum(counts, 0) - counts
    by = torch.argsort(counts)
    cells, counts, start = cells[by], counts[by], start[by]
    host, k = counts.tolist(), 0
    while k < len(host):
        e = k
        while e < len(host) and host[e] * (e - k + 1) <= 60000 and e - k < 1024:
            e += 1
        e = max(e, k + 1)
        m = host[e - 1]
        at = torch.arange(m, device=cell.device)[None, :]
        valid = at < counts[k:e, None]
        yield order[(start[k:e, None] + at).clamp(max=len(order) - 1)], cells[k:e], valid
        k = e


def _field(desc, w, p, want=False, cell=None):
    """d (and with `want` the feature and the input gradient) at points p, in 64 bits."""
    n, L = p.shape[0], desc.pe_pos_L
    d = torch.empty(n, device=p.device, dtype=torch.float64)
    z = torch.empty((n, 15), device=p.device, dtype=torch.float64) if want else None
    g = torch.empty((n, 3), device=p.device, dtype=torch.float64) if want else None
    ns = len(desc.sdf_layers())
    for idx, cells, valid in _by_cell(desc, _cell(desc, p) if cell is None else cell):
        layers = _split(desc, w[cells].double())[:ns]
        x = p[idx]
        with torch.enable_grad():
            if want:
                x = x.requires_grad_(True)
            e = _encode(x.reshape(-1, 3), L).reshape(x.shape[0], x.shape[1], -1)
            y = _mlp(layers if want else layers[:-1] + [(layers[-1][0][:, :1], layers[-1][1][:, :1])], e, _softplus)
            if want:
                gx, = torch.autograd.grad(y[..., 0].sum(), x)
                g[idx[valid]] = gx[valid]
                z[idx[valid]] = y.detach()[valid][:, 1:]
        d[idx[valid]] = y.detach()[valid][:, 0]
    return d, z, g


def _colour(desc, w, p, z, n, v):
    out = torch.empty((p.shape[0], 3), device=p.device, dtype=torch.float64)
    u = torch.cat([z, n, _encode(v, desc.pe_dir_L)], 1)
    ns = len(desc.sdf_layers())
    for idx, cells, valid in _by_cell(desc, _cell(desc, p)):
        y = torch.sigmoid(_mlp(_split(desc, w[cells].double())[ns:], u[idx], torch.relu))
        out[idx[valid]] = y[valid]
    return out


def _clip(o, d):
    with np.errstate(all="ignore"):
        a, b = (-1.0 - o) / d, (1.0 - o) / d
    lo, hi = torch.minimum(a, b).amax(1), torch.maximum(a, b).amin(1)
    return (lo <= hi) & (hi >= 0), lo.clamp(min=0), hi


def _skip(mask, o, d, t, tf):
    """Moves rays in empty voxels to the entry face of their next occupied voxel, voxel by voxel.  Returns
    (t, voxel, left the grid)."""
    n = mask.shape[0]
    flat = mask.reshape(-1)
    v = torch.floor((o + t[:, None] * d + 1.0) * (n / 2.0)).clamp(0, n - 1).long()
    step = torch.where(d > 0, 1, -1)
    out_t, out_v, gone = t.clone(), v.clone(), torch.zeros(len(t), dtype=torch.bool, device=t.device)
    idx = torch.nonzero(~flat[v[:, 0] + n * (v[:, 1] + n * v[:, 2])])[:, 0]
    v, step, oo, dd, ff = v[idx], step[idx], o[idx], d[idx], tf[idx]
    for _ in range(3 * n + 3):
        if not len(idx):
            break
        face = -1.0 + (v + (step > 0)) * (2.0 / n)
        tm, ax = ((face - oo) / dd).min(1)
        v = v + torch.nn.functional.one_hot(ax, 3) * step
        at = v.gather(1, ax[:, None])[:, 0]
        lost = (at < 0) | (at >= n) | (tm > ff)
        u = v.clamp(0, n - 1)
        found = ~lost & flat[u[:, 0] + n * (u[:, 1] + n * u[:, 2])]
        out_t[idx[found]], out_v[idx[found]], gone[idx[lost]] = tm[found], v[found], True
        keep = ~(lost | found)
        idx, v, step, oo, dd, ff = idx[keep], v[keep], step[keep], oo[keep], dd[keep], ff[keep]
    return out_t, out_v, gone


def _trace(scene, o, d, steps):
    """Sphere trace and shading of rays in 64 bits: rgb, depth, normal."""
    desc, w, mask = scene
    n = o.shape[0]
    rgb, normal = (torch.zeros((n, 3), device=DEV, dtype=torch.float64) for _ in range(2))
    depth = torch.full((n,), math.inf, device=DEV, dtype=torch.float64)
    hits = []
    for c0 in range(0, n, 20000000):
        oc, dc = o[c0:c0 + 20000000], d[c0:c0 + 20000000]
        ok, lo, hi = _clip(oc, dc)
        idx = torch.nonzero(ok)[:, 0]
        t = lo[idx]
        for _ in range(steps):
            oo, dd, ll, ff = oc[idx], dc[idx], lo[idx], hi[idx]
            cell = None
            if mask is not None:
                t, vox, gone = _skip(mask, oo, dd, t, ff)
                f = desc.occ_res // desc.N
                cell = vox[:, 0] // f + desc.N * (vox[:, 1] // f + desc.N * (vox[:, 2] // f))
                idx, t, oo, dd, ll, ff, cell = (x[~gone] for x in (idx, t, oo, dd, ll, ff, cell))
            if not len(idx):
                break
            s = _field(desc, w, oo + t[:, None] * dd, cell=cell)[0]
            hit = s.abs() < EPS
            depth[c0 + idx[hit]] = t[hit]
            hits.append(c0 + idx[hit])
            t = t + s
            keep = ~hit & (t >= ll) & (t <= ff)
            idx, t = idx[keep], t[keep]
    h = torch.cat(hits) if hits else torch.zeros(0, dtype=torch.long, device=DEV)
    if len(h):
        p = o[h] + depth[h, None] * d[h]
        _, z, g = _field(desc, w, p, want=True)
        nrm = torch.nn.functional.normalize(g, dim=1)
        normal[h] = nrm
        rgb[h] = _colour(desc, w, p, z, nrm, d[h])
    return rgb, depth, normal


def _pixel_rays(cam, W, H, dj=0.5, di=0.5, pix=None):
    cam = torch.from_numpy(np.asarray(cam, dtype=np.float64)).to(DEV)
    pix = torch.arange(W * H, device=DEV) if pix is None else pix
    x = ((pix % W).double() + dj - cam[14]) / cam[12]
    y = ((pix // W).double() + di - cam[15]) / cam[13]
    R = cam[:12].reshape(3, 4)
    d = torch.nn.functional.normalize(x[:, None] * R[:, 0] + y[:, None] * R[:, 1] + R[:, 2], dim=1)
    return R[:, 3].expand(len(pix), 3), d


def _frame(rgb, depth, normal):
    return dict(rgb=rgb, depth=depth, normal=normal, cell=None, steps=None, hit=None)


def _views(scene, views, steps):
    """Frames of (camera, W, H) views of one scene, traced together."""
    o, d = (torch.cat(v) for v in zip(*(_pixel_rays(*view) for view in views)))
    parts = [v.split([W * H for _, W, H in views]) for v in _trace(scene, o, d, steps)]
    return [_frame(*p) for p in zip(*parts)]


def _uniforms(seed, path, depth, dim):
    """SplitMix64 (Steele, Lea and Flood 2014): output (path * 16 + depth) * 4 + dim, its top 24 bits."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + ((path * np.uint64(16) + np.uint64(depth)) * np.uint64(4) + np.uint64(dim + 1)) * np.uint64(
            0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.from_numpy((z >> np.uint64(40)).astype(np.float64) * 2.0 ** -24).to(DEV)


def _paths(case, seed):
    W, H, spp = case["W"], case["H"], case["spp"]
    scene, cam = _scene(case["grid"]), S.orbit_cameras(1, W, H, seed=seed)[0]
    path = np.arange(W * H * spp, dtype=np.uint64)
    o, d = _pixel_rays(cam, W, H, _uniforms(seed, path, 0, 0), _uniforms(seed, path, 0, 1),
                       torch.arange(W * H, device=DEV).repeat_interleave(spp))
    horizon = torch.tensor(kns.SKY_HORIZON, device=DEV, dtype=torch.float64)
    zenith = torch.tensor(kns.SKY_ZENITH, device=DEV, dtype=torch.float64)
    light, beta = torch.zeros_like(d), torch.ones_like(d)
    alive = torch.arange(len(path), device=DEV)
    for k in range(case["depth"]):
        rgb, t, n = _trace(scene, o, d, case["steps"])
        miss = torch.isinf(t)
        a = 0.5 * (d[miss, 2:3] + 1.0)
        light[alive[miss]] += beta[miss] * ((1 - a) * horizon + a * zenith)
        hit = ~miss
        o, d, n, t, beta, alive = o[hit], d[hit], n[hit], t[hit], beta[hit] * rgb[hit], alive[hit]
        at = path[alive.cpu().numpy()]
        u1, u2 = _uniforms(seed, at, k, 2), _uniforms(seed, at, k, 3)
        sg = torch.where(n[:, 2] >= 0, 1.0, -1.0).double()  # basis of Duff et al. 2017
        q = -1.0 / (sg + n[:, 2])
        b = n[:, 0] * n[:, 1] * q
        e1 = torch.stack([1 + sg * n[:, 0] ** 2 * q, sg * b, -sg * n[:, 0]], 1)
        e2 = torch.stack([b, sg + n[:, 1] ** 2 * q, -n[:, 1]], 1)
        r, phi = torch.sqrt(u2), 2 * math.pi * u1
        o = o + t[:, None] * d + 1e-2 * n
        d = (r * torch.cos(phi))[:, None] * e1 + (r * torch.sin(phi))[:, None] * e2 + torch.sqrt(1 - u2)[:, None] * n
    return light.reshape(W * H, spp, 3).mean(1)


def _place(batch, desc, w, o, d, lo, hi):
    """Stratified and importance sample positions, merged in order."""
    Ns = batch["u_strat"].shape[1]
    t = lo[:, None] + (torch.arange(Ns, device=DEV) + batch["u_strat"].double()) / Ns * (hi - lo)[:, None]
    if batch["u_imp"].shape[1]:
        x = (o[:, None] + t[..., None] * d[:, None]).reshape(-1, 3)
        ls = torch.nn.functional.logsigmoid(64.0 * _field(desc, w, x)[0].reshape(t.shape))
        alpha = (1 - torch.exp(ls[:, 1:] - ls[:, :-1])).clamp(min=0)
        T = torch.cumprod(torch.cat([torch.ones_like(alpha[:, :1]), 1 - alpha], 1), 1)[:, :-1]
        cdf = torch.cumsum(T * alpha + 1e-5, 1)
        cdf = torch.cat([torch.zeros_like(cdf[:, :1]), cdf / cdf[:, -1:]], 1)
        u = batch["u_imp"].double()
        j = torch.searchsorted(cdf[:, 1:].contiguous(), u, right=True).clamp(max=Ns - 2)
        c0, c1, t0, t1 = cdf.gather(1, j), cdf.gather(1, j + 1), t.gather(1, j), t.gather(1, j + 1)
        t = torch.cat([t, t0 + (u - c0) / (c1 - c0) * (t1 - t0)], 1).sort(dim=1)[0]
    return t


def _vjp_field(desc, w, p, up, grad):
    """Adds sum up * d(parameters) to grad (cells, parameters)."""
    ns = len(desc.sdf_layers())
    for idx, cells, valid in _by_cell(desc, _cell(desc, p)):
        with torch.enable_grad():
            wc = w[cells].double().requires_grad_(True)
            layers = _split(desc, wc)[:ns]
            layers[-1] = (layers[-1][0][:, :1], layers[-1][1][:, :1])
            e = _encode(p[idx].reshape(-1, 3), desc.pe_pos_L).reshape(idx.shape[0], idx.shape[1], -1)
            y = _mlp(layers, e, _softplus)[..., 0]
            g, = torch.autograd.grad((y * torch.where(valid, up[idx], 0.0)).sum(), wc)
        grad[cells] += g


def _train(case, seed):
    desc = _train_desc(case)
    w = _weights(desc, seed)
    batch = _batch(case, seed)
    o, d, I = (batch[k].double() for k in ("origins", "dirs", "target"))
    ok, lo, hi = _clip(o, d)
    B = o.shape[0]
    miss = I[~ok].abs().sum()
    o, d, I, u = o[ok], d[ok], I[ok], {k: batch[k][ok] for k in ("u_strat", "u_imp")}
    t = _place(u, desc, w, o, d, lo[ok], hi[ok])
    n, S_ = t.shape
    x = (o[:, None] + t[..., None] * d[:, None]).reshape(-1, 3)
    v = d[:, None].expand(n, S_, 3).reshape(-1, 3)
    h = 1e-2
    q = torch.cat([x, batch["eik_points"].double()])
    off = h * torch.tensor([[1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1]], device=DEV).double()
    fd = (q[:, None] + off).reshape(-1, 3)
    dfd = _field(desc, w, fd)[0].reshape(-1, 6)
    g = (dfd[:, 0::2] - dfd[:, 1::2]) / (2 * h)
    g.requires_grad_(True)
    with torch.enable_grad():
        nrm = torch.nn.functional.normalize(g[:len(x)], dim=1, eps=0.0)
        eik = ((g[len(x):].norm(dim=1) - 1) ** 2).mean() if len(g) > len(x) else g.sum() * 0
    ns = len(desc.sdf_layers())

    def centre(wc, idx, nn):
        layers = _split(desc, wc)
        e = _encode(x[idx].reshape(-1, 3), desc.pe_pos_L).reshape(idx.shape[0], idx.shape[1], -1)
        y = _mlp(layers[:ns], e, _softplus)
        gv = _encode(v[idx].reshape(-1, 3), desc.pe_dir_L).reshape(idx.shape[0], idx.shape[1], -1)
        return y[..., 0], torch.sigmoid(_mlp(layers[ns:], torch.cat([y[..., 1:], nn, gv], -1), torch.relu))

    dc = torch.empty(len(x), device=DEV, dtype=torch.float64)
    cc = torch.empty((len(x), 3), device=DEV, dtype=torch.float64)
    n0 = nrm.detach()
    groups = list(_by_cell(desc, _cell(desc, x)))
    for idx, cells, valid in groups:
        a, b = centre(w[cells].double(), idx, n0[idx])
        dc[idx[valid]], cc[idx[valid]] = a[valid], b[valid]
    dc.requires_grad_(True)
    cc.requires_grad_(True)
    with torch.enable_grad():
        ls = torch.nn.functional.logsigmoid(20.0 * dc.reshape(n, S_))
        alpha = (1 - torch.exp(ls[:, 1:] - ls[:, :-1])).clamp(min=0)
        T = torch.cumprod(torch.cat([torch.ones_like(alpha[:, :1]), 1 - alpha], 1), 1)[:, :-1]
        C = ((T * alpha)[..., None] * cc.reshape(n, S_, 3)[:, :-1]).sum(1)
        colour = ((C - I).abs().sum() + miss) / B
    udc, ucc = torch.autograd.grad(colour, (dc, cc))
    grad = torch.zeros_like(w, dtype=torch.float64)
    un = torch.zeros_like(n0)
    for idx, cells, valid in groups:
        with torch.enable_grad():
            wc, nn = w[cells].double().requires_grad_(True), n0[idx].requires_grad_(True)
            a, b = centre(wc, idx, nn)
            s = (a * torch.where(valid, udc[idx], 0.0)).sum() + (b * torch.where(valid[..., None], ucc[idx], 0.0)).sum()
            gw, gn = torch.autograd.grad(s, (wc, nn))
        grad[cells] += gw
        un[idx[valid]] = gn[valid]
    with torch.enable_grad():
        ug, = torch.autograd.grad((nrm * un).sum() + 0.1 * eik, g)
    up = torch.stack([ug, -ug], 2).reshape(-1) / (2 * h)
    _vjp_field(desc, w, fd, up, grad)
    lc, le = colour.detach(), eik.detach()
    grad = grad.reshape(-1)
    if case["autograd"]:
        return lc + 0.1 * le, grad
    return torch.stack([lc + 0.1 * le, lc, le]), grad


@torch.no_grad()
def exact(case, seed):
    op = case["op"]
    if op == "render":
        W, H = case["W"], case["H"]
        frames = _views(_scene(case["grid"]), [(c, W, H) for c in S.orbit_cameras(case["cams"], W, H, seed=seed)],
                        case["steps"])
        return _frame(*(torch.cat([f[k] for f in frames]) for k in ("rgb", "depth", "normal")))
    if op == "views":
        req = _requests(case, seed)
        frames = [None] * len(req)
        for k in range(case["grids"]):
            at = [i for i, r in enumerate(req) if r[3] == k]
            if at:
                for i, f in zip(at, _views(_scene(case["grid"], k), [req[i][:3] for i in at], case["steps"])):
                    frames[i] = f
        return frames
    if op == "rays":
        o, d = _rays(case, seed)
        return _frame(*_trace(_scene(case["grid"]), o.double(), d.double(), case["steps"]))
    if op == "paths":
        return _paths(case, seed)
    if op == "points":
        desc, w, _ = _scene(case["grid"])
        d, z, g = _field(desc, w, _points(case, seed).double(), want=case["full"])
        return (d, z, g)
    return _train(case, seed)
