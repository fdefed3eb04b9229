"""Performance cases of the Adaptive Multi-NeRF rendering path.

Every case is work that a program using this library asks of it through its public entry
points (`amnerf.Renderer` and the functions beside it): renders of the three seeded scene
families of the repository (c1: the parity scene, <= 16 leaves of 2 x 32; c2: the paper-scale
scene, 256 leaves of 4 x 64; c4: the imbalanced scene, up to 4096 leaves of 4 x 64) in every
precision and with every sampling option, from one 64 x 64 tile to 8 views of 800 x 800, a
render from host buffers, and the training of the proposal sampler.

Inputs are made here from the seed alone, on the GPU (densities, cameras, weights); networks
have a nonzero bias in every layer, as trained ones do.  `exact` restates the method in 64
bits with torch and numpy only: the KD tree, the crossings of every ray with every node, the
sample positions, the networks and the quadrature.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2310_01881_gb300 import amnerf

STEPS = 8          # samples per crossing, as in every workload of the repository
T_TERM = 1e-4      # early-termination transmittance
LX, LD = 10, 4     # frequencies of the position's and the direction's encoding
K0 = 3 + 6 * LX + 3 + 6 * LD
FOV = math.radians(40.0)
RADIUS = 3.0
PIN, PH, PO = 90, 32, 65   # the proposal network's layers
MASK64 = (1 << 64) - 1

# Scene families: guidance grid, leaf networks, samples per ray at most.
FAMILIES = {
    "c1": dict(G=64, width=32, hidden=2, cap=64),
    "c2": dict(G=128, width=64, hidden=4, cap=192),
    "c4": dict(G=256, width=64, hidden=4, cap=192),
}


def _case(name, kind="render", scene="c2", prec="bf16", w=800, h=800, views=1, **more):
    f = FAMILIES[scene]
    c = dict(name=name, kind=kind, scene=scene, prec=prec, w=w, h=h, views=views, G=f["G"], width=f["width"],
             hidden=f["hidden"], cap=f["cap"], depth={"c1": 4, "c2": 8, "c4": 12}[scene],
             frac=1.0 / 256.0 if scene == "c2" else 0.0, density=1.0, jitter=0, skip=-1.0, lod_px=0.0, wave=0,
             coverage=0.0, train_steps=0, batch=0)
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: one 64 x 64 tile of the parity scene with the plain FP32 networks (a
        # thumbnail, or one tile of a progressive preview): launches and latency
        _case("tile_fp32", scene="c1", prec="fp32", w=64, h=64),
        # a crop of odd size through the paper-scale scene (the region a user is editing): a few
        # tiles per leaf network, most of them partly filled
        _case("crop_bf16", w=123, h=77),
        # one 800 x 800 view with the plain FP32 networks: the accurate render
        _case("view_fp32", prec="fp32"),
        # the benchmark's step: 8 views of 800 x 800, BF16 networks
        _case("views_bf16", views=8),
        # one view with E4M3 networks, per-row activation scales (loaded without calibration)
        _case("view_fp8", prec="fp8"),
        # two views with E4M3 networks, static scales from a calibration on other views
        _case("views_fp8s", prec="fp8s", views=2),
        # one 1920 x 1080 frame of the imbalanced scene: 4096 leaf networks
        _case("frame_4096", scene="c4", w=1920, h=1080),
        # four views from page-locked host rays to host pixels: the end-to-end call
        _case("host_bf16", kind="host", views=4),
        # stratified jitter and empty-space skipping together, one view
        _case("view_jitter_skip", jitter=12345, skip=0.01),
        # adaptive hierarchical sampling: 1280 x 720 frame, one network per node
        _case("frame_lod", scene="c4", depth=10, w=1280, h=720, lod_px=128.0),
        # the proposal sampler on an opaque scene (where it pays), 1920 x 1080
        _case("frame_proposal", scene="c1", width=64, hidden=4, w=1920, h=1080, density=1000.0, coverage=0.95),
        # training the proposal sampler: targets of two 480 x 270 views, then Adam steps
        _case("proposal_train", kind="train", w=480, h=270, views=2, train_steps=24, batch=8192),
    ]


def _rays_between(rng, lo, hi):
    """(w, h, views): about exp(uniform(log lo, log hi)) rays, any aspect from 1:1 to 2:1."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    views = rng.choice([1, 1, 1, 2, 3]) if n > 20000 else 1
    aspect = rng.uniform(1.0, 2.0)
    h = max(16, int(math.sqrt(n / views / aspect)))
    return max(16, int(h * aspect)), h, views


def draw(rng: random.Random):
    kind = rng.choice(["render"] * 8 + ["host", "train"])
    if kind == "train":
        w, h, views = _rays_between(rng, 2e4, 2.5e5)
        c = _case("", kind="train", w=w, h=h, views=views, depth=rng.randint(6, 8),
                  density=rng.choice([1.0, 10.0, 100.0]), train_steps=rng.randint(4, 24),
                  batch=rng.choice([1000, 2048, 4096, 8192]))
    else:
        scene = rng.choice(["c1", "c2", "c2", "c4"])
        prec = rng.choice(["fp32", "bf16", "bf16", "bf16", "fp8", "fp8s"])
        most = {"fp32": 5e5, "bf16": 2e6, "fp8": 6e5, "fp8s": 1.2e6}[prec]
        w, h, views = _rays_between(rng, 4096, most)
        c = _case("", kind=kind, scene=scene, prec=prec, w=w, h=h, views=views)
        if scene == "c4":
            c["depth"] = rng.randint(9, 11)
        elif scene == "c2":
            c["depth"] = rng.randint(6, 8)
        else:
            c["depth"] = rng.randint(2, 4)
            c["width"], c["hidden"] = rng.choice([(32, 2), (32, 2), (64, 4), (32, 5), (64, 3)])
            c["density"] = rng.choice([1.0, 1.0, 100.0, 1000.0])
        c["cap"] = rng.choice([c["cap"], c["cap"], 64, 136, 200])
        c["jitter"] = rng.choice([0, 0, 0, rng.randint(1, 10**9)])
        c["skip"] = rng.choice([-1.0, -1.0, -1.0, 0.01])
        if kind == "render":
            option = rng.choice(["none", "none", "none", "lod", "wave", "proposal"])
            if option == "lod" and scene != "c1":
                c["lod_px"] = rng.choice([32.0, 64.0, 128.0])
                c["depth"] = min(c["depth"], 9)
            elif option == "wave":
                c["wave"] = rng.choice([2, 4])
            elif option == "proposal" and scene == "c1" and prec == "bf16":
                c["coverage"] = rng.choice([0.95, 0.99])
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------

def _grid(case, seed):
    """The guidance density at the cell centres of [-1, 1]^3 as float32 [z, y, x] on the GPU."""
    rng = np.random.default_rng([seed, 11])
    G, kind = case["G"], case["scene"]
    dev = torch.device("cuda")
    ax = -1.0 + (torch.arange(G, device=dev, dtype=torch.float64) + 0.5) * (2.0 / G)
    g = torch.zeros((G, G, G), device=dev, dtype=torch.float64)

    def window(c, half):
        lo = np.clip(np.floor((c - half + 1.0) * G / 2), 0, G).astype(int)
        hi = np.clip(np.ceil((c + half + 1.0) * G / 2), 0, G).astype(int)
        x, y, z = (ax[lo[a]:hi[a]] - c[a] for a in range(3))
        return (slice(lo[2], hi[2]), slice(lo[1], hi[1]), slice(lo[0], hi[0])), x[None, None, :], y[None, :, None], \
            z[:, None, None]

    def gauss(c, ic, half, peak):
        at, x, y, z = window(c, half)
        q = ic[0, 0] * x * x + ic[1, 1] * y * y + ic[2, 2] * z * z + 2 * (ic[0, 1] * x * y + ic[0, 2] * x * z
                                                                            + ic[1, 2] * y * z)
        g[at] += peak * torch.exp(-0.5 * q)

    def shell(c, r, width, peak):
        at, x, y, z = window(c, r + 6 * width)
        g[at] += peak * torch.exp(-0.5 * ((torch.sqrt(x * x + y * y + z * z) - r) / width) ** 2)

    if kind == "c1":
        for _ in range(4):
            c, s = rng.uniform(-0.6, 0.6, 3), rng.uniform(0.1, 0.3)
            gauss(c, np.eye(3) / (s * s), 6 * s, 50.0)
    elif kind == "c2":
        for _ in range(8):
            c, s = rng.uniform(-0.6, 0.6, 3), rng.uniform(0.05, 0.3, 3)
            R, _ = np.linalg.qr(rng.normal(size=(3, 3)))
            gauss(c, R @ np.diag(1.0 / (s * s)) @ R.T, 6 * s.max(), 50.0)
        shell(np.zeros(3), 0.7, 0.02, 200.0)
    else:
        for _ in range(64):
            c = rng.uniform(-0.9, 0.9, 3)
            s = float(np.clip(math.exp(rng.normal(math.log(0.05), 0.7)), 0.005, 0.5))
            gauss(c, np.eye(3) / (s * s), 6 * s, 50.0)
        for _ in range(3):
            shell(rng.uniform(-0.3, 0.3, 3), rng.uniform(0.2, 0.6), 0.01, 200.0)
    return (g * case["density"]).to(torch.float32)


def _rays(case, seed, stream=12, views=None, w=None, h=None):
    """float32 (o, d) on the GPU: pinhole views from seeded directions at radius 3."""
    views, w, h = views or case["views"], w or case["w"], h or case["h"]
    dev = torch.device("cuda")
    th = math.tan(FOV / 2.0)
    ii = ((torch.arange(w, device=dev, dtype=torch.float64) + 0.5) / w * 2.0 - 1.0) * th * (w / h)
    jj = (1.0 - (torch.arange(h, device=dev, dtype=torch.float64) + 0.5) / h * 2.0) * th
    os_, ds = [], []
    for v in range(views):
        u = np.random.default_rng([seed, stream, v]).normal(size=3)
        u /= np.linalg.norm(u)
        up = np.array([0.0, 0.0, 1.0]) if abs(u[2]) <= 0.99 else np.array([0.0, 1.0, 0.0])
        right = np.cross(-u, up)
        right /= np.linalg.norm(right)
        tup = np.cross(right, -u)
        f, r, t = (torch.tensor(a, device=dev) for a in (-u, right, tup))
        d = (f + ii[None, :, None] * r + jj[:, None, None] * t).reshape(-1, 3)
        d = d / d.norm(dim=1, keepdim=True)
        ds.append(d.to(torch.float32))
        os_.append(torch.tensor(RADIUS * u, device=dev).to(torch.float32).expand(d.shape))
    return torch.cat(os_).contiguous(), torch.cat(ds).contiguous()


def _net_sizes(case):
    dims = [K0] + [case["width"]] * case["hidden"] + [4]
    return list(zip(dims[1:], dims[:-1]))


def _weights(case, seed, grid, cells):
    """float32 [networks, parameters] on the GPU: Xavier-uniform matrices, small biases, the
    density head's bias at the log of the node's mean guidance density."""
    n = len(cells)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 7919 + 13)
    sizes = _net_sizes(case)
    per = sum(fo * fi + fo for fo, fi in sizes)
    W = torch.rand((n, per), generator=gen, device="cuda").mul_(2.0).sub_(1.0)
    at = 0
    for fo, fi in sizes:
        W[:, at:at + fo * fi] *= math.sqrt(6.0 / (fi + fo))
        W[:, at + fo * fi:at + fo * fi + fo] *= 0.1
        at += fo * fi + fo
    S = torch.zeros([s + 1 for s in grid.shape], device="cuda", dtype=torch.float64)
    S[1:, 1:, 1:] = grid.double().cumsum(0).cumsum(1).cumsum(2)
    c = torch.as_tensor(np.asarray(cells), device="cuda").long()
    x0, y0, z0, x1, y1, z1 = c.unbind(1)
    m = (S[z1, y1, x1] - S[z0, y1, x1] - S[z1, y0, x1] - S[z1, y1, x0] + S[z0, y0, x1] + S[z0, y1, x0]
         + S[z1, y0, x0] - S[z0, y0, x0])
    mean = (m / ((x1 - x0) * (y1 - y0) * (z1 - z0))).clamp_min(1e-3 * case["density"])
    W[:, per - 4] += mean.log().to(torch.float32)
    return W


def _proposal_fit(case, seed, grid):
    """float32 [6113] parameters of a proposal network fitted here, in torch, to the density
    grid's own compositing weights along seeded rays (a stand-in for a trained checkpoint)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 31 + 7)
    P = []
    for fo, fi in ((PH, PIN), (PH, PH), (PO, PH)):
        a = math.sqrt(6.0 / (fi + fo))
        P += [(torch.rand((fo, fi), generator=gen, device="cuda") * 2 - 1) * a, torch.zeros(fo, device="cuda")]
    if case["kind"] == "train":
        return torch.cat([p.reshape(-1) for p in P])
    o, d = _rays(case, seed, stream=14, views=8, w=128, h=128)
    o, d = o.double(), d.double()
    t0, t1 = _slab(torch.tensor([[-1.0] * 3], device="cuda", dtype=torch.float64),
                   torch.tensor([[1.0] * 3], device="cuda", dtype=torch.float64), o, d)
    hit = (t1 > t0)[:, 0]
    o, d, t0, t1 = o[hit], d[hit], t0[hit], t1[hit]
    k = torch.arange(256, device="cuda", dtype=torch.float64)
    t = t0 + (k + 0.5) / 256 * (t1 - t0)
    c = ((o[:, None, :] + t[:, :, None] * d[:, None, :] + 1.0) * case["G"] / 2).long().clamp_(0, case["G"] - 1)
    tau = grid.double()[c[..., 2], c[..., 1], c[..., 0]] * (t1 - t0) / 256
    T = torch.exp(-tau.cumsum(1))
    wgt = torch.cat([1.0 - T[:, :1], T[:, :-1] - T[:, 1:]], 1).reshape(-1, 64, 4).sum(2)
    p = torch.cat([wgt, T[:, -1:]], 1).float()
    x = torch.cat([_gamma(o + t0 * d, LX), _gamma(d, LD)], 1).float()
    P = [q.requires_grad_(True) for q in P]
    m, v = [torch.zeros_like(q) for q in P], [torch.zeros_like(q) for q in P]
    n = x.shape[0]
    for s in range(1, 151):
        i = torch.randint(0, n, (4096,), generator=gen, device="cuda")
        hid = torch.relu(x[i] @ P[0].T + P[1])
        hid = torch.relu(hid @ P[2].T + P[3])
        loss = -(p[i] * torch.log_softmax(hid @ P[4].T + P[5], 1)).sum(1).mean()
        for j, gr in enumerate(torch.autograd.grad(loss, P)):
            m[j] = 0.9 * m[j] + 0.1 * gr
            v[j] = 0.999 * v[j] + 0.001 * gr * gr
            P[j].data -= 5e-3 * (m[j] / (1 - 0.9 ** s)) / ((v[j] / (1 - 0.999 ** s)).sqrt() + 1e-8)
    return torch.cat([q.detach().reshape(-1) for q in P])


def _lod(case):
    """lod_px footprints of a pixel per unit distance (0: leaves only)."""
    return case["lod_px"] * 2.0 * math.tan(FOV / 2.0) / case["h"]


def _options(case):
    kw = dict(steps=STEPS, cap=case["cap"], t_term=T_TERM)
    if case["jitter"]:
        kw["jitter"] = case["jitter"]
    if case["skip"] >= 0:
        kw["skip_empty"] = case["skip"]
    if case["wave"]:
        kw["ert_wave"] = case["wave"]
    if case["lod_px"]:
        kw["lod"] = _lod(case)
    if case["coverage"]:
        kw.update(proposal=True, coverage=case["coverage"], max_bins=64)
    return kw


def prepare(case, seed):
    grid = _grid(case, seed)
    r = amnerf.Renderer(0)
    r.build_tree(grid.cpu().numpy(), case["depth"], case["frac"])
    cells = r.network_cells() if case["lod_px"] else r.leaf_cells()
    W = _weights(case, seed, grid, cells).cpu().numpy().reshape(-1)
    shape = (case["width"], case["hidden"], LX, LD)
    if case["prec"] == "fp8s":
        r.load_mlps(W, *shape, "fp32")
        co, cd = _rays(case, seed, stream=13, views=1, w=96, h=96)
        amax = r.calibrate_fp8(co, cd, case["hidden"], steps=STEPS, cap=case["cap"], t_term=T_TERM,
                               lod=_lod(case))
        r.load_mlps(W, *shape, "fp8", act_max=amax)
    else:
        r.load_mlps(W, *shape, case["prec"])
    o, d = _rays(case, seed)
    s = dict(case=case, r=r, o=o, d=d, options=_options(case))
    n = o.shape[0]
    if case["coverage"]:
        amnerf.amnerf_proposal_set(r.ctx, _proposal_fit(case, seed, grid).cpu().numpy())
    if case["kind"] == "train":
        s["params"] = _proposal_fit(case, seed, grid).cpu().numpy()
        s["seed"] = seed + 1
        s["out"] = [torch.empty((n, 3), device="cuda"), torch.empty(n, device="cuda"), torch.empty(n, device="cuda")]
        s["targets"] = torch.empty((n, PO), device="cuda")
        s["root"] = torch.empty((n, 2), device="cuda")
    if case["kind"] == "host":
        pin = lambda *shape: torch.empty(shape, pin_memory=True)  # noqa: E731
        ho, hd = pin(n, 3), pin(n, 3)
        ho.copy_(o)
        hd.copy_(d)
        s["host"] = [t.numpy() for t in (ho, hd, pin(n, 3), pin(n), pin(n))]
        s["keep"] = (ho, hd)
    return s


def run(s):
    case, r = s["case"], s["r"]
    if case["kind"] == "host":
        ho, hd, rgb, depth, opacity = s["host"]
        amnerf.amnerf_render_host(r.ctx, ho, hd, rgb, depth, opacity, **s["options"])
        return rgb, depth, opacity
    if case["kind"] == "train":
        o, d = s["o"], s["d"]
        amnerf.amnerf_proposal_set(r.ctx, s["params"])
        amnerf.amnerf_proposal_targets(r.ctx, o, d, *s["out"], s["targets"], s["root"], steps=STEPS,
                                       cap=case["cap"], t_term=T_TERM)
        losses = amnerf.amnerf_proposal_train(r.ctx, o, d, s["root"], s["targets"], case["train_steps"],
                                              case["batch"], lr=3e-3, seed=s["seed"])
        params, m, v, _ = amnerf.amnerf_proposal_get(r.ctx)
        return s["out"][0], s["targets"], losses, params, m, v
    return r.render(s["o"], s["d"], **s["options"])


# ---------------------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------------------

def _tree(grid, depth, frac):
    """Density-median KD tree of a float32 [z, y, x] array: (lo, hi) cells [n, 3], split axis (-1:
    leaf), parent, level; nodes in preorder."""
    lo_, hi_, ax_, par_, lev_ = [], [], [], [], []
    total = [None]

    def node(c0, c1, lev, parent):
        n = [c1[a] - c0[a] for a in range(3)]
        axis = n.index(max(n))
        blk = grid[c0[2]:c1[2], c0[1]:c1[1], c0[0]:c1[0]]
        sl = blk.sum(axis=tuple(i for i in range(3) if i != 2 - axis), dtype=np.float64)
        m = float(sl.sum())
        total[0] = m if lev == 0 else total[0]
        me = len(ax_)
        lo_.append(c0)
        hi_.append(c1)
        par_.append(parent)
        lev_.append(lev)
        if lev >= depth or n[axis] <= 1 or (frac > 0 and m <= frac * total[0]):
            ax_.append(-1)
            return
        ax_.append(axis)
        k = n[axis] // 2
        if m > 0:
            past = np.nonzero(np.cumsum(sl[:-1]) >= 0.5 * m)[0]
            k = int(past[0]) + 1 if len(past) else n[axis] - 1
        mid1, mid0 = list(c1), list(c0)
        mid1[axis] = mid0[axis] = c0[axis] + k
        node(c0, tuple(mid1), lev + 1, me)
        node(tuple(mid0), c1, lev + 1, me)

    G = grid.shape[0]
    node((0, 0, 0), (G, G, G), 0, -1)
    return np.array(lo_), np.array(hi_), np.array(ax_), np.array(par_), np.array(lev_)


def _networks(tree):
    """Cells of every network and the network of every node: leaves in order, then inner nodes."""
    lo, hi, ax = tree[:3]
    leaf, inner = np.nonzero(ax < 0)[0], np.nonzero(ax >= 0)[0]
    net = np.empty(len(ax), np.int64)
    net[np.concatenate([leaf, inner])] = np.arange(len(ax))
    cells = np.concatenate([lo, hi], 1)
    return cells[leaf], np.concatenate([cells[leaf], cells[inner]]), net


def _slab(lo, hi, o, d):
    """(entry, exit) [rays, boxes] of rays through boxes lo, hi [boxes, 3]."""
    e = torch.zeros((o.shape[0], lo.shape[0]), device=o.device, dtype=o.dtype)
    x = torch.full_like(e, math.inf)
    for a in range(3):
        inv = 1.0 / d[:, a:a + 1]
        t0, t1 = (lo[None, :, a] - o[:, a:a + 1]) * inv, (hi[None, :, a] - o[:, a:a + 1]) * inv
        e = torch.maximum(e, torch.minimum(t0, t1))
        x = torch.minimum(x, torch.maximum(t0, t1))
    return e, x


def _gamma(p, L):
    f = [p]
    for k in range(L):
        f += [torch.sin(math.pi * 2.0 ** k * p), torch.cos(math.pi * 2.0 ** k * p)]
    return torch.cat(f, 1)


def _mix64(z):
    """splitmix64's finaliser on int64 tensors (wrapping products, logical shifts)."""
    s = lambda v, n: (v >> n) & ((1 << (64 - n)) - 1)  # noqa: E731
    i64 = lambda c: c - (1 << 64) if c >= 1 << 63 else c  # noqa: E731
    z = (z ^ s(z, 30)) * i64(0xBF58476D1CE4E5B9)
    z = (z ^ s(z, 27)) * i64(0x94D049BB133111EB)
    return z ^ s(z, 31)


def _fractions(case, o32, d32, k):
    """[rays, STEPS] places of the samples of crossing k (an int64 tensor, per ray) in their strata."""
    if not case["jitter"]:
        return torch.full((o32.shape[0], STEPS), 0.5, device=o32.device, dtype=torch.float64)
    bits = torch.cat([o32, d32], 1).view(torch.int32).long() & 0xFFFFFFFF
    key = torch.full((o32.shape[0],), case["jitter"], device=o32.device, dtype=torch.int64)
    for i in range(0, 6, 2):
        key = _mix64(key ^ (bits[:, i] | (bits[:, i + 1] << 32)))
    j = torch.arange(STEPS, device=o32.device)[None, :]
    n = k[:, None] * STEPS + j + 1
    z = _mix64(key[:, None] + (0x9E3779B97F4A7C15 - (1 << 64)) * n)
    return ((z >> 40) & 0xFFFFFF).double() / 2.0 ** 24


def _prop_predict(P, o, d, t0):
    """Softmax outputs [rays, 65] of the proposal network with parameters P (float64)."""
    at, x = 0, torch.cat([_gamma(o + t0 * d, LX), _gamma(d, LD)], 1)
    for i, (fo, fi) in enumerate(((PH, PIN), (PH, PH), (PO, PH))):
        x = x @ P[at:at + fo * fi].reshape(fo, fi).T + P[at + fo * fi:at + fo * fi + fo]
        x = torch.relu(x) if i < 2 else x
        at += fo * fi + fo
    return torch.softmax(x, 1)


def _kept_bins(case, P, o, d, t0):
    """[rays, 64] bins kept: by decreasing mass until the coverage is reached (the background
    counts toward it)."""
    q = _prop_predict(P, o, d, t0)
    s, i = torch.sort(q, dim=1, descending=True, stable=True)
    take = torch.cat([torch.zeros_like(s[:, :1]), s.cumsum(1)[:, :-1]], 1) < case["coverage"]
    kept = torch.zeros_like(take).scatter(1, i, take)
    return kept[:, :64]


def _crossings(case, nodes, net, grid, P, o32, d32, maxc):
    """Kept crossings of a chunk of rays, front to back: network (-1: none), entry, exit [rays, maxc]."""
    o, d = o32.double(), d32.double()
    lo, hi, ax, par, lev = nodes
    e, x = _slab(lo, hi, o, d)
    crossed = x > e
    leaf = (ax < 0)[None, :].expand_as(crossed)
    if case["lod_px"]:
        lod = float(np.float32(_lod(case)))
        ext = (hi - lo).gather(1, ax.clamp_min(0)[:, None])[:, 0]
        stop = leaf | ~(ext[None, :] > lod * e)
        reach = crossed.clone()
        for level in range(1, int(lev.max()) + 1):
            i = (lev == level).nonzero()[:, 0]
            reach[:, i] &= reach[:, par[i]] & ~stop[:, par[i]]
        emit = reach & stop
    else:
        emit = crossed & leaf
    key = torch.where(emit, e, torch.full_like(e, math.inf))
    most = max(1, int(emit.sum(1).max()))
    top, idx = torch.topk(key, most, dim=1, largest=False, sorted=True)
    xo = x.gather(1, idx)
    nt = net[idx]
    ok = torch.isfinite(top)
    if P is not None:
        t0, t1 = e[:, :1], x[:, :1]
        miss = ~(t1 > t0)
        t0 = torch.where(miss, torch.zeros_like(t0), t0)
        w = torch.where(miss, torch.zeros_like(t0), (t1 - t0) / 64)
        kept = _kept_bins(case, P, o, d, t0)
        b = torch.arange(64, device=o.device)
        over = ((top[:, :, None] < (t0 + (b + 1) * w)[:, None, :]) & (xo[:, :, None] > (t0 + b * w)[:, None, :])
                & kept[:, None, :]).any(2)
        ok = ok & over
    n = o.shape[0]
    cnt = torch.zeros(n, device=o.device, dtype=torch.int64)
    out_n = torch.full((n, maxc + 1), -1, device=o.device, dtype=torch.int64)
    out_e, out_x = (torch.zeros((n, maxc + 1), device=o.device, dtype=torch.float64) for _ in range(2))
    for k in range(most):
        keep = ok[:, k] & (cnt < maxc)
        if case["skip"] >= 0:
            t = top[:, k:k + 1] + (torch.arange(STEPS, device=o.device) + _fractions(case, o32, d32, cnt)) * (
                (xo[:, k:k + 1] - top[:, k:k + 1]) / STEPS)
            p = torch.nan_to_num(o[:, None, :] + t[:, :, None] * d[:, None, :], 0.0, 0.0, 0.0)
            c = torch.floor((p + 1.0) * case["G"] / 2).long().clamp_(0, case["G"] - 1)
            keep = keep & (grid[c[..., 2], c[..., 1], c[..., 0]] > float(np.float32(case["skip"]))).any(1)
        at = torch.where(keep, cnt, torch.full_like(cnt, maxc))[:, None]  # column maxc takes what is dropped
        out_n.scatter_(1, at, nt[:, k:k + 1])
        out_e.scatter_(1, at, top[:, k:k + 1])
        out_x.scatter_(1, at, xo[:, k:k + 1])
        cnt = cnt + keep
    return torch.where(torch.arange(maxc, device=o.device)[None, :] < cnt[:, None], out_n[:, :maxc], -1), \
        out_e[:, :maxc], out_x[:, :maxc], (e[:, 0], x[:, 0])


def _scene64(case, seed):
    """What the 64-bit method needs: node tensors, networks of nodes, grid, networks' cells."""
    grid = _grid(case, seed)
    tree = _tree(grid.cpu().numpy(), case["depth"], case["frac"])
    leaf_cells, all_cells, net = _networks(tree)
    dev = grid.device
    lo, hi, ax, par, lev = tree
    box = lambda c: torch.tensor(-1.0 + 2.0 * (c / case["G"]), device=dev)  # noqa: E731
    use = np.arange(len(ax)) if case["lod_px"] else np.concatenate([[0], np.nonzero(ax < 0)[0]])  # root first
    if not case["lod_px"] and ax[0] < 0:
        use = use[:1]
    t = lambda v: torch.tensor(v[use], device=dev)  # noqa: E731
    return (box(lo[use]), box(hi[use]), t(ax), t(par), t(lev)), t(net), grid, \
        all_cells if case["lod_px"] else leaf_cells


def _chunk(nodes, case):
    per = nodes[0].shape[0] * 8 * 12 + (64 * 64 * 8 if case["coverage"] else 0)
    return max(256, int(6e9 // per))


def _all_crossings(case, nodes, net, grid, P, o, d, maxc):
    parts = [_crossings(case, nodes, net, grid, P, o[i:i + c], d[i:i + c], maxc)
             for c in (_chunk(nodes, case),) for i in range(0, o.shape[0], c)]
    return torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts]), torch.cat([p[2] for p in parts]), \
        torch.cat([p[3][0] for p in parts]), torch.cat([p[3][1] for p in parts])


def _proposal64(case, seed, grid):
    return _proposal_fit(case, seed, grid).double() if case["coverage"] else None


def _samples_per_ray(case):
    """Samples per ray of the case's scene and options, from 4096 of its rays (seed 1)."""
    nodes, net, grid, _ = _scene64(case, 1)
    o, d = _rays(case, 1)
    i = torch.randperm(o.shape[0], generator=torch.Generator().manual_seed(1))[:4096].to(o.device)
    nt = _all_crossings(case, nodes, net, grid, _proposal64(case, 1, grid), o[i], d[i], case["cap"] // STEPS)[0]
    return float((nt >= 0).sum()) * STEPS / len(i)


def work(case):
    n = case["w"] * case["h"] * case["views"]
    spr = _samples_per_ray(case)
    sizes = _net_sizes(case)
    flops = n * spr * sum(2.0 * fo * fi for fo, fi in sizes)
    nets = min(2 ** case["depth"] * (2 if case["lod_px"] else 1), n * spr / STEPS)
    moved = n * (24 + 20) + nets * sum(fo * fi + fo for fo, fi in sizes) * {"fp32": 4, "bf16": 2}.get(case["prec"], 1)
    if case["coverage"]:
        flops += n * 2.0 * (PH * PIN + PH * PH + PO * PH)
    if case["kind"] == "train":
        rays = case["train_steps"] * case["batch"]
        flops += rays * 6.0 * (PH * PIN + PH * PH + PO * PH)
        moved += n * (PO * 4 + 8) + rays * (24 + 8 + PO * 4)
    return {"bytes": float(moved), "flops": float(flops)}


def _render64(case, seed, bins=False):
    nodes, net, grid, cells = _scene64(case, seed)
    W = _weights(case, seed, grid, cells).double()
    o32, d32 = _rays(case, seed)
    o, d = o32.double(), d32.double()
    n, maxc = o.shape[0], case["cap"] // STEPS
    nt, te, tx, r0, r1 = _all_crossings(case, nodes, net, grid, _proposal64(case, seed, grid), o32, d32, maxc)
    maxc = max(1, int((nt >= 0).sum(1).max()))
    nt, te, tx = nt[:, :maxc], te[:, :maxc], tx[:, :maxc]
    delta = (tx - te) / STEPS
    t = torch.empty((n, maxc, STEPS), device=o.device, dtype=torch.float64)
    j = torch.arange(STEPS, device=o.device)
    for k in range(maxc):
        kk = torch.full((n,), k, device=o.device, dtype=torch.int64)
        t[:, k] = te[:, k:k + 1] + (j + _fractions(case, o32, d32, kk)) * delta[:, k:k + 1]
    out = torch.zeros((n, maxc, STEPS, 4), device=o.device, dtype=torch.float64)
    flat = nt.reshape(-1)
    order = torch.argsort(flat, stable=True)
    counts = torch.bincount(flat + 1, minlength=W.shape[0] + 1).cpu().tolist()
    at = counts[0]
    sizes = _net_sizes(case)
    outf, tf = out.view(-1, STEPS, 4), t.view(-1, STEPS)
    for m, c in enumerate(counts[1:]):
        w, mats = 0, []
        for fo, fi in sizes if c else ():
            mats.append((W[m, w:w + fo * fi].reshape(fo, fi).T, W[m, w + fo * fi:w + fo * fi + fo]))
            w += fo * fi + fo
        for i in range(at, at + c, 1 << 18):
            ids = order[i:min(i + (1 << 18), at + c)]
            ray = torch.div(ids, maxc, rounding_mode="floor")
            dd = d[ray]
            p = (o[ray][:, None, :] + tf[ids][:, :, None] * dd[:, None, :]).reshape(-1, 3)
            gd = _gamma(dd, LD)[:, None, :].expand(-1, STEPS, -1).reshape(p.shape[0], -1)
            hdn = torch.cat([_gamma(p, LX), gd], 1)
            for A, b in mats[:-1]:
                hdn = torch.addmm(b, hdn, A).relu_()
            z = torch.addmm(mats[-1][1], hdn, mats[-1][0])
            v = torch.cat([torch.nn.functional.softplus(z[:, :1], threshold=100.0), torch.sigmoid(z[:, 1:])], 1)
            outf[ids] = v.view(-1, STEPS, 4)
        at += c
    T = torch.ones(n, device=o.device, dtype=torch.float64)
    rgb, depth = torch.zeros((n, 3), device=o.device, dtype=torch.float64), torch.zeros_like(T)
    hist = torch.zeros((n, PO), device=o.device, dtype=torch.float64) if bins else None
    bw = torch.where(r1 > r0, (r1 - r0) / 64, torch.ones_like(r0))
    for k in range(maxc):
        live = nt[:, k] >= 0
        for s in range(STEPS):
            act = live & (T >= T_TERM)
            e = torch.exp(-out[:, k, s, 0] * delta[:, k])
            wgt = torch.where(act, T * (1.0 - e), torch.zeros_like(T))
            rgb += wgt[:, None] * out[:, k, s, 1:]
            depth += wgt * t[:, k, s]
            if bins:
                b = torch.floor((t[:, k, s] - r0) / bw).long().clamp_(0, 63)
                hist.scatter_add_(1, b[:, None], wgt[:, None])
            T = torch.where(act, T * e, T)
    if bins:
        hist[:, 64] = T
        root = torch.where(r1 > r0, r0, torch.zeros_like(r0))
        return rgb, hist, root, o, d, grid
    return rgb, depth, 1.0 - T


def _train64(case, seed):
    rgb, targets, t0, o, d, grid = _render64(case, seed, bins=True)
    P = _proposal_fit(case, seed, grid).double()
    m, v = torch.zeros_like(P), torch.zeros_like(P)
    n, losses = o.shape[0], []
    for s in range(1, case["train_steps"] + 1):
        with np.errstate(over="ignore"):
            i = np.arange(case["batch"], dtype=np.uint64)
            z = np.uint64(seed + 1) + np.uint64(0x9E3779B97F4A7C15) * (np.uint64(s) * np.uint64(0x100000001) + i
                                                                       + np.uint64(1))
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z ^= z >> np.uint64(31)
        r = torch.as_tensor((z % np.uint64(n)).astype(np.int64), device=o.device)
        p = P.clone().requires_grad_(True)
        q = _prop_predict(p, o[r], d[r], t0[r][:, None])
        tg = targets[r]
        loss = -(torch.where(tg > 0, tg * torch.log(q.clamp_min(1e-300)), torch.zeros_like(tg))).sum(1).mean()
        g, = torch.autograd.grad(loss, p)
        losses.append(loss.detach())
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        P = P - 3e-3 * (m / (1 - 0.9 ** s)) / ((v / (1 - 0.999 ** s)).sqrt() + 1e-8)
    return rgb, targets, torch.stack(losses), P, m, v


def exact(case, seed):
    # over about 200 M samples the double-precision networks would take more than 20 seconds
    if case["w"] * case["h"] * case["views"] * (70 if case["scene"] != "c1" else 17) > 2.0e8:
        return None
    if case["kind"] == "train":
        # the targets have no such value: samples of rays inside one leaf lie on the edges of the
        # depth bins, and rounding says on which side
        rgb, _, *rest = _train64(case, seed)
        return (rgb, None, *rest)
    return _render64(case, seed)
