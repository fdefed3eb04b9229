"""How accurate the split FP32 networks (tensor cores) are, held to what FP32 arithmetic gives.

A layer takes six of the nine partial products of its operands' three BF16 parts; the smallest
taken (m m, h l, l h) are up to 2^-16 of a product.  The CPU test restates that composition in
numpy (exact partial sums, accumulators cut to 24 bits) and finds, against 64 bits, an error
below that of the FP32-mode oracle's chain on the same samples, and one of at least six times it
when any one of those three products is left out.  So three times the chain's error, between
the two, is the bound of the GPU test: it holds for the kernel, whose own
sine, exponential and logarithm add up to a rounding each, and fails when a product or a
part's offset is wrong."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2310_01881_gb300 import scenes as S

FACTOR = 3.0
SHAPES = [(64, 1), (64, 2), (64, 4), (64, 7), (32, 2), (32, 8)]
SMALL = [(1, 1), (2, 0), (0, 2)]  # m m, l h, h l
f32 = np.float32


def _bf16(x):
    u = np.ascontiguousarray(x, f32).view(np.uint32)
    return ((u + ((u >> 16) & 1) + 0x7fff) & 0xffff0000).astype(np.uint32).view(f32)


def _split(v):
    v = np.asarray(v, f32)
    h = _bf16(v)
    m = _bf16(v - h)
    return [p.astype(np.float64) for p in (h, m, _bf16(v - h - m))]


def _cut(x):
    m, e = np.frexp(x)
    return np.ldexp(np.trunc(m * 2.0 ** 24), e - 24)


def _gamma(p, L):
    out = [p.astype(np.float64)]
    for i in range(L):
        v = np.remainder(out[0] * 2.0 ** i, 2.0)  # exact
        out += [np.sin(np.pi * v), np.cos(np.pi * v)]
    return np.concatenate(out, 1).astype(f32)


def _six_products(P, width, hidden, x, d, without=None):
    a = np.concatenate([_gamma(x, 10), _gamma(d, 4)], 1)
    at = 0
    for fo, fi in [(width, 90)] + [(width, width)] * (hidden - 1) + [(4, width)]:
        A, W, b = _split(a), _split(P[at:at + fo * fi].reshape(fo, fi)), P[at + fo * fi:at + fo * fi + fo]
        at += fo * fi + fo
        acc = np.zeros((len(a), fo))
        for p, q in SMALL + [(1, 0), (0, 1)]:
            if (p, q) != without:
                for s in range(0, fi, 16):
                    acc = _cut(acc + A[p][:, s:s + 16] @ W[q][:, s:s + 16].T)
        if fo != 4:
            acc = _cut(acc + b)
        for s in range(0, fi, 16):
            acc = _cut(acc + A[0][:, s:s + 16] @ W[0][:, s:s + 16].T)
        a = np.maximum(acc, 0.0).astype(f32)
    z = (acc.astype(f32) + b).astype(np.float64)
    out = np.concatenate([np.logaddexp(0.0, z[:, :1]), 1.0 / (1.0 + np.exp(-z[:, 1:]))], 1)
    return out.astype(f32).astype(np.float64)


def _rms(got, want):
    return np.sqrt(np.mean(((got - want) / np.maximum(np.abs(want), 1.0)) ** 2))


@pytest.mark.parametrize("width,hidden", SHAPES)
def test_the_bound_lies_between_fp32_and_an_omitted_product(width, hidden):
    rng = np.random.default_rng(100 * width + hidden)
    e = {k: [] for k in ("chain", "six", *SMALL)}
    for net in range(6):
        P = np.concatenate([np.concatenate([rng.uniform(-1, 1, fo * fi) * np.sqrt(6 / (fi + fo)), rng.uniform(-0.1, 0.1, fo)])
                            for fo, fi in [(width, 90)] + [(width, width)] * (hidden - 1) + [(4, width)]]).astype(f32)
        x = rng.uniform(-1, 1, (1500, 3)).astype(f32)
        d = rng.normal(size=(1500, 3))
        d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(f32)
        want, chain = (O.mlp_eval(P, width, hidden, 10, 4, x, d, mode)[0] for mode in (0, 1))
        e["chain"].append(_rms(chain, want))
        e["six"].append(_rms(_six_products(P, width, hidden, x, d), want))
        if net < 2:
            for p in SMALL:
                e[p].append(_rms(_six_products(P, width, hidden, x, d, p), want))
    r = {k: np.mean(v) / np.mean(e["chain"]) for k, v in e.items()}
    print({str(k): round(float(v), 2) for k, v in r.items()})
    assert r["six"] <= 1.0
    assert min(r[p] for p in SMALL) >= 2.0 * FACTOR


@pytest.mark.gpu
@pytest.mark.parametrize("width,hidden", SHAPES)
def test_split_networks_are_as_accurate_as_fp32(width, hidden):
    torch = pytest.importorskip("torch")
    from paper_2310_01881_gb300 import amnerf, build
    build.build()
    cfg = dataclasses.replace(S.CONFIGS["c1"], width=width, hidden=hidden)
    grid = S.density_grid(S.scene_for(cfg.scene, 1), cfg.G)
    steps, cap = 8, 64
    R = amnerf.Renderer(0)
    try:
        n = R.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac)
        P = S.xavier_weights(1, S.leaf_mean_density(grid, R.leaf_cells()), width, hidden, cfg.lx, cfg.ld)
        P = S.with_biases(P, 1, width, hidden, cfg.lx, cfg.ld).reshape(n, -1)
        R.load_mlps(P, width, hidden, cfg.lx, cfg.ld, "fp32")
        o, d = S.view_rays(cfg, 1, 0, 40, 40)
        *_, dbg, _ = R.render_debug(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), steps, cap)
        R.sync()
    finally:
        R.close()
    n_x = dbg["n_x"].astype(int)
    x = O.samples(o, d, n_x, dbg["t_in"], dbg["t_out"], cap // steps, steps, cap, mode=1)[2]
    ray, k = np.nonzero(np.arange(cap // steps)[None] < n_x[:, None])
    slot = steps * k[:, None] + np.arange(steps)
    got, x = dbg["slot_out"][ray[:, None], slot].reshape(-1, 4), x[ray[:, None], slot].reshape(-1, 3)
    dd, net = np.repeat(d[ray], steps, 0), np.repeat(dbg["leaf"][ray, k], steps)
    want, chain = np.empty((len(net), 4)), np.empty((len(net), 4))
    for m in np.unique(net):
        i = net == m
        want[i], chain[i] = (O.mlp_eval(P[m], width, hidden, 10, 4, x[i], dd[i], mode)[0] for mode in (0, 1))
    split, ref = _rms(got, want), _rms(chain, want)
    print(f"{hidden} x {width}: split {split:.2e}, FP32 chain {ref:.2e}, ratio {split / ref:.2f}")
    assert split <= FACTOR * ref
