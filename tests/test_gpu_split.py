"""FP32 networks on the tensor cores (split BF16 operands) at the sizes where their tiling can
go wrong: one crossing, partly filled tiles, leaf changes inside a CTA's range, every number of
hidden layers, samples per crossing from 1 to 32, and the shapes that stay on the SIMT kernel
(other encodings, weights beyond the shared memory).  Against the FP32-mode oracle at the FP32
path's 1e-5; and the network outputs themselves against 64 bits: an FP32 chain of K products
rounds K times, so a layer's error is within K 2^-24 of the sum of its products' magnitudes,
which Xavier weights keep below 16 per layer: 90 x 2^-24 x 16 < 1e-4 bounds five layers' first
order with room for their propagation (the split's own error is measured far below that)."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2310_01881_gb300 import scenes as S
from pixtol import check_pixels

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_2310_01881_gb300 import amnerf, build
    build.build()
    r = amnerf.Renderer(0)
    yield r
    r.close()


@pytest.mark.parametrize("width,hidden,lx,ld", [(32, 1, 10, 4), (32, 2, 10, 4), (32, 8, 10, 4), (64, 1, 10, 4),
                                                (64, 2, 10, 4), (64, 4, 10, 4), (64, 7, 10, 4), (64, 2, 6, 2)])
def test_split_networks_against_the_oracle(R, width, hidden, lx, ld):
    cfg = dataclasses.replace(S.CONFIGS["c1"], width=width, hidden=hidden, lx=lx, ld=ld)
    grid = S.density_grid(S.scene_for(cfg.scene, 2), cfg.G)
    tree = O.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac)
    assert R.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac) == tree.n_leaves
    P = S.with_biases(S.xavier_weights(2, S.leaf_mean_density(grid, tree.leaf_cells()), width, hidden, lx, ld),
                      2, width, hidden, lx, ld)
    R.load_mlps(P, width, hidden, lx, ld, "fp32")
    o, d = S.view_rays(cfg, 2, 0)
    for lo, n, steps, cap, jitter in ((2016, 1, 8, 64, 0), (2016, 17, 8, 64, 5), (0, 4096, 8, 64, 0), (1500, 700, 1, 24, 0),
                                      (1500, 700, 32, 96, 0), (1900, 300, 4, 30, 9)):
        oo, dd = o[lo:lo + n], d[lo:lo + n]
        got = [t.cpu().numpy() for t in R.render(torch.from_numpy(oo).cuda(), torch.from_numpy(dd).cuda(),
                                                 steps=steps, cap=cap, jitter=jitter)]
        R.sync()
        ref = O.render(tree, P, width, hidden, lx, ld, oo, dd, steps, cap, mode=1, jitter=jitter, threads=8)
        check_pixels(list(zip(got, (ref["rgb"], ref["depth"], ref["opacity"]))), ref["ert_margin"],
                     f"{hidden} x {width} n {n} steps {steps}")


def test_split_network_outputs_against_64_bits(R):
    width, hidden = 64, 4
    cfg = S.CONFIGS["c2"]
    grid = S.density_grid(S.scene_for(cfg.scene, 1), cfg.G)
    R.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac)
    P = S.xavier_weights(1, S.leaf_mean_density(grid, R.leaf_cells()), width, hidden, cfg.lx, cfg.ld)
    P = S.with_biases(P, 1, width, hidden, cfg.lx, cfg.ld)
    R.load_mlps(P, width, hidden, cfg.lx, cfg.ld, "fp32")
    o, d = S.view_rays(cfg, 1, 0, 40, 40)
    _, _, _, dbg, _ = R.render_debug(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), 8, cfg.cap)
    ray, k = np.nonzero(np.arange(cfg.cap // 8)[None] < dbg["n_x"].astype(int)[:, None])
    f = np.float32
    t_in, t_out = dbg["t_in"][ray, k][:, None], dbg["t_out"][ray, k][:, None]
    t = t_in + (np.arange(8, dtype=f) + f(0.5)) * ((t_out - t_in) * f(0.125))
    x = (o[ray][:, None] + t[..., None] * d[ray][:, None]).astype(np.float64).reshape(-1, 3)
    dd = np.repeat(d[ray].astype(np.float64), 8, 0)

    def gamma(p, L):
        out = [p]
        for i in range(L):
            v = np.remainder(p * 2.0 ** i, 2.0)  # exact
            out += [np.sin(np.pi * v), np.cos(np.pi * v)]
        return np.concatenate(out, 1)

    feat, net = np.concatenate([gamma(x, cfg.lx), gamma(dd, cfg.ld)], 1), np.repeat(dbg["leaf"][ray, k], 8)
    W = P.reshape(R.n_leaves, -1).astype(np.float64)
    want = np.empty((len(net), 4))
    for m in np.unique(net):
        h, at, rows = feat[net == m], 0, net == m
        for fo, fi in [(width, 90)] + [(width, width)] * (hidden - 1) + [(4, width)]:
            h = h @ W[m, at:at + fo * fi].reshape(fo, fi).T + W[m, at + fo * fi:at + fo * fi + fo]
            at += fo * fi + fo
            h = np.maximum(h, 0.0) if fo != 4 else h
        want[rows] = np.concatenate([np.logaddexp(0.0, h[:, :1]), 1.0 / (1.0 + np.exp(-h[:, 1:]))], 1)
    got = dbg["slot_out"][ray[:, None], 8 * k[:, None] + np.arange(8)].reshape(-1, 4)
    err = np.abs(got - want) / np.maximum(np.abs(want), 1.0)
    print(f"network outputs: max error {err.max():.2e}, rms {np.sqrt((err ** 2).mean()):.2e}")
    assert err.max() < 1e-4


@pytest.mark.parametrize("width,hidden", [(32, 1), (32, 2), (64, 4)])
def test_split_networks_overflow_as_fp32_does(R, width, hidden):
    """Weights beyond the largest BF16 and activations that overflow FP32: an infinite density is
    opaque and infinite logits saturate, as in the oracle (no NaN from the split)."""
    cfg = dataclasses.replace(S.CONFIGS["c1"], width=width, hidden=hidden)
    grid = S.density_grid(S.scene_for(cfg.scene, 2), cfg.G)
    tree = O.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac)
    R.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac)
    parts = [np.zeros(width * 90), np.full(width, 3.4e38)]
    for _ in range(hidden - 1):
        parts += [np.full(width * width, 0.5), np.zeros(width)]
    parts += [np.repeat([0.1, 0.1, -0.1, -0.2], width), np.zeros(4)]
    P = np.tile(np.concatenate(parts).astype(np.float32), (tree.n_leaves, 1))
    R.load_mlps(P, width, hidden, cfg.lx, cfg.ld, "fp32")
    o, d = S.view_rays(cfg, 2, 0)
    o, d = o[1500:2200], d[1500:2200]
    got = [t.cpu().numpy() for t in R.render(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), steps=8, cap=64)]
    R.sync()
    ref = O.render(tree, P, width, hidden, cfg.lx, cfg.ld, o, d, 8, 64, mode=1, threads=8)
    assert ref["opacity"].max() == 1.0 and np.isfinite(ref["rgb"]).all()
    for name, a in zip(("rgb", "depth", "opacity"), got):
        assert np.abs(a - ref[name]).max() <= 1e-5, name
