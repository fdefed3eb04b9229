"""FP32 networks whose activations overflow, on the tensor cores (split operands): what a network
gives is what FP32 arithmetic gives.  Two families, whose FP32 results do not depend on the
order of a sum, so that they are compared exactly (infinities, NaN) or at the FP32 path's 1e-5
with the FP32-mode oracle, sample by sample:

  signs      layer 1 overflows to infinity; later layers meet infinities with weights of one
             sign (an infinity, or below it zero) or of both (NaN, which ReLU makes 0), also
             with weights far below one and below 1e-37
  positions  an infinity in some samples only (those with x above 0.567), next to weights that
             are zero: 0 x inf is NaN, ReLU makes it 0, and the head gives its bias alone;
             every other sample is an ordinary one
"""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2310_01881_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FMAX = np.float64(np.finfo(np.float32).max)


@pytest.fixture(scope="module")
def R():
    from paper_2310_01881_gb300 import amnerf, build
    build.build()
    r = amnerf.Renderer(0)
    yield r
    r.close()


def _scene(width, hidden):
    cfg = dataclasses.replace(S.CONFIGS["c1"], width=width, hidden=hidden)
    grid = S.density_grid(S.scene_for(cfg.scene, 2), cfg.G)
    return cfg, grid, O.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac)


def _slots(R, cfg, grid, P, o, d, steps, cap, jitter):
    """(samples' slot values, positions, directions, networks) of a render."""
    R.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac)
    R.load_mlps(P, cfg.width, cfg.hidden, cfg.lx, cfg.ld, "fp32")
    *_, dbg, _ = R.render_debug(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), steps, cap, jitter=jitter)
    R.sync()
    maxc, n_x = cap // steps, dbg["n_x"].astype(int)
    _, _, x = O.samples(o, d, n_x, dbg["t_in"], dbg["t_out"], maxc, steps, cap, mode=1, jitter=jitter)
    ray, k = np.nonzero(np.arange(maxc)[None] < n_x[:, None])
    slot = steps * k[:, None] + np.arange(steps)
    got = dbg["slot_out"][ray[:, None], slot].reshape(-1, 4)
    return got, x[ray[:, None], slot].reshape(-1, 3), np.repeat(d[ray], steps, 0), np.repeat(dbg["leaf"][ray, k], steps)


def _want(cfg, P, x, d, net):
    out = np.empty((len(net), 4))
    for m in np.unique(net):
        out[net == m] = O.mlp_eval(P[m], cfg.width, cfg.hidden, cfg.lx, cfg.ld, x[net == m], d[net == m], mode=1)[0]
    return out


def _agree(got, want):
    finite = np.isfinite(want)
    np.testing.assert_array_equal(got[~finite], want[~finite])  # NaN where NaN, infinity where infinity
    assert np.isfinite(got[finite]).all()
    err = np.abs(got[finite] - want[finite]) / np.maximum(np.abs(want[finite]), 1.0)
    assert err.max(initial=0.0) <= 1e-5
    return finite


@pytest.mark.parametrize("width,hidden", [(32, 2), (32, 3), (32, 8), (64, 2), (64, 4), (64, 7)])
def test_infinite_activations_and_weights_of_either_sign(R, width, hidden):
    cfg, grid, tree = _scene(width, hidden)
    rng = np.random.default_rng(width + hidden)
    nets = []
    for _ in range(tree.n_leaves):
        parts = [np.zeros(width * 90), np.where(rng.random(width) < 0.5, 3.0e38, 0.0)]
        for l in range(1, hidden):
            # of one sign; from the third layer on some rows of both
            w = rng.uniform(1.0, 2.0, (width, width)) * rng.choice([1.0, 1.0, -1.0], (width, 1))
            if l > 1:
                w *= rng.choice([1.0, 0.1, 1e-3, 1e-38], (width, 1))
                both = rng.random(width) < 0.3
                w[both] *= rng.choice([1.0, -1.0], (int(both.sum()), width))
            parts += [w.reshape(-1), np.zeros(width)]
        head = rng.uniform(1.0, 2.0, (4, width)) * rng.choice([1.0, 0.1, 1e-38], (4, 1))
        head *= rng.choice([1.0, -1.0], (4, 1))
        head[rng.random(4) < 0.4] *= rng.choice([1.0, -1.0], width)
        nets.append(np.concatenate(parts + [head.reshape(-1), np.zeros(4)]).astype(np.float32))
    P = np.stack(nets)
    o, d = S.view_rays(cfg, 2, 0)
    for lo, n, steps, cap, jitter in ((1500, 700, 8, 64, 0), (2016, 17, 8, 64, 5), (1800, 300, 1, 8, 0)):
        got, x, dd, net = _slots(R, cfg, grid, P, o[lo:lo + n], d[lo:lo + n], steps, cap, jitter)
        want = _want(cfg, P, x, dd, net)
        finite = _agree(got, want)
        assert n < 700 or (np.isnan(want).any() and np.isinf(want).any() and finite.any())


@pytest.mark.parametrize("width,hidden", [(32, 2), (32, 4), (64, 3), (64, 4)])
def test_infinite_activations_of_some_samples(R, width, hidden):
    cfg, grid, tree = _scene(width, hidden)
    P = S.xavier_weights(2, S.leaf_mean_density(grid, tree.leaf_cells()), width, hidden, cfg.lx, cfg.ld)
    P = S.with_biases(P, 2, width, hidden, cfg.lx, cfg.ld).reshape(tree.n_leaves, -1).copy()
    # neuron 0: 3e38 x, doubled by layer 1, and nothing else reads either
    P[:, :90] = 0.0
    P[:, 0] = 3.0e38
    P[:, width * 90] = 0.0
    at = width * 90 + width
    for l in range(1, hidden):
        w = P[:, at:at + width * width].reshape(-1, width, width)
        w[:, :, 0] = 0.0
        if l == 1:
            w[:, 0, :] = 0.0
            w[:, 0, 0] = 2.0
            P[:, at + width * width] = 0.0
        P[:, at:at + width * width] = w.reshape(tree.n_leaves, -1)
        at += width * width + width
    P[:, at:at + 4 * width].reshape(-1, 4, width)[:, :, 0] = 0.0
    head = P[:, at:at + 4 * width].reshape(-1, 4, width).copy()
    head[:, :, 0] = 0.0
    P[:, at:at + 4 * width] = head.reshape(tree.n_leaves, -1)
    o, d = S.view_rays(cfg, 2, 0)
    # every sample's distance from the threshold is over a rounding: 3e38 (x + 1e-6) cannot
    # change side for the samples kept here
    for lo, n, steps, cap, jitter in ((0, 4096, 8, 64, 0), (1500, 700, 8, 64, 5), (1500, 700, 1, 24, 0),
                                      (1500, 700, 32, 96, 3), (1900, 300, 4, 30, 9)):
        got, x, dd, net = _slots(R, cfg, grid, P, o[lo:lo + n], d[lo:lo + n], steps, cap, jitter)
        clear = np.abs(6.0e38 * x[:, 0] / FMAX - 1.0) > 1e-5
        want = _want(cfg, P, x, dd, net)
        _agree(got[clear], want[clear])
        inf = clear & (6.0e38 * x[:, 0] > FMAX)
        assert n < 1000 or (inf.sum() > 100 and (clear & ~inf).sum() > 100)
