"""Tile pipeline of the tensor-core network: few and odd numbers of tiles per worker, partly
filled tiles, every number of hidden layers and samples per crossing, and all schedules.
The two BF16 kernels (one and two threads per sample row) share no pipeline, so their equal
pixels check both; E4M3 has one kernel, checked across launch configurations that give its
workers different tiles."""
import numpy as np
import pytest

from paper_2310_01881_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_2310_01881_gb300 import amnerf, build
    build.build()
    r = amnerf.Renderer(0)
    yield r
    r.close()


def _render(R, A, rays, tuning, **kw):
    A.amnerf_set_tuning(R.ctx, *tuning)
    out = [t.cpu().numpy() for t in R.render(*rays, **kw)]
    R.sync()
    return out


@pytest.mark.parametrize("prec", ["bf16", "fp8", "fp8s"])
@pytest.mark.parametrize("width,hidden", [(32, 1), (32, 2), (64, 1), (64, 2), (64, 3), (64, 4), (64, 5), (64, 8)])
def test_configurations_give_identical_pixels(R, prec, width, hidden):
    from paper_2310_01881_gb300 import amnerf as A
    cfg = S.CONFIGS["c1"]
    grid = S.density_grid(S.scene_for(cfg.scene, 1), cfg.G)
    R.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac)
    P = S.with_biases(S.xavier_weights(1, S.leaf_mean_density(grid, R.leaf_cells()), width, hidden, cfg.lx, cfg.ld),
                      1, width, hidden, cfg.lx, cfg.ld)
    rays = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in S.view_rays(cfg, 1, 0)]
    if prec == "fp8s":
        R.load_mlps(P, width, hidden, cfg.lx, cfg.ld, act_max=np.full((R.n_leaves, hidden), 2.0, np.float32))
    else:
        R.load_mlps(P, width, hidden, cfg.lx, cfg.ld, prec)
    other = [(0, 0, 2), (3, 1, 2)] if prec == "bf16" else [(1, 0, 1)]
    try:
        for n in (1, 17, 129, 4096):
            part = [r[:n].contiguous() for r in rays] if n > 17 else [r[2016:2016 + n].contiguous() for r in rays]
            for steps, cap in ((8, 64), (1, 24), (4, 30), (32, 96)):
                kw = dict(steps=steps, cap=cap, jitter=7 if n == 129 else 0)
                want = _render(R, A, part, other[0], **kw)
                for tuning in other[1:] + [(0, 0, 1), (1, 0, 1), (2, 1, 1), (0, 2, 1)]:
                    for a, b in zip(_render(R, A, part, tuning, **kw), want):
                        np.testing.assert_array_equal(a, b, err_msg=f"n {n} steps {steps} tuning {tuning}")
    finally:
        A.amnerf_set_tuning(R.ctx, 0, 0, 0)


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8", "fp8s"])
@pytest.mark.parametrize("width,hidden", [(32, 1), (64, 1), (32, 2)])
def test_shallow_networks_over_many_tiles(R, prec, width, hidden):
    """A hundred tiles and more per worker with one or two hidden layers, where the staging of
    the next tiles' crossings has the least slack: every wait is met (no timeout in the status
    word) and a second render gives the same pixels."""
    cfg = S.CONFIGS["c1"]
    grid = S.density_grid(S.scene_for(cfg.scene, 1), cfg.G)
    R.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac)
    P = S.xavier_weights(1, S.leaf_mean_density(grid, R.leaf_cells()), width, hidden, cfg.lx, cfg.ld)
    act = np.full((R.n_leaves, hidden), 2.0, np.float32) if prec == "fp8s" else None
    R.load_mlps(P, width, hidden, cfg.lx, cfg.ld, "fp8" if act is not None else prec, act_max=act)
    rays = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in S.view_rays(cfg, 1, 0, 800, 700)]
    first = [t.clone() for t in R.render(*rays, steps=8, cap=64)]
    R.sync()
    for a, b in zip(R.render(*rays, steps=8, cap=64), first):
        assert torch.equal(a, b)
    R.sync()
