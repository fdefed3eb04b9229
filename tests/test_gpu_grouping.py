"""Grouping around the rule that takes small batches to one launch (every CTA scans the counts):
batches on both sides of its 300 CTAs of 256 rays, partly filled CTAs, crossing capacities that
are and are not a multiple of eight and beyond the per-ray scatter's 32, few networks and one
per node of a 1024-leaf tree; and the traversal's rays-per-warp rule (4, 8, 32) on the same
batches.  Counts and offsets exactly, segments as sets, against numpy on the crossing list; the
crossing lists of a batch and of the same rays in a larger batch are equal."""
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


@pytest.mark.parametrize("depth,lod,cap", [(4, 0.0, 64), (4, 0.0, 24), (10, 0.0, 192), (10, 0.15, 200), (10, 0.0, 264)])
def test_groups_of_small_and_large_batches(R, depth, lod, cap):
    cfg = S.CONFIGS["c1"]
    grid = S.density_grid(S.scene_for(cfg.scene, 4), cfg.G)
    leaves = R.build_tree(grid, depth, 0.0)
    nets = 2 * leaves - 1 if lod else leaves
    rng = np.random.default_rng(0)
    R.load_mlps(rng.normal(0, 0.1, nets * S.params_per_leaf(32, 1, 10, 4)).astype(np.float32), 32, 1, 10, 4, "bf16")
    o, d = S.view_rays(cfg, 4, 0, 281, 275)  # 77 275 rays
    o, d = torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda()
    maxc = cap // 8
    full = None
    for n in (77275, 76801, 76800, 50001, 50000, 16001, 16000, 257, 1):
        _, _, _, dbg, st = R.render_debug(o[:n].contiguous(), d[:n].contiguous(), 8, cap, lod=lod)
        valid = np.arange(maxc)[None] < dbg["n_x"].astype(int)[:, None]
        leaf = dbg["leaf"][valid]
        counts = np.bincount(leaf, minlength=nets)
        np.testing.assert_array_equal(dbg["counts"], counts)
        np.testing.assert_array_equal(dbg["offsets"], np.concatenate([[0], np.cumsum(counts)]))
        assert st["crossings"] == counts.sum() and st["tiles"] == ((counts + 15) // 16).sum()
        order = dbg["order"][: counts.sum()]
        ids = np.flatnonzero(valid.reshape(-1))
        np.testing.assert_array_equal(np.sort(order), ids)
        np.testing.assert_array_equal(dbg["leaf"].reshape(-1)[order], np.repeat(np.arange(nets), counts))
        if full is None:
            full = dbg
        for key in ("n_x", "t_in", "t_out", "leaf"):
            a, b = dbg[key], full[key][:n]
            np.testing.assert_array_equal(a if key == "n_x" else a[valid], b if key == "n_x" else b[valid])
