"""What is loaded from host memory is on the device, in the context's stream, before a render can
read it: a plain cudaMemcpy or cudaMemset works on the legacy stream, may return before it has
run, and a context on a non-blocking stream (every stream torch hands out but the default one)
does not wait for it."""
import os
import re

import numpy as np
import pytest

import oracle as O
from paper_2310_01881_gb300 import scenes as S
from paper_2310_01881_gb300.build import CSRC

torch = pytest.importorskip("torch")


def test_no_upload_or_memset_on_the_legacy_stream():
    for name in sorted(os.listdir(CSRC)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        calls = re.findall(r"cuda(?:Memcpy|Memset)(?:2D|3D)?\s*\([^;]*;", src)
        assert not [c for c in calls if "DeviceToHost" not in c], name


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
def test_loads_beside_a_busy_default_stream(prec):
    from paper_2310_01881_gb300 import amnerf as A, build
    build.build()
    cfg = S.CONFIGS["c1"]
    grid = S.density_grid(S.scene_for("c1", 0), cfg.G)
    tree = O.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac)
    P = S.xavier_weights(0, S.leaf_mean_density(grid, tree.leaf_cells()), cfg.width, cfg.hidden, cfg.lx, cfg.ld)
    o, d = (torch.from_numpy(a).cuda() for a in S.view_rays(cfg, 0, 0))
    prop = S.proposal_init(3)
    out = {}
    for busy in (False, True):
        side = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            r = A.Renderer(0)
        try:
            if busy:
                torch.cuda._sleep(400_000_000)  # about 0.2 s of the default stream
            with torch.cuda.stream(side):
                r.build_tree(grid, cfg.max_depth, cfg.leaf_mass_frac)
                r.load_mlps(P, cfg.width, cfg.hidden, cfg.lx, cfg.ld, prec)
                A.amnerf_proposal_set(r.ctx, prop)
                frames = r.render(o, d, proposal=True, coverage=0.9) + r.render(o, d)
                side.synchronize()
                out[busy] = [t.cpu().numpy() for t in frames] + list(A.amnerf_proposal_get(r.ctx)[:3])
                r.sync()
        finally:
            torch.cuda.synchronize()
            r.close()
    for a, b in zip(out[False], out[True]):
        np.testing.assert_array_equal(a, b)
