"""The training step's gradient over batches that fill its 64-ray tiles and its CTAs unevenly:
one ray, one short of and one past a tile, one ray past a full round of its 304 CTAs, several
rounds.  Against the FP64 backward pass with the tolerance of the suite's gradient check; and
two runs of the same training agree bit for bit (its sums have a fixed order)."""
import numpy as np
import pytest

import oracle as O
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


def _batch(n):
    """Rays at the scene, entry distances, and targets of positive mass summing to 1."""
    rng = np.random.default_rng(n)
    o, d = S.view_rays(S.CONFIGS["c1"], 0, 1, 200, 200)
    i = rng.permutation(len(o))[:n]
    t0 = rng.uniform(1.5, 2.5, n).astype(np.float32)
    tg = rng.dirichlet(np.full(65, 0.2), n).astype(np.float32)
    return o[i], d[i], t0, tg


@pytest.mark.parametrize("n", [1, 63, 64, 65, 128, 304 * 64 + 1, 39000])
def test_gradient_over_uneven_tiles(R, n):
    from paper_2310_01881_gb300 import amnerf as A
    o, d, t0, tg = _batch(n)
    params = S.proposal_init(5)
    A.amnerf_proposal_set(R.ctx, params)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    loss, g = A.amnerf_proposal_grad(R.ctx, dev(o), dev(d), dev(np.stack([t0, t0 + 1], 1)), dev(tg))
    l_ref, g_ref = O.prop_loss_grad(params.astype(np.float64), o, d, t0.astype(np.float64), tg.astype(np.float64))
    assert loss == pytest.approx(l_ref, rel=1e-5)
    err = np.abs(g.astype(np.float64) - g_ref)
    assert np.linalg.norm(err) <= 1e-4 * np.linalg.norm(g_ref)


def test_training_repeats_bit_for_bit(R):
    from paper_2310_01881_gb300 import amnerf as A
    o, d, t0, tg = _batch(5000)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    args = (dev(o), dev(d), dev(np.stack([t0, t0 + 1], 1)), dev(tg))
    runs = []
    for _ in range(2):
        A.amnerf_proposal_set(R.ctx, S.proposal_init(6))
        losses = A.amnerf_proposal_train(R.ctx, *args, steps=12, batch=1000, lr=3e-3, seed=9)
        runs.append((losses, *A.amnerf_proposal_get(R.ctx)))
    for a, b in zip(*runs):
        np.testing.assert_array_equal(a, b)
