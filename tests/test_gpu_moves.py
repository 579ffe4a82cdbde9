"""Moves of the fused kernel in both directions and of any length: lines driven up and down from below
the threshold to where sites move by two cells a step.  A cache that a move left wrong shows in the next
forces, so that the line relaxed on is compared, bit for bit, with one whose caches are drawn afresh
from its state; and the forces of the fresh caches with the oracle's."""
import numpy as np
import pytest

import oracle
from qew_workloads import RB, RBG_CUBIC, RBG_LINEAR, RF, SEED

pytestmark = pytest.mark.gpu
F_C = {RF: 0.72057, RB: 0.90749, RBG_LINEAR: 1.5652, RBG_CUBIC: 1.9475}
L = np.array([1537, 100, 4096, 1, 449])


@pytest.fixture(scope="module")
def qew():
    import paper_1211_7275_gb300 as q
    return q


@pytest.mark.parametrize("kind", [RF, RB, RBG_LINEAR, RBG_CUBIC])
@pytest.mark.parametrize("drive", [0.6, 1.5, 3.0, 8.0, 40.0])
@pytest.mark.parametrize("shape", [None, (224, 16, 2), (480, 32, 1), (992, 32, 2), (1248, 16, 1)])
def test_caches_after_moves(qew, kind, drive, shape):
    """Drives of both signs, and none, in one batch."""
    f = F_C[kind] * drive * np.array([1.0, -1.0, -1.0, 1.0, 0.0])
    rng = np.random.default_rng(7)
    u0 = np.concatenate([0.8 * rng.standard_normal(n) for n in L])
    with qew.Relaxation(L, f, kind, dt=0.1, seed=SEED) as r, qew.Relaxation(L, f, kind, dt=0.1, seed=SEED) as fresh:
        if shape:
            r.set_tuning(*shape)
        for start in (None, u0):
            if start is None:
                r.reset()
            else:
                r.set_state(start)
            for _ in range(3):
                r.advance(23)
                u, _ = r.state()
                assert np.array_equal(r.cells(), np.floor(u).astype(np.int32))
                fresh.set_state(u)
                r.advance(5)
                fresh.advance(5)
                assert np.array_equal(r.state()[0], fresh.state()[0])


@pytest.mark.parametrize("kind", [RF, RB, RBG_LINEAR, RBG_CUBIC])
@pytest.mark.parametrize("sign", [1.0, -1.0, 0.0])
def test_forces_of_fresh_caches(qew, kind, sign):
    """v and u after one step, from lines far from a cell's edge: one FP32 rounding of each operation."""
    rng = np.random.default_rng(11)
    u0 = rng.integers(-3, 4, L.sum()) + rng.uniform(0.1, 0.9, L.sum())
    f = sign * F_C[kind]
    ref = oracle.run(L, f, 0.1, kind, SEED, np.array([0, 1]), u0=u0, want_state=True)
    with qew.Relaxation(L, f, kind, dt=0.1, seed=SEED) as r:
        r.set_state(u0)
        obs = r.observe([0, 1])
        u, _ = r.state()
    np.testing.assert_allclose(u, ref["u"], atol=2e-6)
    np.testing.assert_allclose(obs["v"][0], ref["v"][0], atol=2e-5)


@pytest.mark.parametrize("kind", [RF, RB, RBG_LINEAR, RBG_CUBIC])
@pytest.mark.parametrize("sites", [(3 << 20) - 64, 3 << 20])
def test_signs_in_one_launch_and_in_two(qew, kind, sites):
    """A chain of either sign beside others, below and above the size from which each sign has a launch of
    its own, against the same chain alone."""
    n = np.array([5000, 7001])
    f = F_C[kind] * np.array([1.5, -1.5])
    lines = []
    with qew.Relaxation(np.append(n, sites - n.sum()), np.append(f, -f[0]), kind, dt=0.1, seed=SEED) as r:
        r.advance(60)
        lines.append(r.state()[0][:n.sum()])
    alone = []
    for c in range(2):
        with qew.Relaxation([n[c]], f[c], kind, dt=0.1, seed=SEED) as r:
            r.set_samples([c])
            r.advance(60)
            alone.append(r.state()[0])
    assert np.array_equal(lines[0], np.concatenate(alone))
