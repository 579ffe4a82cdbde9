"""The default shape's choices for chains shorter than a tile and for launches of a few steps: the line
and the observables are those of the default shape given explicitly."""
import numpy as np
import pytest

from qew_workloads import NONE, RB, RBG_CUBIC, RBG_LINEAR, RF, SEED

pytestmark = pytest.mark.gpu
F = {RF: 0.9, RB: 1.1, NONE: 0.3, RBG_LINEAR: 1.6, RBG_CUBIC: 2.0}


def both(L, f, kind, given, calls):
    import paper_1211_7275_gb300 as qew
    outs = []
    for shape in (None, given):
        with qew.Relaxation(L, f, kind, dt=0.1, seed=SEED) as r:
            if shape:
                r.set_tuning(*shape)
            obs = r.observe([0, 3, 20, 90])
            for n in calls:
                r.advance(n)
            outs.append((obs, r.state()[0], r.tuning()))
    (a, ua, ta), (b, ub, tb) = outs
    assert ta == tb
    assert np.array_equal(ua, ub)
    for k in ("v", "ubar", "w2"):   # one FP64 rounding of sums relative to another integer cell
        np.testing.assert_allclose(a[k], b[k], rtol=1e-13, atol=1e-13)


def given(kind):
    return (224, 16, 2) if kind in (RB, RBG_CUBIC) else (736, 16, 2)


@pytest.mark.parametrize("kind", [RF, RB, NONE, RBG_LINEAR, RBG_CUBIC])
@pytest.mark.parametrize("L", [np.full(12000, 100), np.full(3000, 150), np.full(700, 192), np.full(4000, 300), np.full(900, 1025),
                               np.arange(1, 1500)], ids=["100", "150", "192", "300", "1025", "uneven"])
def test_short_chains(kind, L):
    both(L, F[kind], kind, given(kind), [48, 100])


@pytest.mark.parametrize("kind", [RF, RB, NONE, RBG_LINEAR, RBG_CUBIC])
@pytest.mark.parametrize("L", [(1 << 17) - 1, 1 << 17, 1 << 18, 3 << 18, (1 << 20) + 5, 1 << 21])
def test_launches_of_a_few_steps(kind, L):
    both([L], F[kind], kind, given(kind), [1, 2, 3, 4, 15, 16, 17, 5])


def test_short_launches_of_a_mixed_batch():
    L = np.array([3000, 400097, 777, 250025, 20480, 250001])
    kind = np.array([RF, RB, NONE, RBG_LINEAR, RBG_CUBIC, RF], dtype=np.int32)
    f = np.array([F[k] for k in kind]) * np.array([1, -1, 1, -1, 1, 1])
    both(L, f, kind, (224, 16, 2), [1, 2, 3, 16, 17])
