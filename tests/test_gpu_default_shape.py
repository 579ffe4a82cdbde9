"""A handle in its default shape runs the launches between observations in a shape of their own,
chosen by the number of sites: the line and the observables are those of the default shape given
explicitly, below and above each size where the choice changes."""
import numpy as np
import pytest

from qew_workloads import NONE, RB, RBG_CUBIC, RBG_LINEAR, RF, SEED

pytestmark = pytest.mark.gpu
F = {RF: 0.9, RB: 1.1, NONE: 0.3, RBG_LINEAR: 1.6, RBG_CUBIC: 2.0}
# no steps between two observations, fewer than a launch holds, whole launches, one more, many
STEPS = [0, 1, 15, 16, 17, 33, 34, 130, 131, 400]


@pytest.fixture(scope="module")
def qew():
    import paper_1211_7275_gb300 as q
    return q


def both(qew, L, f, kind, given):
    outs = []
    for shape in (None, given):
        with qew.Relaxation(L, f, kind, dt=0.1, seed=SEED) as r:
            if shape:
                r.set_tuning(*shape)
            obs = r.observe(STEPS)
            r.advance(77)
            outs.append((obs, r.state()[0], r.tuning()))
    (a, ua, ta), (b, ub, tb) = outs
    assert ta == tb
    assert np.array_equal(ua, ub)
    for k in ("v", "ubar", "w2"):   # one FP64 rounding of sums relative to another integer cell
        np.testing.assert_allclose(a[k], b[k], rtol=1e-13, atol=1e-13)


@pytest.mark.parametrize("kind", [RF, RB, NONE, RBG_LINEAR, RBG_CUBIC])
@pytest.mark.parametrize("L", [[1, 129, 777, 5000], [3 << 15], [(3 << 16) - 1], [(3 << 16)], [3 << 17], [(3 << 18) - 1, 1], [(3 << 19) + 5]])
def test_default_shape_equals_the_same_shape_given(qew, kind, L):
    given = (224, 16, 2) if kind in (RB, RBG_CUBIC) else (736, 16, 2)
    both(qew, np.array(L), F[kind], kind, given)


def test_mixed_batch(qew):
    L = np.array([3000, 4097, 777, 5025, 2048, 250001])
    kind = np.array([RF, RB, NONE, RBG_LINEAR, RBG_CUBIC, RF], dtype=np.int32)
    both(qew, L, np.array([F[k] for k in kind]), kind, (224, 16, 2))
