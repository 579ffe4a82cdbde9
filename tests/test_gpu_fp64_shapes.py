"""The plain FP64 path at the sizes where its launch shape changes, against the oracle to the path's
1e-12: batches just below and above each line of the rule, chains shorter than a tile and of one site,
and a steep line whose sites move by many cells, up and down."""
import numpy as np
import pytest

import oracle
from qew_workloads import NONE, RB, RBG_CUBIC, RBG_LINEAR, RF, SEED

pytestmark = pytest.mark.gpu
KINDS = [RF, RB, NONE, RBG_LINEAR, RBG_CUBIC]
F = {RF: 0.9, RB: 1.1, NONE: 0.3, RBG_LINEAR: 1.6, RBG_CUBIC: 2.0}


@pytest.fixture(scope="module")
def qew():
    import paper_1211_7275_gb300 as q
    return q


def check(qew, L, kind, steps, f=None, u0=None):
    L = np.asarray(L)
    f = np.full(L.size, F[kind]) if f is None else f
    ref = oracle.run(L, f, 0.1, np.full(L.size, kind, dtype=np.int32), SEED, steps, u0=u0, want_state=True)
    with qew.Relaxation(L, f, kind, dt=0.1, seed=SEED, precision=qew.FP64) as r:
        if u0 is not None:
            r.set_state(u0)
        obs = r.observe(steps)
        u, _ = r.state()
        cells = r.cells()
    np.testing.assert_allclose(u, ref["u"], rtol=1e-12, atol=1e-12)
    assert np.array_equal(cells, np.floor(ref["u"]).astype(np.int32))
    for k in ("v", "ubar", "w2"):
        np.testing.assert_allclose(obs[k], ref[k], rtol=1e-10, atol=1e-11)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("L", [[1, 2, 3, 66, 67, 65, 1537, 130], [4096, 4096], [4096, 4097], [1 << 14, 1 << 14], [(1 << 15) + 1]])
def test_small_batches(qew, kind, L):
    # whole launches, parts of them, single steps and repeated observations of one launch's end
    check(qew, L, kind, np.array([0, 1, 2, 31, 32, 33, 80, 97]))


@pytest.mark.parametrize("kind,L", [(RF, [1 << 20]), (RF, [(1 << 20) + 1]), (RBG_LINEAR, [(1 << 20) + 1]), (RB, [(1 << 20) - 497, 499])])
def test_large_batches(qew, kind, L):
    check(qew, L, kind, np.array([0, 1, 7, 8, 9, 29]))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("L", [777, (1 << 20) + 3])
def test_steep_line(qew, kind, L):
    """Neighbours hundreds of cells apart: moves of many cells, up and down, every step.  (Smooth enough
    that every step stays far from the edge of a cell by more than rounding.)"""
    u0 = 300.0 * np.sin(2 * np.pi * np.arange(L) / 7.0) + 0.37
    check(qew, [L], kind, np.array([1, 2, 9]), u0=u0)
