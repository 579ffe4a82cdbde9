"""Moves of the plain FP64 path under drives of both signs and from steep lines, whose sites lose all of
their nodes at once.  Small batches hold the node that a move in the drive's direction will need and draw
in gathered rounds; large ones draw where they are.  The rounding sequence is the same: a chain relaxed in
a small batch and beside 2^20 other sites gives the same line and the same observables, bit for bit."""
import numpy as np
import pytest

from qew_workloads import NONE, RB, RBG_CUBIC, RBG_LINEAR, RF, SEED

pytestmark = pytest.mark.gpu
F = {RF: 0.9, RB: 1.1, RBG_LINEAR: 1.6, RBG_CUBIC: 2.0}
STEPS = np.array([0, 1, 2, 31, 40, 100])


def both(L, f, kind, u0):
    import paper_1211_7275_gb300 as qew
    outs = []
    for beside in ([], [1 << 20]):
        kinds = [kind] * len(L) + [NONE] * len(beside)
        with qew.Relaxation(L + beside, np.append(f, [0.3] * len(beside)), kinds, dt=0.1, seed=SEED, precision=qew.FP64) as r:
            r.set_state(np.append(u0, np.zeros(sum(beside))))
            obs = r.observe(STEPS)
            outs.append([obs[k][:, :len(L)] for k in ("v", "ubar", "w2")] + [r.state()[0][:sum(L)], r.cells()[:sum(L)]])
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("kind", [RF, RB, RBG_LINEAR, RBG_CUBIC])
@pytest.mark.parametrize("drive", [-0.5, -1.0, 1.0, -4.0, 4.0, -40.0, 40.0])
@pytest.mark.parametrize("L", [[777, 4, 130, 1], [12000, 3000], [40001]])
def test_driven_lines(kind, drive, L):
    """From a rough line; the drives of a batch alternate in sign."""
    f = drive * F[kind] * np.where(np.arange(len(L)) % 2, -1.0, 1.0)
    both(L, f, kind, 0.7 * np.random.default_rng(3).standard_normal(sum(L)))


@pytest.mark.parametrize("L", [(3 << 18) - 1, 3 << 18])
def test_where_the_uniform_random_bond_changes_shape(L):
    both([L], np.array([F[RB]]), RB, 0.7 * np.random.default_rng(3).standard_normal(L))


@pytest.mark.parametrize("kind", [RF, RB, RBG_LINEAR, RBG_CUBIC])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("L", [777, 9000, 60000])
def test_steep_lines_that_calm_down(kind, sign, L):
    """Steep stretches: moves of many cells there and single ones elsewhere, in the same tile."""
    x = np.arange(L)
    u0 = 0.37 + np.where(x % 256 < 40, 60.0 * np.sin(2 * np.pi * x / 9.0), 0.1 * np.sin(2 * np.pi * x / 50.0))
    both([L], np.array([sign * F[kind]]), kind, u0)
