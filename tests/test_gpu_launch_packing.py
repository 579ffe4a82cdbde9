"""How observations and steps are spread over launches changes nothing: a launch records every
observation that falls into its K steps, on windows aligned to four sites, and its sums are those of
one launch per observation.  Against one-observation calls (each its own launch) bit for bit, and
against the oracle's plain sums."""
import numpy as np
import pytest

from qew_workloads import NONE, RB, RBG_CUBIC, RBG_LINEAR, RF, SEED

pytestmark = pytest.mark.gpu

F = {RF: 0.9, RB: 1.1, NONE: 0.3, RBG_LINEAR: 1.6, RBG_CUBIC: 2.0}


@pytest.fixture(scope="module")
def qew():
    import paper_1211_7275_gb300 as q
    return q


# crowded observations (more than one launch holds), a step apart, K apart, one off K, and far apart
CROWDED = list(range(0, 31)) + [32, 33, 63, 64, 65, 95, 128, 161, 200, 201]


@pytest.mark.parametrize("kind", [RF, RB, NONE, RBG_LINEAR, RBG_CUBIC])
@pytest.mark.parametrize("shape", [(224, 16, 2), (480, 32, 1), (224, 5, 4), (480, 7, 1), (480, 1, 2)])
def test_packed_observations_equal_single_ones(qew, kind, shape):
    """v, ubar, w2 and the line; chains of odd length, shorter than a tile, and of one site."""
    L = np.array([1537, 100, 4096, 1, 449])
    outs = []
    for one_by_one in (False, True):
        with qew.Relaxation(L, F[kind], kind, dt=0.1, seed=SEED) as r:
            r.set_tuning(*shape)
            if one_by_one:
                o = [r.observe([t]) for t in CROWDED]
                obs = {k: np.concatenate([x[k] for x in o]) for k in ("v", "ubar", "w2")}
            else:
                obs = r.observe(CROWDED)
            outs.append((obs, r.state()[0]))
    (a, ua), (b, ub) = outs
    assert np.array_equal(ua, ub)
    # one rounding of an FP64 sum that is taken relative to another integer cell
    for k in ("v", "ubar", "w2"):
        np.testing.assert_allclose(a[k], b[k], rtol=1e-13, atol=1e-13)


@pytest.mark.parametrize("kind", [RF, RBG_LINEAR])
def test_crowded_observations_match_the_oracle(qew, kind):
    import oracle
    L = [1537, 700]
    ref = oracle.run(L, F[kind], 0.1, kind, SEED, np.array(CROWDED))
    with qew.Relaxation(np.array(L), F[kind], kind, dt=0.1, seed=SEED) as r:
        r.set_tuning(480, 32, 1)
        obs = r.observe(CROWDED)
    # FP32 sums over 448-site tiles, and the per-site bar of 1e-4
    np.testing.assert_allclose(obs["v"], ref["v"], atol=1e-4)
    np.testing.assert_allclose(obs["ubar"], ref["ubar"], atol=1e-4)
