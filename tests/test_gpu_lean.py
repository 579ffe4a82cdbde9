"""The forms that a handle falls back to when device memory is short, and FP64 batches beyond 2^29 sites
with it (one step per launch, the disorder caches updated in place): against the oracle in FP64 to the
path's 1e-12, and against the ordinary form in FP32-split, bit for bit."""
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


def lean(r):
    r._check(r._lib.qew_selftest_lean(r._h))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("L", [[1, 2, 3, 66, 1023, 1024, 1025, 130], [4096, 4097], [(1 << 17) + 1]])
@pytest.mark.parametrize("steep", [False, True])
def test_fp64_in_place(qew, kind, L, steep):
    n = sum(L)
    u0 = 300.0 * np.sin(2 * np.pi * np.arange(n) / 7.0) + 0.37 if steep else None
    steps = np.array([1, 2, 9]) if steep else np.array([0, 1, 2, 31, 32, 33])
    ref = oracle.run(L, F[kind], 0.1, kind, SEED, steps, u0=u0, want_state=True)
    with qew.Relaxation(L, F[kind], kind, dt=0.1, seed=SEED, precision=qew.FP64) as r:
        lean(r)
        if steep:
            r.set_state(u0)
        obs = r.observe(steps)
        u, _ = r.state()
    np.testing.assert_allclose(u, ref["u"], rtol=1e-12, atol=1e-12)
    for k in ("v", "ubar", "w2"):
        np.testing.assert_allclose(obs[k], ref[k], rtol=1e-10, atol=1e-11)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", [None, (224, 16, 2), (480, 7, 1), (736, 32, 2), (992, 16, 1)])
def test_fp32_lean_equals_the_ordinary_form(qew, kind, shape):
    """Drives of both signs; chains of odd length, shorter than a tile, of one site, and long ones."""
    L = np.array([1537, 100, 4096, 1, 449, 300001])
    f = F[kind] * np.array([1.0, -1.0, -2.0, 1.0, 0.0, -1.0])
    steps = [0, 1, 2, 30, 31, 32, 100, 217]
    outs = []
    for is_lean in (False, True):
        with qew.Relaxation(L, f, kind, dt=0.1, seed=SEED) as r:
            if shape:
                r.set_tuning(*shape)
            if is_lean:
                lean(r)
            obs = r.observe(steps)
            r.advance(45)
            S = r.state()[0]
            r.set_state(S)
            r.advance(20)
            outs.append((obs, S, r.state()[0], r.cells()))
    (a, *sa), (b, *sb) = outs
    for x, y in zip(sa, sb):
        assert np.array_equal(x, y)
    for k in ("v", "ubar", "w2"):   # one FP64 rounding of sums relative to another integer cell
        np.testing.assert_allclose(a[k], b[k], rtol=1e-13, atol=1e-13)


def test_mixed_batch(qew):
    L = np.array([3000, 4097, 777, 5025, 2048, 25001])
    kind = np.array([RF, RB, NONE, RBG_LINEAR, RBG_CUBIC, RBG_LINEAR], dtype=np.int32)
    f = np.array([F[k] for k in kind]) * np.array([1, -1, 1, -1, 1, 1])
    outs = []
    for is_lean in (False, True):
        with qew.Relaxation(L, f, kind, dt=0.1, seed=SEED) as r:
            if is_lean:
                lean(r)
            r.advance(100)
            outs.append(r.state()[0])
    assert np.array_equal(*outs)
