"""The plain FP64 path from lines that hold negative zeros, which belong to cell 0 like the positive
one, against the oracle to the path's 1e-12, in small batches (whose sites hold look-ahead nodes) and in
large ones."""
import numpy as np
import pytest

import oracle
from qew_workloads import NONE, RB, RBG_CUBIC, RBG_LINEAR, RF, SEED

pytestmark = pytest.mark.gpu
F = {RF: 0.9, RB: 1.1, NONE: 0.3, RBG_LINEAR: 1.6, RBG_CUBIC: 2.0}


@pytest.mark.parametrize("kind", [RF, RB, NONE, RBG_LINEAR, RBG_CUBIC])
@pytest.mark.parametrize("line", ["negative", "mixed"])
@pytest.mark.parametrize("L", [777, 40001, (1 << 20) + 3])
def test_negative_zero_is_in_cell_zero(kind, line, L):
    import paper_1211_7275_gb300 as qew
    u0 = np.full(L, -0.0)
    if line == "mixed":
        u0[::3], u0[1::7], u0[4::11] = 0.0, 0.25, -0.25
    steps = np.array([0, 1, 2, 9])
    ref = oracle.run([L], F[kind], 0.1, kind, SEED, steps, u0=u0, want_state=True)
    with qew.Relaxation([L], F[kind], kind, dt=0.1, seed=SEED, precision=qew.FP64) as r:
        r.set_state(u0)
        assert np.array_equal(r.cells(), np.floor(u0).astype(np.int32))
        obs = r.observe(steps)
        u, _ = r.state()
        cells = r.cells()
    np.testing.assert_allclose(u, ref["u"], rtol=1e-12, atol=1e-12)
    assert np.array_equal(cells, np.floor(ref["u"]).astype(np.int32))
    for k in ("v", "ubar", "w2"):
        np.testing.assert_allclose(obs[k], ref[k], rtol=1e-10, atol=1e-11)
