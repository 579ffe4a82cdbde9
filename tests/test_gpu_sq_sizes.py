"""The structure factor at the lengths where its transform changes (even lengths go through a complex
transform of half the length, odd lengths and L = 2 through a real one), all modes and the first ones,
against numpy's transform of the same FP64 line.  A transform's error is a few units of rounding per
level relative to the largest mode: 1e-13 leaves two orders of magnitude."""
import numpy as np
import pytest

from qew_workloads import NONE, random_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qew():
    import paper_1211_7275_gb300 as q
    return q


@pytest.mark.parametrize("L,batch", [(2, 3), (3, 1), (4, 2), (5, 2), (6, 1), (7, 5), (8, 3), (10, 4), (509, 2), (510, 2), (1018, 17),
                                     (1 << 14, 5), ((1 << 14) + 1, 2), (60724, 1)])
def test_against_numpy(qew, L, batch):
    u = np.concatenate([random_state(L, 0.3, seed=7 + c) for c in range(batch)])
    ref = np.mean(np.abs(np.fft.rfft(u.reshape(batch, L), axis=1)[:, 1:L // 2 + 1] / L) ** 2, axis=0)
    with qew.Relaxation(L, 0.5, NONE, precision=qew.FP64, batch=batch) as r:
        r.set_state(u)
        for m in (L // 2, 1, max(1, L // 3), L // 2):   # the work area is reused and grows
            S = r.structure_factor(m)
            assert np.max(np.abs(S - ref[:m])) <= 1e-13 * ref.max(), m
