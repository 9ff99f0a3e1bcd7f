"""Products small enough for the lane-split kernel, against the oracle.

Tiny and lopsided systems, where every product has fewer terms than one tile:
one occupied or one virtual orbital (sums of length 1), sums that are not a
multiple of the lane split, and the block-per-output form (few outputs, sums
above 512).  Bounds: FP64 1e-10; FP32 1e-5 of the largest residual (a chain of
at most a few thousand FP32 roundings of 6e-8, as in the other FP32 tests).
"""
import numpy as np
import pytest
import torch

from oracle import cc3
from paper_2407_18947_gb300.synth import make_system, random_amplitudes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [(0, 1e-10), (1, 1e-5)])
@pytest.mark.parametrize("o,v", [(1, 1), (1, 5), (2, 1), (2, 3), (3, 9), (4, 14)])
def test_small_products_match_oracle(o, v, precision, tol):
    from paper_2407_18947_gb300.api import RTCC3
    s = make_system(o, v, seed=400 + 7 * o + v)
    amps = random_amplitudes(o, v, seed=401)
    eng = RTCC3(o, v, precision=precision)
    eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
    eng.set_field(0, 1, 0.02, direction=(0.0, 0.3, 1.0))
    eng.set_amplitudes(0, *amps)
    eng.set_profiling(True)
    r = eng.compute_residuals(0, 0.0)
    name = "contract_fine_c128" if precision == 0 else "contract_fine_c64"
    assert eng.kernel_stats()[name]["launches"] > 0
    eng.set_profiling(False)
    eng.close()
    ham = cc3.Hamiltonian.from_system(s)
    ref = cc3.evaluate(ham, *[torch.from_numpy(x) for x in amps],
                       ham.field_operator([0.0, 0.006, 0.02]))
    for k in ("r_t1", "r_t2", "r_l1", "r_l2"):
        want = getattr(ref, k).numpy()
        assert np.abs(r[k] - want).max() <= tol * np.abs(want).max(), k
