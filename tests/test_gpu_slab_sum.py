"""Slabs of the triples at the edges of the 8 x 8 x 8 bricks, against the oracle.

The sum over the images of a slab and its division take one brick of one pair
j <= k at a time: virtual counts below, at and above a multiple of 8 and one
virtual or one occupied index, whole and ragged slabs.  Bounds: FP64 1e-10,
FP32 1e-5 of the largest residual, as for the other blocked and FP32 tests.
"""
import numpy as np
import pytest
import torch

from oracle import cc3
from paper_2407_18947_gb300.synth import make_system, random_amplitudes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [(0, 1e-10), (1, 1e-5)])
@pytest.mark.parametrize("o,v,chunk", [(1, 8, 1), (2, 9, 1), (3, 16, 2), (4, 1, 3), (5, 7, 5)])
def test_slab_bricks_match_oracle(o, v, chunk, precision, tol):
    from paper_2407_18947_gb300.api import RTCC3
    s = make_system(o, v, seed=600 + 5 * o + v)
    amps = random_amplitudes(o, v, seed=601)
    eng = RTCC3(o, v, precision=precision, triples_chunk=chunk)
    eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
    eng.set_field(0, 1, 0.01, direction=(0.0, 0.3, 1.0))
    eng.set_amplitudes(0, *amps)
    eng.set_profiling(True)
    r = eng.compute_residuals(0, 0.0)
    assert eng.kernel_stats()["slab_sym"]["launches"] > 0
    eng.set_profiling(False)
    eng.close()
    ham = cc3.Hamiltonian.from_system(s)
    ref = cc3.evaluate(ham, *[torch.from_numpy(x) for x in amps],
                       ham.field_operator([0.0, 0.003, 0.01]))
    for k in ("r_t1", "r_t2", "r_l1", "r_l2"):
        want = getattr(ref, k).numpy()
        assert np.abs(r[k] - want).max() <= tol * np.abs(want).max(), k


def test_more_blocks_than_one_grid_dimension():
    """41 occupied orbitals in one slab: 68,921 occupied blocks, above the 65,535 of
    a grid dimension; FP64, 1e-10 of the largest residual as above."""
    from paper_2407_18947_gb300.api import RTCC3
    o, v = 41, 2
    s = make_system(o, v, seed=640)
    amps = random_amplitudes(o, v, seed=641)
    eng = RTCC3(o, v, precision=0, triples_chunk=o)
    eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
    eng.set_field(0, 1, 0.001, direction=(0.0, 0.3, 1.0))
    eng.set_amplitudes(0, *amps)
    r = eng.compute_residuals(0, 0.0)
    eng.close()
    ham = cc3.Hamiltonian.from_system(s)
    ref = cc3.evaluate(ham, *[torch.from_numpy(x) for x in amps],
                       ham.field_operator([0.0, 0.0003, 0.001]))
    for k in ("r_t1", "r_t2", "r_l1", "r_l2"):
        want = getattr(ref, k).numpy()
        assert np.abs(r[k] - want).max() <= 1e-10 * np.abs(want).max(), k
