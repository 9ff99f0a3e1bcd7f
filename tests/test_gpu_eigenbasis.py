"""The field eigenbasis where its solver can go wrong, against the oracle.

Weak fields (the correction of the identity converges), equal and nearly equal
orbital energies (each coupled pair is a full rotation), strong fields (the QR
algorithm takes over) and orders below, at and above the eight rows per
cluster.  The oracle solves the field-coupled triples by a fixed point and
shares nothing with either solver; FP64 bound 1e-10 as elsewhere.
"""
import numpy as np
import pytest
import torch

from oracle import cc3
from paper_2407_18947_gb300.synth import make_system, random_amplitudes

pytestmark = pytest.mark.gpu


def _check(s, o, v, field, seed):
    from paper_2407_18947_gb300.api import RTCC3
    amps = random_amplitudes(o, v, seed=seed)
    eng = RTCC3(o, v, precision=0)
    eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
    eng.set_field(0, 1, field, direction=(0.2, 0.0, 1.0))
    eng.set_amplitudes(0, *amps)
    r = eng.compute_residuals(0, 0.0)
    eng.close()
    ref = cc3.evaluate(cc3.Hamiltonian.from_system(s), *[torch.from_numpy(x) for x in amps],
                       cc3.Hamiltonian.from_system(s).field_operator([0.2 * field, 0.0, field]))
    for k in ("r_t1", "r_t2", "r_l1", "r_l2"):
        want = getattr(ref, k).numpy()
        assert np.abs(r[k] - want).max() <= 1e-10 * np.abs(want).max(), k


@pytest.mark.parametrize("o,v", [(1, 2), (3, 7), (4, 8), (5, 9), (8, 17)])
@pytest.mark.parametrize("field", [0.0, 0.002, 0.08])
def test_orders_and_field_strengths(o, v, field):
    _check(make_system(o, v, seed=500 + v), o, v, field, 501)


@pytest.mark.parametrize("gap", [0.0, 1e-9, 1e-5])
def test_nearly_equal_orbital_energies(gap):
    o, v = 4, 11
    s = make_system(o, v, seed=510)
    s.eps[1] = s.eps[0] + gap                      # an occupied pair
    s.eps[o + 3] = s.eps[o + 2] + gap              # a virtual pair
    s.eps[o + 7] = s.eps[o + 6] + gap              # and three virtuals together
    s.eps[o + 8] = s.eps[o + 6] + 2.0 * gap
    _check(s, o, v, 0.01, 511)
