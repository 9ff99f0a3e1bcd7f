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


@pytest.mark.parametrize("precision,tol", [(0, 1e-10), (1, 1e-5)])
@pytest.mark.parametrize("o,v,pair", [(2, 2, "vir"), (2, 2, "occ"), (2, 6, "vir"), (3, 4, "occ")])
@pytest.mark.parametrize("split", [-0.3, 0.3])
def test_real_pair_with_couplings_of_opposite_sign(precision, tol, o, v, pair, split):
    """Purely real amplitudes dress two nearly equal orbitals with couplings
    +-0.1 E and half a diagonal difference of 0.1 E split: the eigenvalues are
    a complex pair, alone in its matrix or uncoupled from the rest of it."""
    from paper_2407_18947_gb300.api import RTCC3
    field = 0.02
    s = make_system(o, v, seed=520 + o + v)
    amps = [x.real.astype(np.complex128) for x in random_amplitudes(o, v, seed=521)]
    p, q = 0, 1                                     # the two orbitals of the pair
    gap = 0.2 * field * (1.0 - split)
    amps[0][:] = 0.0
    s.dipole[:] = 0.0
    if pair == "vir":
        s.eps[o + q] = s.eps[o + p] + gap
        amps[0][0, p], amps[0][0, q] = 0.1, -0.1    # w~_ab = -t_0a w_0b
        for x in (o + p, o + q):
            s.dipole[2, 0, x] = s.dipole[2, x, 0] = 1.0
    else:
        s.eps[q] = s.eps[p] - gap
        amps[0][p, 0], amps[0][q, 0] = 0.1, -0.1    # w~_ij = w_i0 t_j0
        for x in (p, q):
            s.dipole[2, x, o] = s.dipole[2, o, x] = 1.0
    eng = RTCC3(o, v, precision=precision)
    eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
    eng.set_field(0, 1, field, direction=(0.0, 0.0, 1.0))
    eng.set_amplitudes(0, *amps)
    r = eng.compute_residuals(0, 0.0)
    eng.close()
    ham = cc3.Hamiltonian.from_system(s)
    ref = cc3.evaluate(ham, *[torch.from_numpy(x) for x in amps],
                       ham.field_operator([0.0, 0.0, field]))
    for k in ("r_t1", "r_t2", "r_l1", "r_l2"):
        want = getattr(ref, k).numpy()
        assert np.abs(r[k] - want).max() <= tol * np.abs(want).max(), k


@pytest.mark.parametrize("precision,big", [(0, 1e308), (1, 1e38)])
@pytest.mark.parametrize("o,v", [(1, 1), (1, 2), (2, 1)])
def test_overflowing_coupling_is_reported(precision, big, o, v):
    """A dressed matrix with an infinite element is refused, also where its
    diagonal is finite ((1, 2) and (2, 1): w~_01 = -t_0 w_1 alone overflows)."""
    from paper_2407_18947_gb300._lib import ERR_NONFINITE, RTCC3Error
    from paper_2407_18947_gb300.api import RTCC3
    s = make_system(o, v, seed=530)
    amps = [np.zeros_like(x) for x in random_amplitudes(o, v, seed=531)]
    s.dipole[:] = 0.0
    s.eps[:o] -= 1000.0                             # (a field of 20 is not too strong)
    s.eps[o:] += 1000.0
    amps[0][0, 0] = big
    i, a = o - 1, o + v - 1                         # the last occupied and virtual
    s.dipole[2, i, a] = s.dipole[2, a, i] = 1000.0
    eng = RTCC3(o, v, precision=precision)
    eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
    eng.set_field(0, 1, 0.02, direction=(0.0, 0.0, 1.0))
    eng.set_amplitudes(0, *amps)
    with pytest.raises(RTCC3Error) as ei:
        eng.compute_residuals(0, 0.0)
    assert ei.value.code == ERR_NONFINITE and "dressed field matrix" in str(ei.value)
    eng.close()
