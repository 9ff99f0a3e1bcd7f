"""FP64 products as sliced tensor-core products, against the oracle.

Sizes are chosen at the edges of the kernel's tiles (128 rows, 16/32/64 real
columns, 128-long K segments, 16-long stages): rows and sums just below, at
and above them, one operand much wider than the other.  A sliced product
keeps 62 bits of every row, so the FP64 bound of the other parity tests
(1e-10 of the largest residual) applies unchanged.
"""
import numpy as np
import pytest
import torch

from oracle import cc3
from paper_2407_18947_gb300.synth import make_system, random_amplitudes

pytestmark = pytest.mark.gpu


def _residuals(s, amps, field=0.02, **opt):
    from paper_2407_18947_gb300.api import RTCC3
    eng = RTCC3(s.nocc, s.nvir, precision=0, **opt)
    eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
    eng.set_field(0, 1, field, direction=(0.0, 0.3, 1.0))
    eng.set_amplitudes(0, *amps)
    eng.set_profiling(True)
    r = eng.compute_residuals(0, 0.0)
    sliced = eng.kernel_stats().get("contract_sliced_c128", {"launches": 0})["launches"]
    eng.set_profiling(False)
    eng.close()
    return r, sliced


@pytest.mark.parametrize("o,v", [(8, 16), (7, 17), (5, 26), (3, 43), (9, 15)])
def test_sliced_products_match_oracle(o, v):
    s = make_system(o, v, seed=300 + o)
    amps = random_amplitudes(o, v, seed=301 + v)
    r, sliced = _residuals(s, amps)
    assert sliced > 0
    ham = cc3.Hamiltonian.from_system(s)
    ref = cc3.evaluate(ham, *[torch.from_numpy(x) for x in amps],
                       ham.field_operator([0.0, 0.006, 0.02]))
    for k in ("r_t1", "r_t2", "r_l1", "r_l2"):
        want = getattr(ref, k).numpy()
        assert np.abs(r[k] - want).max() <= 1e-10 * np.abs(want).max(), k


def test_rows_of_very_different_magnitude():
    """Amplitudes whose rows span 1e-8 .. 1: the rows are scaled one by one."""
    o, v = 7, 17
    s = make_system(o, v, seed=310)
    amps = list(random_amplitudes(o, v, seed=311))
    w = np.logspace(-8, 0, v)
    amps[1] = amps[1] * np.sqrt(w[:, None] * w[None, :])
    r, sliced = _residuals(s, amps)
    assert sliced > 0
    ham = cc3.Hamiltonian.from_system(s)
    ref = cc3.evaluate(ham, *[torch.from_numpy(x) for x in amps],
                       ham.field_operator([0.0, 0.006, 0.02]))
    for k in ("r_t1", "r_t2", "r_l1", "r_l2"):
        want = getattr(ref, k).numpy()
        assert np.abs(r[k] - want).max() <= 1e-10 * np.abs(want).max(), k


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_amplitudes_stay_non_finite(bad):
    """The integer conversion has no code for them: such rows are marked."""
    from paper_2407_18947_gb300.api import RTCC3
    o, v = 8, 16
    s = make_system(o, v, seed=320)
    t1, t2, _, _ = random_amplitudes(o, v, seed=321)
    t2 = t2.copy()
    t2[1, 2, 3, 4] = bad
    eng = RTCC3(o, v, precision=0)
    eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
    T1, T2 = torch.tensor(t1, device="cuda"), torch.tensor(t2, device="cuda")
    x1, x2 = torch.empty_like(T1), torch.empty_like(T2)
    eng.set_profiling(True)
    eng.triples_forward_dev(0, 0.0, T1.data_ptr(), T2.data_ptr(), x1.data_ptr(), x2.data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    sliced = eng.kernel_stats().get("contract_sliced_c128", {"launches": 0})["launches"]
    eng.set_profiling(False)
    eng.close()
    assert sliced > 0
    assert not torch.isfinite(torch.view_as_real(x2)).all()
