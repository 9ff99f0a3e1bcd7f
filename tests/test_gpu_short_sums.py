"""Short split-TF32 sums with a large output, at the kernel's edges, against FP64.

The persistent kernel takes sums of up to six 16-term K tiles: one and two
accumulators in tensor memory (four tiles is the line), a last K tile of one or
two terms, row and column blocks with remainders, overwriting and accumulating
products (the blocked triples accumulate).  Bound 1e-5 of the largest residual,
as in the FP32 tests: a split product is off by up to 2**-21 of its factors, and
the residuals' sums of magnitudes are of the order of ten times the residuals.
A wrong edge or a lost tile is off by percents.
"""
import numpy as np
import pytest

from paper_2407_18947_gb300.synth import make_system, random_amplitudes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("o,v,chunk", [(5, 34, -1), (5, 34, 2), (4, 49, 3), (3, 66, 2), (3, 82, 1),
                                       (18, 21, 2), (2, 97, 1)])
def test_short_sums_match_fp64(o, v, chunk):
    from paper_2407_18947_gb300.api import RTCC3
    s = make_system(o, v, seed=720 + 3 * o + v)
    amps = random_amplitudes(o, v, seed=721)
    out = {}
    for precision in (0, 2):
        eng = RTCC3(o, v, precision=precision, triples_chunk=chunk)
        eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
        eng.set_field(0, 1, 0.002, direction=(0.0, 0.3, 1.0))
        eng.set_amplitudes(0, *amps)
        out[precision] = eng.compute_residuals(0, 0.0)
        if precision == 2:
            eng.set_profiling(True)
            eng.compute_residuals(0, 0.0)
            assert eng.kernel_stats()["contract_tc_tf32"]["launches"] > 0
        eng.close()
    for k in ("r_t1", "r_t2", "r_l1", "r_l2"):
        assert np.abs(out[2][k] - out[0][k]).max() <= 1e-5 * np.abs(out[0][k]).max(), k
