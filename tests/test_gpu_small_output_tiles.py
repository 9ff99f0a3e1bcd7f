"""Long sums with a small output, at the edges of the output tiles, FP32.

The triples densities sum over five of six triples indices onto a vir x vir and
an occ x occ output; the kernel takes the smallest tile that holds the output.
Sizes are one below, at and one above tile edges on either side (17 to 96
virtuals, 17 to 33 occupieds), where a wrong edge mask or a wrong choice shows.
Bound 1e-5 of the largest residual: chains of at most a few thousand FP32
roundings of 6e-8, as in the other FP32 tests.
"""
import numpy as np
import pytest
import torch

from oracle import cc3
from paper_2407_18947_gb300.synth import make_system, random_amplitudes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("o,v", [(3, 20), (3, 21), (3, 24), (3, 32), (3, 33), (1, 65), (1, 80),
                                 (1, 81), (1, 96), (1, 97), (17, 3), (20, 2), (21, 2), (24, 2),
                                 (32, 2), (33, 2)])
def test_density_tiles_match_oracle(o, v):
    from paper_2407_18947_gb300.api import RTCC3
    s = make_system(o, v, seed=500 + 3 * o + v)
    amps = random_amplitudes(o, v, seed=501)
    eng = RTCC3(o, v, precision=1)
    eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
    eng.set_field(0, 1, 0.002, direction=(0.0, 0.3, 1.0))
    eng.set_amplitudes(0, *amps)
    r = eng.compute_residuals(0, 0.0)
    eng.close()
    ham = cc3.Hamiltonian.from_system(s)
    ref = cc3.evaluate(ham, *[torch.from_numpy(x) for x in amps],
                       ham.field_operator([0.0, 0.0006, 0.002]))
    for k in ("r_t1", "r_t2", "r_l1", "r_l2"):
        want = getattr(ref, k).numpy()
        assert np.abs(r[k] - want).max() <= 1e-5 * np.abs(want).max(), k
