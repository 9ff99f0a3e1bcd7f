"""Short split-TF32 sums and small-output tiles, with the kernel that ran checked.

The detailed statistics name the K tiles of a short sum and the output tile of
a long one, so that a size which takes another route is not counted as
coverage.  Bounds as in the tests of these kernels' results: 1e-5 of the
largest residual.
"""
import re

import numpy as np
import pytest
import torch

from oracle import cc3
from paper_2407_18947_gb300.synth import make_system, random_amplitudes

pytestmark = pytest.mark.gpu


def _residuals(s, amps, precision, **opt):
    from paper_2407_18947_gb300.api import RTCC3
    eng = RTCC3(s.nocc, s.nvir, precision=precision, **opt)
    eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
    eng.set_field(0, 1, 0.002, direction=(0.0, 0.3, 1.0))
    eng.set_amplitudes(0, *amps)
    r = eng.compute_residuals(0, 0.0)
    eng.set_profiling(True)
    eng.compute_residuals(0, 0.0)
    names = list(eng.kernel_stats())
    eng.close()
    return r, names


# chunk >= 1: blocked, so every product accumulates.  (5, 34): three K tiles;
# (4, 64): four and five, two accumulators and one; (3, 82): six; (3, 97): the
# sum over virtuals has seven and is no short sum.
@pytest.mark.parametrize("o,v,chunk,tiles", [(5, 34, 5, 3), (4, 64, 2, 4), (3, 66, 2, 5),
                                             (3, 82, 1, 6), (3, 97, 1, 1)])
def test_short_sums(monkeypatch, o, v, chunk, tiles):
    monkeypatch.setenv("RTCC3_PROFILE_DETAIL", "1")
    s = make_system(o, v, seed=740 + 3 * o + v)
    amps = random_amplitudes(o, v, seed=741)
    got, names = _residuals(s, amps, 2, triples_chunk=chunk)
    ran = {int(m.group(1)) for m in (re.search(r"\|short=(\d+) ", n) for n in names) if m}
    assert tiles in ran and max(ran) <= 6, ran
    ref, _ = _residuals(s, amps, 0, triples_chunk=chunk)
    for k in ("r_t1", "r_t2", "r_l1", "r_l2"):
        assert np.abs(got[k] - ref[k]).max() <= 1e-5 * np.abs(ref[k]).max(), k


@pytest.mark.parametrize("o,v,side", [(3, 20, 20), (3, 21, 24), (3, 24, 24), (3, 32, 32), (3, 33, 40),
                                      (1, 65, 80), (1, 80, 80), (1, 81, 96), (1, 96, 96),
                                      (20, 3, 20), (21, 3, 24), (24, 3, 24), (32, 3, 32), (33, 3, 40)])
def test_density_tiles(monkeypatch, o, v, side):
    monkeypatch.setenv("RTCC3_PROFILE_DETAIL", "1")
    s = make_system(o, v, seed=760 + 3 * o + v)
    amps = random_amplitudes(o, v, seed=761)
    got, names = _residuals(s, amps, 1)
    density = "ijkabc,ijkdbc->ad" if v > o else "ijkabc,ljkabc->li"
    assert any(n.startswith(f"contract_small_c64|tile={side * side} {density}") for n in names), \
        [n for n in names if "contract_small" in n]
    ham = cc3.Hamiltonian.from_system(s)
    ref = cc3.evaluate(ham, *[torch.from_numpy(x) for x in amps],
                       ham.field_operator([0.0, 0.0006, 0.002]))
    for k in ("r_t1", "r_t2", "r_l1", "r_l2"):
        want = getattr(ref, k).numpy()
        assert np.abs(got[k] - want).max() <= 1e-5 * np.abs(want).max(), k
