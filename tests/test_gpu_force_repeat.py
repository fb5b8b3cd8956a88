"""Ionic derivatives of the GEMM force path repeat bit for bit: a nucleus's
terms are added in one order whatever the warps' timing.  One water has fewer
shell runs than a CTA has warps, so the two spins' runs of a nucleus are in
flight together."""
import numpy as np
import pytest

from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("m,W", [(1, 1500), (14, 96)])
def test_forces_of_the_gemm_path_repeat(precision, m, W, monkeypatch):
    from paper_2504_07948_gb300 import qmc as Q
    monkeypatch.setenv("QMC_FORCE_GEMM_MIN_N", "1")
    s = synth.water_system(m)
    g = Q.QMC(s, precision=precision)
    g.set_walkers(synth.initial_walkers(s, W, seed=8))
    first = g.forces()
    for _ in range(4):
        again = g.forces()
        assert all(np.array_equal(a, b) for a, b in zip(first, again))
    g.close()
