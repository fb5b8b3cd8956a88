"""FP64 Jastrow terms at the end of the range: with b = 8e307 the denominators
1 + b r are huge or infinite, their reciprocals at most 1e-307, and the factor
leaves E_L, gradients and moves as they are without it."""
import numpy as np
import pytest

from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


def test_infinite_denominators():
    from paper_2504_07948_gb300 import qmc as Q
    out = []
    for a, b in ((0.0, 1.0), (0.5, 8e307)):
        s = synth.water_system(2).copy()
        s.a_anti, s.a_par, s.b_ee, s.b_en = a, a / 2, b, b
        s.a_en = np.full(s.n_nuc, -a)
        g = Q.QMC(s, precision="fp64", seed=3)
        g.set_walkers(synth.initial_walkers(s, 20, seed=2))
        ev = g.evaluate()
        g.vmc(2, 0.02)
        out.append([ev[k].copy() for k in ("logpsi", "eloc", "grad")] + [g.get_walkers()[0]])
        g.close()
    for x, y in zip(*out):
        assert np.all(np.isfinite(y)) and np.array_equal(x, y)
