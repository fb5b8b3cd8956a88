"""FP64 Sherman-Morrison sweep beyond the small clusters: 256-thread CTAs with
the inverse in shared memory (70 electrons per spin) and in global memory (120),
and a basis whose lists exceed shared memory, which falls back to the general
sweep and to FP64 orbital sums.  Trajectories and the propagated state against
the oracle; rounding differences are 1e-13 at these sizes, a flipped decision
would move an electron by ~0.1 bohr."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


def large_basis():
    """One water with 3300 tight s functions more, each in the orbitals with a small weight."""
    s = synth.water_system(1).copy()
    extra = 3300
    rng = np.random.default_rng(5)
    s.shell_center = np.r_[s.shell_center, rng.integers(0, s.n_nuc, extra)].astype(np.int32)
    for f, v in (("shell_l", 0), ("shell_pure", 0), ("shell_nprim", 1)):
        setattr(s, f, np.r_[getattr(s, f), np.full(extra, v)].astype(np.int32))
    s.alpha = np.r_[s.alpha, np.exp(rng.uniform(np.log(0.3), np.log(50.0), extra))]
    s.coef = np.r_[s.coef, np.ones(extra)]
    s.C = np.concatenate([s.C, 0.01 * rng.normal(size=(s.C.shape[0], extra))], 1)
    return s


@pytest.mark.parametrize("name,W", [("water14", 3), ("water24", 2), ("large_basis", 5)])
def test_sweep_follows_the_oracle(name, W):
    from paper_2504_07948_gb300 import qmc as Q
    s = large_basis() if name == "large_basis" else synth.water_system(int(name[5:]))
    R = synth.initial_walkers(s, W, seed=51)
    g = Q.QMC(s, precision="fp64", seed=77)
    g.set_walkers(R)
    fresh = g.evaluate()
    g.vmc(1, 0.02)
    Rg, ev = g.get_walkers()[0], g.eval_cached()
    g.close()
    o = O.Oracle(s)
    Ro, _, _ = o.vmc(R, 1, 0.02, seed=77, step0=0, trace=False)
    assert np.abs(Rg - Ro).max() <= 1e-8
    for got, ref, tol in ((fresh, o.evaluate(R), 1e-10), (ev, o.evaluate(Rg), 1e-9)):
        for k in ("logpsi", "eloc"):
            assert np.all(np.abs(got[k] - ref[k]) <= tol * np.maximum(1.0, np.abs(ref[k]))), k
