"""Two distant fragments with orbitals of their own and electrons shared out
unevenly: ln|psi| hangs on orbitals that are tiny where the electrons are, far
below the largest basis functions there, so fixed-point sums must give way to
FP64 ones.  FP64 form against the oracle, at the FP64 path's 1e-10."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu
CASES = [(1, 8.0), (1, 11.0), (1, 14.0), (1, 17.0), (3, 12.0), (3, 16.0), (3, 19.0)]


def fragments(m, D):
    """Two m-water clusters, the second D bohr along x; orbitals of one fragment each."""
    a = synth.water_system(m)
    s = a.copy()
    s.Z, s.R, s.a_en = np.r_[a.Z, a.Z], np.r_[a.R, a.R + [D, 0, 0]], np.r_[a.a_en, a.a_en]
    s.n_up, s.n_dn = 2 * a.n_up, 2 * a.n_dn
    s.shell_center = np.r_[a.shell_center, a.shell_center + a.n_nuc].astype(np.int32)
    for f in ("shell_l", "shell_pure", "shell_nprim", "alpha", "coef"):
        setattr(s, f, np.r_[getattr(a, f), getattr(a, f)])
    n, nb = a.n_up, a.C.shape[1]
    s.C = np.zeros((2 * n, 2 * nb))
    s.C[:n, :nb] = s.C[n:, nb:] = a.C[:n]
    s.occ_up = np.arange(2 * n, dtype=np.int32)
    s.occ_dn = s.occ_up.copy()
    return s


def walkers(m, D, W, seed=0):
    """One spin-up electron of the first fragment sits on the second."""
    a = synth.water_system(m)
    R = np.concatenate([synth.initial_walkers(a, W, seed=seed), synth.initial_walkers(a, W, seed=seed + 1) + [D, 0, 0]], 1)
    n = a.n_up
    R = R[:, np.r_[np.arange(n), 2 * n + np.arange(n), n + np.arange(n), 3 * n + np.arange(n)]]
    R[:, 0, 0] += D
    return R


def close(got, ref, tol):
    err = np.abs(got - ref).reshape(len(ref), -1).max(1) / np.maximum(1.0, np.abs(ref).reshape(len(ref), -1).max(1))
    assert err.max() <= tol, err.max()


@pytest.mark.parametrize("m,D", CASES + [(7, 20.0)])
def test_rebuild(m, D):
    from paper_2504_07948_gb300 import qmc as Q
    s, R = fragments(m, D), walkers(m, D, 16)
    g = Q.QMC(s, precision="fp64")
    g.set_walkers(R)
    ev = g.evaluate()
    g.close()
    ref = O.Oracle(s).evaluate(R)
    for k in ("logpsi", "eloc", "grad"):
        close(ev[k], ref[k], 1e-10)
    assert np.array_equal(ev["sign"], ref["sign"])


@pytest.mark.parametrize("m,D", CASES)
def test_sweeps(m, D):
    """Two sweeps: the oracle's moves, and a propagated state that its evaluation confirms."""
    from paper_2504_07948_gb300 import qmc as Q
    s, R = fragments(m, D), walkers(m, D, 16)
    g = Q.QMC(s, precision="fp64", seed=5)
    g.set_walkers(R)
    g.vmc(2, 0.02)
    Rg, ev = g.get_walkers()[0], g.eval_cached()
    g.close()
    Ro, _, _ = O.Oracle(s).vmc(R, 2, 0.02, seed=5, step0=0, trace=False)
    assert np.abs(Rg - Ro).max() <= 1e-8
    ref = O.Oracle(s).evaluate(Rg)
    for k in ("logpsi", "eloc", "grad"):
        close(ev[k], ref[k], 1e-8)


@pytest.mark.parametrize("path", ["fused", "gemm"])
@pytest.mark.parametrize("m,D", CASES)
def test_forces(m, D, path, monkeypatch):
    from paper_2504_07948_gb300 import qmc as Q
    monkeypatch.setenv("QMC_FORCE_GEMM_MIN_N", "1" if path == "gemm" else "1000")
    s, R = fragments(m, D), walkers(m, D, 16)
    g = Q.QMC(s, precision="fp64")
    g.set_walkers(R)
    pw = g.forces()[1]
    g.close()
    for c, ref in enumerate(O.Oracle(s).forces(R)):   # E_L, ln|psi|
        close(pw[:, c], ref, 1e-10)


def test_forces_some_walkers(monkeypatch):
    """More than a chunk of walkers, every third of them with the electrons shared out unevenly, spins of different size."""
    from paper_2504_07948_gb300 import qmc as Q
    monkeypatch.setenv("QMC_FORCE_GEMM_MIN_N", "1")
    m, D = 3, 16.0
    s = fragments(m, D)
    s.n_dn -= 3
    s.occ_dn = s.occ_dn[:s.n_dn]
    few, even = walkers(m, D, 4)[:, :-3], walkers(m, D, 8, seed=7)[:, :-3]
    even[:, 0, 0] -= D
    R = np.stack([few, even[:4], even[4:]], 1).reshape(12, -1, 3)
    g = Q.QMC(s, precision="fp64")
    g.set_walkers(np.tile(R, (27, 1, 1)))
    pw = g.forces()[1]
    g.close()
    for c, ref in enumerate(O.Oracle(s).forces(R)):
        close(pw[:, c], np.tile(ref, (27, 1, 1)), 1e-10)
