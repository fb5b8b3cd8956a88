"""Non-local term over the primitives that each pseudopotential nucleus sees,
against the oracle: electrons at the edges of the cutoff and next to the
nucleus (no primitive dropped that is alive on the sphere of the points), all
shell kinds with exponents from diffuse to sharper than the cutoff, and rules
that do not fill the register batches.  FP64 at the 1e-10 and mixed at the 1e-5
of the E_L checks."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2504_07948_gb300 import qmc
    return qmc


def rule(nq):
    rng = np.random.default_rng(nq)
    p = rng.normal(size=(nq, 3))
    return p / np.linalg.norm(p, axis=1, keepdims=True), np.full(nq, 1.0 / nq)


def walkers_at_edges(s, W, seed):
    """Initial walkers with electron w mod N of walker w moved to one of the
    listed distances from the nearest pseudopotential nucleus."""
    rng = np.random.default_rng(seed)
    R = synth.initial_walkers(s, W, seed=seed)
    nuc = np.flatnonzero(s.pp_rcut > 0.0)
    for w in range(W):
        a = nuc[w % len(nuc)]
        rc = s.pp_rcut[a]
        d = [1e-3, 0.05, 0.5 * rc, rc * (1 - 1e-12), rc * (1 + 1e-12), rc * (1 - 1e-6)][w % 6]
        u = rng.normal(size=3)
        R.reshape(W, -1, 3)[w, w % (s.n_up + s.n_dn)] = s.R[a] + d * u / np.linalg.norm(u)
    return R


def rel(a, b):
    return float((np.abs(a - b) / np.maximum(1.0, np.abs(b))).max())


@pytest.mark.parametrize("nq", [1, 12, 13, 27])
def test_all_shell_kinds_fp64(Q, nq):
    rng = np.random.default_rng(nq)
    s = synth.random_small_system(rng, n_nuc=3, n_up=4, n_dn=3)
    s.alpha *= np.where(np.arange(len(s.alpha)) % 4 == 0, 60.0, 1.0)
    z = {int(round(v)): {"core": 0, "rcut": 1.4, "terms": [(-1, 2, 1.1, 0.3), (0, 2, 2.0, 1.5), (1, 1, 1.3, 0.7),
                                                          (2, 2, 0.9, -0.4)]} for v in s.Z}
    s = synth.with_pseudopotential(s, species=z, rule=rule(nq))
    R = walkers_at_edges(s, 24, 5)
    g = Q.QMC(s, precision="fp64", seed=9)
    Q.qmc_set_rng(g.h, 9, 2)
    g.set_walkers(R)
    e = g.evaluate()["eloc"]
    ref = O.Oracle(s).evaluate(R, pp_seed=9, pp_sweep=2)["eloc"]
    assert rel(e, ref) <= 1e-10, rel(e, ref)
    g.close()


@pytest.mark.parametrize("m,nq", [(1, 12), (6, 13), (6, 27)])
@pytest.mark.parametrize("tc", ["0", "1"])
def test_water_mixed(Q, monkeypatch, m, nq, tc):
    monkeypatch.setenv("QMC_NLPP_TC", tc)
    monkeypatch.setenv("QMC_NLPP_TC_MIN_N", "1")
    s = synth.with_pseudopotential(synth.water_system(m), rule=rule(nq))
    R = walkers_at_edges(s, 36, 7)
    g = Q.QMC(s, precision="mixed", seed=9)
    Q.qmc_set_rng(g.h, 9, 2)
    g.set_walkers(R)
    e = g.eval_cached()["eloc"]
    ref = O.Oracle(s).evaluate(R, pp_seed=9, pp_sweep=2)["eloc"]
    assert rel(e, ref) <= 1e-5, rel(e, ref)
    g.close()


@pytest.mark.parametrize("m,W", [(9, 5), (17, 3), (32, 2)])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("mixed", 1e-5)])
def test_walkers_in_slices(Q, m, W, prec, tol):
    """Few walkers of many electrons (the energy pass runs 2, 4 and 8 CTAs per
    walker), and the same result a second time."""
    s = synth.with_pseudopotential(synth.water_system(m))
    R = walkers_at_edges(s, W, 11)
    g = Q.QMC(s, precision=prec, seed=9)
    Q.qmc_set_rng(g.h, 9, 2)
    g.set_walkers(R)
    e = g.eval_cached()["eloc"]
    ref = O.Oracle(s).evaluate(R, pp_seed=9, pp_sweep=2)["eloc"]
    assert rel(e, ref) <= tol, rel(e, ref)
    assert np.array_equal(e, g.eval_cached()["eloc"])
    g.close()
