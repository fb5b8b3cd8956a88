"""FP64 orbitals (listed basis, fixed-point contraction) at the edges of their
shapes: 1 to 130 orbitals per spin (16 to one lanes per orbital, one and two
rounds), every shell kind, bases of 6 functions and of too many for the
lists, and electrons far outside every shell, against the oracle."""
import numpy as np
import pytest

from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


def _cut(s, n_up, n_dn):
    s = s.copy()
    s.n_up, s.n_dn = n_up, n_dn
    s.occ_up, s.occ_dn = np.arange(n_up, dtype=np.int32), np.arange(n_dn, dtype=np.int32)
    return s


def _check(s, R):
    from oracle import oracle as O
    from paper_2504_07948_gb300 import qmc as Q
    g = Q.QMC(s, precision="fp64")
    g.set_walkers(R)
    got = g.evaluate()
    g.close()
    ref = O.Oracle(s).evaluate(R)
    for k in ("logpsi", "eloc"):
        assert np.all(np.abs(got[k] - ref[k]) <= 1e-10 * np.maximum(1.0, np.abs(ref[k]))), k
    scale = np.maximum(1.0, np.abs(ref["grad"]).max(axis=(1, 2), keepdims=True))
    assert np.all(np.abs(got["grad"] - ref["grad"]) <= 1e-10 * scale)


@pytest.mark.parametrize("m,n_up,n_dn", [(1, 1, 0), (1, 7, 5), (2, 9, 8), (3, 17, 16), (6, 33, 31), (13, 65, 64),
                                         (17, 130, 3)])
def test_orbital_counts(m, n_up, n_dn):
    s = _cut(synth.water_system(m), n_up, n_dn)
    _check(s, synth.initial_walkers(s, 3, seed=40 + m))


@pytest.mark.parametrize("seed", range(4))
def test_every_shell_kind(seed):
    rng = np.random.default_rng(seed)
    s = synth.random_small_system(rng, n_nuc=1 + seed, n_up=3, n_dn=2)
    _check(s, rng.normal(0.0, 1.0, size=(5, 5, 3)))


def test_screened_shells():
    """Tight shells only: an electron outside sees the diffuse function of the other centre alone."""
    s = synth.single_gaussian_atom(0.5, 1.0, 1, 0)
    t = s.copy()
    t.Z, t.R, t.a_en = np.array([1.0, 1.0]), np.array([[0.0, 0.0, 0.0], [9.0, 0.0, 0.0]]), np.zeros(2)
    t.shell_center, t.shell_l, t.shell_pure = (np.array(v, np.int32) for v in ([0, 1, 1], [0, 1, 2], [0, 0, 1]))
    t.shell_nprim = np.array([1, 1, 1], np.int32)
    t.alpha, t.coef = np.array([0.5, 300.0, 400.0]), np.ones(3)
    t.C = np.eye(9)
    _check(t, np.array([[[1.0, 0.2, -0.4]], [[8.9, 0.01, 0.02]], [[2.0, 0.0, 0.0]]]))


def test_basis_beyond_the_lists():
    """More functions than the lists hold: the plain contraction."""
    nb = 2700
    s = synth.single_gaussian_atom(0.5, 1.0, 1, 1)
    t = s.copy()
    rng = np.random.default_rng(2)
    t.shell_center, t.shell_l, t.shell_pure = np.zeros(nb, np.int32), np.zeros(nb, np.int32), np.zeros(nb, np.int32)
    t.shell_nprim = np.ones(nb, np.int32)
    t.alpha, t.coef = 10.0 ** rng.uniform(-1, 1, nb), np.ones(nb)
    t.C = rng.uniform(0.1, 1.0, size=(1, nb)) / nb
    _check(t, rng.normal(0.0, 0.7, size=(3, 2, 3)))
