"""Reciprocals of the mixed form's Jastrow terms in the local energy are
rounded once.

u = r / (1 + b r) with r a power of two and b a multiple of 2^-19 below 2^-4:
b r and 1 + b r are exact in FP32, and so is the product with r, so u carries
the rounding of the division alone, at most 2^-24 of it.  ln|psi| with and
without the term differ by u, their determinant part being FP64."""
import numpy as np
import pytest

from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pair", ["electrons", "nucleus"])
def test_pair_reciprocal_is_correctly_rounded(pair):
    from paper_2504_07948_gb300 import qmc as Q
    ee = pair == "electrons"
    i0 = np.zeros(1, dtype=np.int32)
    s = synth.System(Z=np.ones(1), R=np.zeros((1, 3)), n_up=1, n_dn=int(ee), shell_center=i0, shell_l=i0, shell_pure=i0,
                     shell_nprim=i0 + 1, alpha=np.array([0.02]), coef=np.ones(1), C=np.ones((1, 1)), occ_up=i0,
                     occ_dn=i0 if ee else i0[:0], a_anti=0.0, a_par=0.0, b_ee=1.0, a_en=np.zeros(1), b_en=1.0)
    r = 2.0 ** np.arange(-4, 5)
    if ee:
        R = np.zeros((len(r), 2, 3))
        R[:, :, 2] = 0.5
        R[:, 1, 0] = r
    else:
        R = np.zeros((len(r), 1, 3))
        R[:, 0, 0] = r

    def logpsi(a, b):
        t = s.copy()
        t.a_anti, t.a_en, t.b_ee, t.b_en = (a, np.zeros(1), b, 1.0) if ee else (0.0, np.array([a]), 1.0, b)
        g = Q.QMC(t, precision="mixed")
        g.set_walkers(R)
        out = g.evaluate()["logpsi"].copy()
        g.close()
        return out

    rng = np.random.default_rng(4)
    for i in rng.integers(1, 1 << 15, size=60):
        b = float(i) * 2.0 ** -19
        u = logpsi(1.0, b) - logpsi(0.0, b)
        ref = r / (1.0 + b * r)
        assert np.all(np.abs(u - ref) <= 2.0 ** -24 * ref + 1e-13), (b, (np.abs(u - ref) / ref).max() * 2 ** 24)
