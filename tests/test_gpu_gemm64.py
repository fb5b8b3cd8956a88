"""The FP64 force path of large determinants (bf16-digit GEMMs on the tensor
cores) at the edges of its tiles, against the fused force kernel: spins of
odd, equal-to-tile and unequal size, one walker and more than a chunk row
block, and walkers with an electron far out (rows of the inverse of very
different magnitude)."""
import numpy as np
import pytest

from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


def _both(s, R, monkeypatch, warp=False):
    from paper_2504_07948_gb300 import qmc as Q
    out = []
    for min_n in ("1", "1000"):
        monkeypatch.setenv("QMC_FORCE_GEMM_MIN_N", min_n)
        g = Q.QMC(s, precision="fp64", space_warp=warp)
        g.set_walkers(R)
        out.append(g.forces()[1])
        g.close()
    scale = np.maximum(1.0, np.abs(out[1]).max(axis=(2, 3), keepdims=True))
    return np.abs(out[0] - out[1]) / scale


@pytest.mark.parametrize("m,n_up,n_dn,W", [(1, 5, 4, 3), (3, 15, 7, 5), (7, 32, 33, 1), (13, 64, 65, 2),
                                           (14, 70, 63, 2), (26, 128, 129, 1)])
def test_against_the_fused_kernel(m, n_up, n_dn, W, monkeypatch):
    s = synth.water_system(m).copy()
    s.n_up, s.n_dn = n_up, n_dn
    s.occ_up, s.occ_dn = np.arange(n_up, dtype=np.int32), np.arange(n_dn, dtype=np.int32)
    assert _both(s, synth.initial_walkers(s, W, seed=70 + m), monkeypatch).max() <= 1e-10


def test_more_walkers_than_a_chunk(monkeypatch):
    s = synth.water_system(1)
    assert _both(s, synth.initial_walkers(s, 259, seed=3), monkeypatch, warp=True).max() <= 1e-10


def test_orbitals_and_electrons_of_different_magnitude(monkeypatch):
    """Orbitals scaled by powers of ten (the derivatives do not change) and an electron 6 bohr out."""
    s = synth.water_system(2)
    R = synth.initial_walkers(s, 4, seed=9)
    R[1, 0] += np.array([6.0, 0.0, 0.0])
    t = s.copy()
    t.C = s.C * (10.0 ** np.linspace(-9, 9, s.n_mo))[:, None]
    assert _both(t, R, monkeypatch).max() <= 1e-10
    from paper_2504_07948_gb300 import qmc as Q
    out = []
    for sy in (s, t):
        monkeypatch.setenv("QMC_FORCE_GEMM_MIN_N", "1")
        g = Q.QMC(sy, precision="fp64")
        g.set_walkers(R)
        out.append(g.forces()[1])
        g.close()
    scale = np.maximum(1.0, np.abs(out[0]).max(axis=(2, 3), keepdims=True))
    assert (np.abs(out[1] - out[0]) / scale).max() <= 1e-10
