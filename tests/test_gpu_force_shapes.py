"""Ionic derivatives of the per-walker force kernel at the edges of its
shapes: spin blocks of 1 to 35 electrons (one and two warps of electrons,
partial row groups), unequal and empty spins, tiles of the whole basis and of
32 functions, and a determinant too large to stage, against the oracle or the
GEMM force path."""
import numpy as np
import pytest

from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


def _cut(m, n_up, n_dn):
    s = synth.water_system(m).copy()
    s.n_up, s.n_dn = n_up, n_dn
    s.occ_up, s.occ_dn = np.arange(n_up, dtype=np.int32), np.arange(n_dn, dtype=np.int32)
    return s


@pytest.mark.parametrize("m,n_up,n_dn", [(1, 1, 0), (1, 5, 4), (2, 8, 3), (5, 20, 11), (7, 32, 31), (7, 33, 35)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_force_shapes_against_oracle(m, n_up, n_dn, precision):
    from oracle import oracle as O
    from paper_2504_07948_gb300 import qmc as Q
    s = _cut(m, n_up, n_dn)
    R = synth.initial_walkers(s, 3, seed=11 + n_up)
    g = Q.QMC(s, precision=precision)
    g.set_walkers(R)
    _, pw = g.forces()
    g.close()
    dEL, dlg = O.Oracle(s).forces(R)
    # the path's tolerances: 1e-10 (FP64) and 1e-2 (mixed) of the larger of 1 and
    # the derivative, the mixed form's taken on each walker's largest component
    for got, ref in ((pw[:, 0], dEL), (pw[:, 1], dlg)):
        if precision == "fp64":
            assert np.all(np.abs(got - ref) <= 1e-10 * np.maximum(1.0, np.abs(ref).max(axis=(1, 2), keepdims=True)))
        else:
            assert np.all(np.abs(got - ref) <= 1e-2 * np.maximum(1.0, np.abs(ref).max(axis=(1, 2), keepdims=True)))


@pytest.mark.parametrize("m", [14, 20])
@pytest.mark.parametrize("warp", [False, True])
def test_fused_force_of_large_determinants_against_gemm_path(m, warp, monkeypatch):
    """70 electrons per spin (staged) and 100 (not staged) in the fused kernel."""
    from paper_2504_07948_gb300 import qmc as Q
    s = synth.water_system(m)
    R = synth.initial_walkers(s, 2, seed=5)
    out = []
    for min_n in ("65", "1000"):
        monkeypatch.setenv("QMC_FORCE_GEMM_MIN_N", min_n)
        g = Q.QMC(s, precision="fp64", space_warp=warp)
        g.set_walkers(R)
        out.append(g.forces()[1])
        g.close()
    scale = np.maximum(1.0, np.abs(out[0]).max(axis=(2, 3), keepdims=True))
    assert np.all(np.abs(out[1] - out[0]) <= 1e-10 * scale)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_gemm_force_path_with_fewer_down_electrons(precision, monkeypatch):
    """The two spins' weights M and Y must not share memory when n_dn < n_up."""
    from oracle import oracle as O
    from paper_2504_07948_gb300 import qmc as Q
    monkeypatch.setenv("QMC_FORCE_GEMM_MIN_N", "1")
    s = _cut(3, 16, 8)
    R = synth.initial_walkers(s, 3, seed=21)
    g = Q.QMC(s, precision=precision)
    g.set_walkers(R)
    _, pw = g.forces()
    g.close()
    for got, ref in zip((pw[:, 0], pw[:, 1]), O.Oracle(s).forces(R)):
        tol = 1e-10 if precision == "fp64" else 1e-2
        assert np.all(np.abs(got - ref) <= tol * np.maximum(1.0, np.abs(ref).max(axis=(1, 2), keepdims=True)))
