"""FP64 ionic derivatives of large determinants against the oracle (the digit
GEMMs from 65 electrons per spin, the fused kernel's limb products below and on
request): walkers as drawn, with an electron of each spin 6 to 12 bohr out, and
orbitals scaled by powers of ten.  Bound: the FP64 path's 1e-10 of the larger of
1 and a walker's largest derivative."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["gemm", "fused"])
@pytest.mark.parametrize("m,kind", [(6, "far"), (14, "near"), (14, "far"), (14, "scaled"), (20, "far")])
def test_against_the_oracle(m, kind, path, monkeypatch):
    from paper_2504_07948_gb300 import qmc as Q
    monkeypatch.setenv("QMC_FORCE_GEMM_MIN_N", "1" if path == "gemm" else "1000")
    s = synth.water_system(m)
    W = 4
    R = synth.initial_walkers(s, W, seed=60 + m)
    if kind == "far":
        rng = np.random.default_rng(m)
        for w in range(W):
            for i in (rng.integers(s.n_up), s.n_up + rng.integers(s.n_dn)):
                v = rng.normal(size=3)
                R[w, i] += v / np.linalg.norm(v) * rng.uniform(6.0, 12.0)
    ref = O.Oracle(s).forces(R)   # (the derivatives do not change with the orbitals' scales)
    if kind == "scaled":
        s = s.copy()
        s.C = s.C * (10.0 ** np.linspace(-9, 9, s.n_mo))[:, None]
    g = Q.QMC(s, precision="fp64")
    g.set_walkers(R)
    pw = g.forces()[1]
    g.close()
    for c in range(2):
        scale = np.maximum(1.0, np.abs(ref[c]).max(axis=(1, 2), keepdims=True))
        assert np.all(np.abs(pw[:, c] - ref[c]) <= 1e-10 * scale)
