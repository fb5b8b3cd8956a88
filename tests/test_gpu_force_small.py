"""FP64 ionic derivatives of the fused kernel on both sides of the size up to
which a spin's products are FP64 sums (16 electrons), the two forms within one
walker among them, plain and space-warped, against the oracle at the FP64
path's bound (1e-10 of the larger of 1 and a walker's largest derivative)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_up,n_dn", [(1, 1), (15, 3), (16, 16), (16, 17), (17, 16), (17, 1)])
@pytest.mark.parametrize("warp", [False, True])
def test_against_the_oracle(n_up, n_dn, warp):
    from paper_2504_07948_gb300 import qmc as Q
    s = synth.water_system(4).copy()
    s.n_up, s.n_dn = n_up, n_dn
    s.occ_up, s.occ_dn = np.arange(n_up, dtype=np.int32), np.arange(n_dn, dtype=np.int32)
    R = synth.initial_walkers(s, 5, seed=40 + n_up)
    g = Q.QMC(s, precision="fp64", space_warp=warp)
    g.set_walkers(R)
    pw = g.forces()[1]
    g.close()
    o = O.Oracle(s)
    ref = o.warped_forces(R) if warp else o.forces(R)
    for c in range(2):
        scale = np.maximum(1.0, np.abs(ref[c]).max(axis=(1, 2), keepdims=True))
        assert np.all(np.abs(pw[:, c] - ref[c]) <= 1e-10 * scale)
