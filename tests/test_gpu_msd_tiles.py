"""E_L of determinant expansions whose reference matrices take several tiles of
rows in the energy kernel (B_0 and A0^-1 by tiles of 1024 entries: 22 and 17 rows
of 45 and 60) and whose electrons' grad J is summed in parts, against the
oracle's determinant-by-determinant sum at the bound of the one-tile systems."""
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


@pytest.mark.parametrize("m,n_active", [(9, 7), (12, 12)])
def test_expansion_energy(Q, m, n_active):
    s = synth.with_multidet(synth.water_system(m), 60, n_active=n_active, max_exc=4, seed=6)
    R = synth.initial_walkers(s, 5, seed=14)
    g = Q.QMC(s, precision="fp64")
    g.set_walkers(R)
    e = g.evaluate()["eloc"]
    ref = O.Oracle(s).evaluate(R)["eloc"]
    rel = float((np.abs(e - ref) / np.maximum(1.0, np.abs(ref))).max())
    assert rel <= 1e-10, rel
    g.close()
