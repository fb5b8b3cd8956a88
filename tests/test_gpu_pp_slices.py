"""The non-local energy of a walker is the same to the last bit beside few and
many walkers: the kernel splits a walker over more CTAs when there are few, and
adds its electron-nucleus pairs in one order either way."""
import numpy as np
import pytest

from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tc", [("mixed", "1"), ("mixed", "0"), ("fp64", "1")])
def test_walkers_do_not_depend_on_their_number(precision, tc, monkeypatch):
    from paper_2504_07948_gb300 import qmc as Q
    monkeypatch.setenv("QMC_NLPP_TC", tc)
    monkeypatch.setenv("QMC_NLPP_TC_MIN_N", "1")
    s = synth.with_pseudopotential(synth.water_system(16))   # 128 valence electrons
    R = synth.initial_walkers(s, 1900, seed=12)
    out = []
    for W in (17, 300, 1900):
        g = Q.QMC(s, precision=precision, seed=7)
        g.set_walkers(R[:W])
        out.append(g.eval_cached()["eloc"][:17].copy())
        g.close()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
