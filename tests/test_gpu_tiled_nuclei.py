"""The tiled sweep takes systems of many nuclei (its CTAs keep their offsets in
shared memory, beyond 48 KB here): nuclei without charge, basis functions or
Jastrow term leave the moves as they are, bit for bit."""
import numpy as np
import pytest

from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


def test_many_nuclei(monkeypatch):
    from paper_2504_07948_gb300 import qmc as Q
    monkeypatch.setenv("QMC_SWEEP_TILED", "1")
    monkeypatch.setenv("QMC_SWEEP_TILED_MIN_N", "4")
    s = synth.water_system(4)
    R = synth.initial_walkers(s, 40, seed=31)
    out = []
    for extra in (0, 1800):
        t = s.copy()
        t.Z = np.r_[s.Z, np.zeros(extra)]
        t.a_en = np.r_[s.a_en, np.zeros(extra)]
        far = 60.0 + np.stack(np.meshgrid(np.arange(12.0), np.arange(12.0), np.arange(13.0), indexing="ij"), -1)
        t.R = np.concatenate([s.R, far.reshape(-1, 3)[:extra]])
        g = Q.QMC(t, precision="mixed", delay_rank=8, seed=4)
        g.set_walkers(R)
        g.vmc(2, 0.02)
        out.append(g.get_walkers()[0])
        g.close()
    assert not np.array_equal(out[0], R)
    assert np.array_equal(*out)
