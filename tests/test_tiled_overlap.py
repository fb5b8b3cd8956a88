"""Overlapped launches of the walker-tiled sweep (programmatic dependent
launch of the accept kernels behind the orbital GEMM).

A grid launched this way may read what earlier grids wrote only after its own
grid_wait, so ahead of it the accept kernels may touch constants and random
numbers alone.  One chain of launches (overlapped) and several groups on their
streams (plain launches) do the same arithmetic per walker: positions and state
agree bit for bit.  Kernel timing stays off here: its events between the
launches would keep them apart.
"""
import os
import re

import numpy as np
import pytest

from paper_2504_07948_gb300 import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_07948_gb300", "csrc")


def _strip(text):
    return re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", text), flags=re.S)


@pytest.mark.parametrize("kernel", ["k_tiled_accept", "k_tiled_accept_propose"])
def test_nothing_mutable_is_read_ahead_of_the_wait(kernel):
    src = _strip(open(os.path.join(CSRC, "k_sweep_tiled.cu")).read())
    body = re.search(r"__global__[^;{]*\b" + kernel + r"\([^{]*\{(.*?)\n\}", src, re.S).group(1)
    assert "grid_wait();" in body, "no wait in the kernel itself"
    ahead = body.split("grid_wait();")[0]
    assert not re.search(r"\bts\b|\bwk\b", ahead), ahead
    # and the helpers called there see neither the walkers nor the sweep's state
    for f in re.findall(r"\b(tiled_\w+)\(", ahead):
        args = re.search(r"\b" + f + r"\(([^)]*)\)\s*\{", src).group(1)
        assert "TiledState" not in args and "DevWalkers" not in args, (f, args)


@pytest.mark.gpu
@pytest.mark.parametrize("m,k,W,groups", [(4, 8, 600, 2), (4, 8, 1100, 3), (8, 32, 2500, 4), (32, 32, 600, 2)])
def test_overlapped_chain_matches_plain_launches(monkeypatch, m, k, W, groups):
    """Three sweeps; walker counts with a ragged last group, fewer and more than
    the resident CTAs (152 x 8)."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2504_07948_gb300 import qmc as Q
    s = synth.water_system(m)
    R = synth.initial_walkers(s, W, seed=300 + m)
    monkeypatch.setenv("QMC_SWEEP_TILED", "1")
    monkeypatch.setenv("QMC_SWEEP_TILED_MIN_N", "4")
    out = []
    for g in ("1", str(groups)):
        monkeypatch.setenv("QMC_SWEEP_TILED_GROUPS", g)
        h = Q.QMC(s, precision="mixed", seed=61, delay_rank=k)
        h.set_walkers(R)
        h.vmc(3, 0.02)
        out.append((h.get_walkers()[0], h.eval_cached()))
        h.close()
    a, b = out
    assert not np.array_equal(a[0], R)
    assert np.array_equal(a[0], b[0])
    for key in ("logpsi", "eloc"):
        assert np.array_equal(a[1][key], b[1][key]), key
