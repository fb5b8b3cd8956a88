"""A call that runs out of device memory is refused with QMC_ERR_OOM and leaves
the handle usable: with memory back, the same call gives what it gives on a
fresh handle."""
import numpy as np
import pytest

from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


class Full:
    """Leaves about `room` bytes of device memory free."""

    def __init__(self, room):
        self.room = room

    def __enter__(self):
        import torch
        self.held = []
        torch.cuda.empty_cache()
        for block in (1 << 34, 1 << 31, 1 << 28, 1 << 25, 1 << 22):
            while torch.cuda.mem_get_info()[0] > self.room + block:
                self.held.append(torch.empty(block, dtype=torch.uint8, device="cuda"))
        return self

    def __exit__(self, *_):
        import torch
        self.held.clear()
        torch.cuda.empty_cache()


def refused(Q, f):
    with pytest.raises(Q.QmcError) as e:
        f()
    assert e.value.code == -8   # QMC_ERR_OOM


@pytest.mark.parametrize("room", [16 << 20, 96 << 20, 224 << 20])
@pytest.mark.parametrize("warp", [False, True])
def test_forces_of_large_determinants(room, warp):
    from paper_2504_07948_gb300 import qmc as Q
    s = synth.water_system(14)
    R = synth.initial_walkers(s, 256, seed=4)

    def handle():
        g = Q.QMC(s, precision="fp64", space_warp=warp)
        g.set_walkers(R)
        return g

    g = handle()
    with Full(room):
        refused(Q, g.forces)
        refused(Q, g.forces)
    a = g.forces()[1]
    g.close()
    g = handle()
    assert np.array_equal(a[:, 1], g.forces()[1][:, 1])
    g.close()


def test_tiled_sweep_that_could_not_grow():
    from paper_2504_07948_gb300 import qmc as Q
    s = synth.water_system(24)
    R = synth.initial_walkers(s, 2000, seed=6)
    out = []
    for full in (True, False):
        g = Q.QMC(s, precision="mixed", delay_rank=16, seed=9, cap_factor=1)
        g.set_walkers(R)
        if full:
            with Full(64 << 20):
                refused(Q, lambda: g.vmc(1, 0.02))
        g.vmc(1, 0.02)
        out.append(g.get_walkers()[0])
        g.close()
    assert np.array_equal(*out)
