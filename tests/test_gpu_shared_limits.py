"""Kernels' shared-memory limits belong to the device, not to a handle: a system
whose kernels need much must run beside, and after, one whose kernels need
little, in batches and on threads of their own."""
import threading

import numpy as np
import pytest

from paper_2504_07948_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("graph", [True, False])
def test_large_batch_runs_after_a_small_one_was_made(precision, graph):
    from paper_2504_07948_gb300 import qmc as Q

    def batch(sizes, W):
        members = []
        for i, m in enumerate(sizes):
            s = synth.water_system(m)
            g = Q.QMC(s, precision=precision, seed=3 + i, fixed_population=True, recompute_period=2)
            g.set_walkers(synth.initial_walkers(s, W, seed=i))
            members.append(g)
        b = Q.Batch(members)
        if not graph:
            b.set_options(use_graph=False)
        return b, members

    def close(b, members):
        b.close()
        for g in members:
            g.close()

    def run(b, members):
        b.dmc(3, 0.005, [-76.0] * len(members), forces_every=1)
        return [g.get_walkers()[0] for g in members]

    large = batch([12, 16], 8)
    small = batch([1, 1], 8)
    run(*small)
    got = run(*large)
    close(*small)
    close(*large)
    alone = batch([12, 16], 8)
    ref = run(*alone)
    close(*alone)
    assert all(np.array_equal(a, b) for a, b in zip(got, ref))


def test_sweeps_and_forces_on_threads(monkeypatch):
    import torch
    from paper_2504_07948_gb300 import qmc as Q
    monkeypatch.setenv("QMC_SWEEP_TILED", "1")
    monkeypatch.setenv("QMC_SWEEP_TILED_MIN_N", "4")
    sizes = [(4, 200, "mixed", 8), (16, 700, "mixed", 16), (2, 900, "mixed", 4), (14, 24, "fp64", 1), (1, 300, "fp64", 1)]
    systems = [synth.water_system(c[0]) for c in sizes]

    def run(i, out, errors):
        try:
            _, W, precision, k = sizes[i]
            stream = torch.cuda.Stream()
            g = Q.QMC(systems[i], precision=precision, delay_rank=k, seed=20 + i, stream=stream.cuda_stream)
            g.set_walkers(synth.initial_walkers(systems[i], W, seed=i))
            for _ in range(8):
                g.vmc(1, 0.02)
                f = g.forces()[1]
                g.evaluate()
            out[i] = (g.get_walkers()[0], f)
            g.close()
        except Exception as e:   # reported by the test
            errors.append((i, e))

    alone, together, errors = {}, {}, []
    for i in range(len(sizes)):
        run(i, alone, errors)
    threads = [threading.Thread(target=run, args=(i, together, errors)) for i in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i in range(len(sizes)):
        assert np.array_equal(alone[i][0], together[i][0]), sizes[i]
        assert np.array_equal(alone[i][1], together[i][1]), sizes[i]
