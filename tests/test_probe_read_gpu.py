"""Probe reads around the size of a staging block (64 KB, 64 bytes of it for
the flags: 16368 samples), where a read takes a second copy."""
import threading

import numpy as np
import pytest

from paper_2207_06908_gb300 import workloads as W
from test_parity_gpu import fdtd  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu

STEPS = 16500


def grid(F):
    sc = W.random_scenario(5, n=(9, 8, 7), n_wires=0, n_sources=1, n_probes=2, n_steps=64)
    g = F.from_scenario(sc, probe_capacity=STEPS)
    for c, f in enumerate(sc.fields):
        g.set_field(c, f)
    return g


def test_read_sizes(fdtd):  # noqa: F811
    g = grid(fdtd)
    g.step(STEPS)
    for p in range(2):
        parts = np.concatenate([g.read_probe(p, q, min(1000, STEPS - q)) for q in range(0, STEPS, 1000)])
        assert np.any(parts)
        for n in (0, 1, 16367, 16368, 16369, STEPS):
            assert np.array_equal(g.read_probe(p, STEPS - n, n), parts[STEPS - n:])
    g.close()


def test_reads_from_threads_and_after_the_last_grid(fdtd):  # noqa: F811
    g = grid(fdtd)
    g.step(50)
    want = g.read_probe(0, 0, 50)
    g.close()                        # the staging blocks go back with the process's last grid
    gs = [grid(fdtd) for _ in range(12)]
    got = [None] * len(gs)

    def work(q):
        gs[q].step(50)
        got[q] = gs[q].read_probe(0, 0, 50)

    ts = [threading.Thread(target=work, args=(q,)) for q in range(len(gs))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for g, r in zip(gs, got):
        g.close()
        assert np.array_equal(r, want)
