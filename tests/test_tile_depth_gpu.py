"""The step kernel's two-cell groups and layer variants, and the rule that
picks the depth of its work items, at the sizes where they can go wrong.

Against the FP64 oracle in parity mode the bars are the parity suite's
(fields 1e-5, probes 1e-4): 20 steps of FP32 arithmetic on coefficients the
oracle rounds alike stay two orders below them.  Results do not depend on the
depth, alone or in a batch, so those comparisons are bit for bit.
"""
import numpy as np
import pytest

from paper_2207_06908_gb300 import workloads as W
from test_parity_gpu import compare, fdtd, run_gpu, run_oracle  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu

STEPS = 20
# (nx, ny, nz), CPML cells: the smallest grid of a layer (its two x layers two
# cells apart), an odd layer or side (pairs cut by the layer or the wall),
# tile edges (32 x 16) and one cell past them, layers that start inside a tile
CASES = [((10, 10, 10), 4), ((8, 8, 8), 3), ((12, 13, 12), 5), ((33, 17, 18), 3), ((31, 15, 19), 4), ((32, 16, 16), 7),
         ((64, 32, 20), 8), ((65, 33, 23), 5), ((34, 49, 21), 6), ((97, 18, 14), 6), ((4, 3, 5), 0), ((33, 16, 9), 0),
         ((31, 47, 40), 0)]


def scenario(n, d, seed=3):
    room = min(n) - 2 * d > 4
    return W.random_scenario(seed, n=n, cpml=d, n_steps=STEPS, n_wires=1 if room else 0, n_sources=1 if room else 0,
                             n_blocks=3, n_mat=3)


@pytest.mark.parametrize("n,d", CASES)
def test_edges_against_oracle(fdtd, n, d):  # noqa: F811
    sc = scenario(n, d)
    compare(*run_gpu(fdtd, sc, STEPS), *run_oracle(sc, STEPS), steps=STEPS)


def fields_after(fdtd, sc, block, steps):  # noqa: F811
    g = fdtd.from_scenario(sc, probe_capacity=steps, block=block)
    for c, f in enumerate(sc.fields):
        g.set_field(c, f)
    g.step(steps)
    out = [g.get_field(c) for c in range(6)]
    g.close()
    return out


@pytest.mark.parametrize("n,d", [((40, 24, 30), 5), ((64, 64, 64), 8), ((48, 48, 48), 0), ((100, 70, 40), 4),
                                 ((160, 96, 80), 10)])
def test_depth_does_not_change_results(fdtd, n, d):  # noqa: F811
    """the chosen depth (one CTA per SM, one wave, several waves) against 16
    and 3 planes per item"""
    sc = scenario(n, d, seed=5)
    ref = fields_after(fdtd, sc, 16, 8)
    for block in (0, 3):
        for a, b in zip(ref, fields_after(fdtd, sc, block, 8)):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("copies", [1, 3, 12])
def test_batch_depth_does_not_change_results(fdtd, copies):  # noqa: F811
    """domains whose caller set a depth beside domains whose caller set none,
    in batches that fill the chip differently"""
    scs = [scenario((40 + 3 * (q % 3), 30 + q % 5, 26), 4, seed=9 + q) for q in range(copies)]
    grids = []
    for q, sc in enumerate(scs):
        g = fdtd.from_scenario(sc, probe_capacity=8, block=0 if q % 2 == 0 else 7)
        for c, f in enumerate(sc.fields):
            g.set_field(c, f)
        grids.append(g)
    b = fdtd.Batch(grids)
    b.step(7)
    b.synchronize()
    for sc, g in zip(scs, grids):
        for c, ref in enumerate(fields_after(fdtd, sc, 16, 7)):
            assert np.array_equal(g.get_field(c), ref)
    b.close()
    for g in grids:
        g.close()
