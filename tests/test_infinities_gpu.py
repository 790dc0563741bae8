"""How an infinity spreads in grids with an absorbing layer: one step moves it
by one cell, and a lane of a tile that meets a layer but lies outside it gives
what it gives anywhere else.

One component of one cell is set to infinity in a vacuum grid of small random
fields.  After one step the cells that hold a NaN, and after one and two steps
those that hold a NaN or an infinity, are the FP64 oracle's (the cell is at
least four away from the walls, so no wall coefficient of zero meets it).
E on the node where a high layer begins (depth 0, coefficients one and zero)
counts to the layer here and not in the oracle: there an infinite difference
may be a NaN, and those nodes are left out of the comparison of NaNs."""
import numpy as np
import pytest

from oracle.oracle import OracleGrid
from paper_2207_06908_gb300 import workloads as W
from test_parity_gpu import fdtd  # noqa: F401 (fixture)

# (sides, layer, block, component, cell): rows of a tile outside its y layer
# (the tile's first layer row holds the infinity), cells on both sides of the
# x layers in whole pairs and in pairs cut by the layer, planes above and
# below a work item of 4 planes
CASES = [((64, 48, 40), 6, 0, c, at) for c, at in
         [(2, (20, 43, 20)), (0, (20, 42, 20)), (5, (20, 42, 19)), (2, (10, 20, 20)), (1, (58, 20, 20)),
          (2, (57, 20, 20)), (2, (20, 8, 20)), (3, (20, 41, 20)), (4, (9, 20, 20)), (0, (30, 30, 34))]]
CASES += [((63, 48, 41), 5, 4, c, (x, y, z)) for c in (1, 2, 4) for x, y, z in
          [(4, 20, 8), (5, 20, 9), (57, 20, 12), (58, 20, 13), (20, 43, 17), (20, 42, 16)]]


def scenario(n, d):
    sc = W.random_scenario(11, n=n, cpml=d, n_steps=4, n_wires=0, n_sources=0, n_probes=1, n_blocks=1, n_mat=1)
    sc.cell_material = np.zeros_like(sc.cell_material)
    sc.materials = [(1.0, 0.0, 1.0)]
    return sc


def fields_of(sc, comp, at):
    fs = [np.array(f, np.float32) for f in sc.fields]
    fs[comp][at[2], at[1], at[0]] = np.inf
    return fs


def oracle_steps(sc, fs, steps):
    o = OracleGrid(*sc.n, sc.dx, courant=sc.courant, parity=True)
    o.set_cpml(sc.cpml)
    o.set_materials(sc.cell_material, [1.0], [0.0], [1.0])
    o.finalize(steps)
    for c, f in enumerate(fs):
        o.set_field(c, f.astype(np.float64))
    o.step(steps)
    return [o.get_field(c) for c in range(6)]


@pytest.mark.gpu
@pytest.mark.parametrize("n,d,block,comp,at", CASES)
def test_spread_is_the_oracles(fdtd, n, d, block, comp, at):  # noqa: F811
    sc = scenario(n, d)
    fs = fields_of(sc, comp, at)
    for steps in (1, 2):
        g = fdtd.from_scenario(sc, probe_capacity=4, block=block)
        for c, f in enumerate(fs):
            g.set_field(c, f)
        g.step(steps)
        got = [g.get_field(c) for c in range(6)]
        g.close()
        want = oracle_steps(sc, fs, steps)
        for c in range(6):
            assert np.array_equal(np.isfinite(got[c]), np.isfinite(want[c])), (steps, c)
            if steps == 1:
                inner = np.ones(got[c].shape, bool)
                for axis, m in enumerate(reversed(n)):
                    if c < 3:
                        inner[(slice(None),) * axis + (m - d,)] = False
                assert np.array_equal(np.isnan(got[c])[inner], np.isnan(want[c])[inner]), c
