"""A grid of more than 2^31 cells per array: sources, fields and probes on both
sides of the plane that starts at element 2^31, against a small grid with the
same surroundings.  The cells a step reads spread by one a step, so over 24
steps neither grid's far walls are met and the probes agree bit for bit."""
import numpy as np
import pytest

from paper_2207_06908_gb300 import workloads as W
from test_parity_gpu import fdtd  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu

STEPS = 24


def traces(F, ny, nz, j, k):
    """3 x ny x nz cells between perfectly conducting walls, sources at (1, j, k) and a plane below"""
    t = np.arange(STEPS)
    sc = W.Scenario("tall", (3, ny, nz), 0.1, 0.99, 0, np.zeros((nz, ny, 3), np.uint8), [(1.0, 0.0, 1.0)],
                    sources=[((1, j, k), 2, np.sin(0.3 * t)), ((2, j + 1, k - 1), 0, np.cos(0.2 * t))],
                    probes=[(W.PROBE_E, (1 + a % 2, j + b, k + c), a, 1)
                            for a in range(3) for b in (-2, 0, 3) for c in (-3, -1, 0, 1, 2)] +
                           [(W.PROBE_I, (1, j + b, k + c), 2, 1) for b in (0, 2) for c in (-2, -1, 0, 1)])
    g = F.from_scenario(sc, probe_capacity=STEPS, torch_arena=False)
    g.step(STEPS)
    out = np.stack([g.read_probe(p, 0, STEPS) for p in range(len(sc.probes))])
    g.close()
    return out


def test_planes_around_element_2_31(fdtd):  # noqa: F811
    import torch
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 120e9:
        pytest.skip("needs 106 GB of device memory")
    # rows of 16 elements, 8192 to a plane: plane 16384 starts at element 2^31
    small, large = traces(fdtd, 64, 64, 30, 32), traces(fdtd, 8192, 16384 + 40, 4000, 16384)
    assert np.all(np.any(small != 0, axis=1))
    assert np.array_equal(small, large)
