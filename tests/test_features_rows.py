"""surrogate.features encodes all rows at once: the same values as the domain
builder's cells, row by row, at halves, below zero and for no rows at all; a
value that has no cell raises what the builder raises."""
import numpy as np
import pytest

from paper_2207_06908_gb300 import surrogate as S, workloads as W


def test_rows_match_the_builder():
    r = np.random.default_rng(4)
    p = np.stack([r.uniform(-5, 50, 3000), r.uniform(-5, 0, 3000), r.uniform(-3, 12, 3000), r.uniform(1e-3, 2e-2, 3000),
                  r.uniform(-2, 3, 3000), r.uniform(0, 1e-6, 3000)], axis=1)
    p[:1000, 2] = np.arange(1000) * 0.125 - 3          # halves of a cell among them
    p[:1000, 4] = np.arange(1000) * 0.125 - 50
    F = S.features(p)
    cells = np.array([W.grounding_cells(l, d) for l, d in p[:, [2, 4]]], np.float64) * W.GROUND_DX
    assert np.array_equal(F[:, 2], ((cells[:, 0] - 5.0) / 4.0).astype(np.float32))
    assert np.array_equal(F[:, 4], ((cells[:, 1] - 0.5) / 0.5).astype(np.float32))
    assert np.array_equal(S.features(p[7]), F[7:8])
    assert S.features(np.zeros((0, 6))).shape == (0, 6)


@pytest.mark.parametrize("value,error", [(np.nan, ValueError), (np.inf, OverflowError), (-np.inf, OverflowError)])
@pytest.mark.parametrize("column", [2, 4])
def test_no_cell(column, value, error):
    p = np.ones((3, 6))
    p[1, column] = value
    with pytest.raises(error):
        S.features(p)
