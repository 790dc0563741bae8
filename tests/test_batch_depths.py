"""Depths of the package's own batches: tuned ones only where they leave every
SM a work item, the library's choice in smaller batches (and no tuning where
no candidate could)."""
import numpy as np
import pytest

from paper_2207_06908_gb300 import grounding as G, workloads as W


class Domain:
    def __init__(self, m, cpml=8):
        self.n, self.cpml = (m, m, m), cpml


# 64^3 with 8 cells: 8 column tiles, one item of 48 planes each
@pytest.mark.parametrize("sides,want", [([64] * 2, [0] * 2), ([64] * 18, [0] * 18), ([64] * 19, [48] * 19),
                                        ([64] * 64, [48] * 64), ([33] * 10 + [128] * 5, [48] * 10 + [32] * 5),
                                        ([128], [0]), ([128] * 2, [32] * 2)])
def test_tuned_where_every_sm_has_an_item(monkeypatch, sides, want):
    monkeypatch.setattr(G, "_sms", lambda: 152)
    monkeypatch.setattr(G, "tune_block", lambda n: 32 if n > 96 else 48)
    assert G.depths([Domain(m) for m in sides]) == want


def test_small_batches_are_not_tuned(monkeypatch):
    def tune(n):
        raise AssertionError("tuned")
    monkeypatch.setattr(G, "_sms", lambda: 152)
    monkeypatch.setattr(G, "tune_block", tune)
    assert G.depths([Domain(64)] * 3) == [0] * 3


@pytest.mark.gpu
def test_two_domains_run_at_the_librarys_depth():
    """the re-run of two rejected surrogate inputs: the tuned depth of full
    batches took more than three times as long"""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    scs = [W.surrogate_domain(W.surrogate_inputs(s)) for s in (3, 4)]
    ms, waves = {}, {}
    for tuned in (False, True, False, True):
        t = {}
        waves[tuned], _ = G.run_batch(scs, tuned=tuned, timings=t)
        ms[tuned] = min(ms.get(tuned, 1e9), t["device_ms"])
    assert np.array_equal(waves[False], waves[True])
    assert ms[True] <= 1.3 * ms[False], ms
