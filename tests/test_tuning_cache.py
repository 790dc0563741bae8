"""The cache of tuned depths: an entry measured with other kernels is not
reused, one of these kernels is (no GPU: building the first timed grid is
where a new measurement begins)."""
import json

import pytest

from paper_2207_06908_gb300 import grounding as G


class Measures(Exception):
    pass


@pytest.fixture
def cache(tmp_path, monkeypatch):
    def build(*a, **k):
        raise Measures
    monkeypatch.setattr(G, "_CACHE", str(tmp_path / "tuning.json"))
    monkeypatch.setattr(G.fdtd, "from_scenario", build)
    return tmp_path / "tuning.json"


@pytest.mark.parametrize("key", ["ground_batch_n64", "ground_batch_n64_0123456789abcdef"])
def test_entry_of_other_kernels(cache, key):
    cache.write_text(json.dumps({key: 16}))
    with pytest.raises(Measures):
        G.tune_block(64)


def test_entry_of_these_kernels(cache):
    cache.write_text(json.dumps({G._key(64): 24}))
    assert G.tune_block(60) == 24
    with pytest.raises(Measures):
        G.tune_block(65)
