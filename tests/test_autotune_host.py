"""The autotuner's cache: options found under another schedule of the pool are not applied,
those found under this one are, without a launch."""
import json
import types

import pytest

from paper_1201_3588_gb300 import autotune


class Measured(Exception):
    pass


def _grid():
    def launch(*a, **k):
        raise Measured
    tree = types.SimpleNamespace(max_level=2)
    return types.SimpleNamespace(N=1000, S=2, B=100, model=types.SimpleNamespace(tree=tree),
                                 n_total=10, transport=launch, reset=launch)


@pytest.fixture
def no_gpu(monkeypatch):
    import torch
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: None)
    monkeypatch.setattr(autotune.rt, "Batch", lambda *a, **k: _grid().transport())


def test_options_of_another_schedule_are_measured_again(tmp_path, no_gpu):
    path, g = tmp_path / "cache.json", _grid()
    opts = {"blocks_per_sm": 5, "threads": 256, "interaction_batch": 12, "refill_period": 16,
            "walk": 1}
    # keys as the packages-bound-to-lanes schedule wrote them
    key = autotune.workload_key(g, 30.0)
    old = key[key.index("cells2^"):]
    batch = autotune.batch_key([g], [30.0], [10])
    h = 0
    for ch in old.encode():
        h = (h * 131 + ch) % (1 << 61)
    path.write_text(json.dumps({old: {"opts": opts}, f"batch1-pk2^3-{h:016x}": {"opts": opts}}))
    with pytest.raises(Measured):
        autotune.tune(g, 30.0, cache=str(path))
    with pytest.raises(Measured):
        autotune.tune_batch([g], [30.0], [10], cache=str(path))
    path.write_text(json.dumps({key: {"opts": opts}, batch: {"opts": opts}}))
    assert autotune.tune(g, 30.0, cache=str(path)) == opts
    assert autotune.tune_batch([g], [30.0], [10], cache=str(path)) == opts
