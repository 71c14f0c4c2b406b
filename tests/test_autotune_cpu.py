"""The tuner's choices on a model whose times are given: no GPU, a stand-in for the library."""
import contextlib
from types import SimpleNamespace

import pytest

torch = pytest.importorskip("torch")

from paper_2209_13443_b200 import autotune, binding


class Model:
    """One stage: an expand layer and the depthwise layer behind it, one launch until the expand layer has an entry."""

    n_stages = 1

    def __init__(self, cost):
        self.cost, self.variant, self.timed = cost, {}, 0

    def entries(self):
        return [v for v in self.variant.values() if v]

    def set_wait_limit(self, cycles):
        pass

    def layer_config(self, s, i, b):
        return {"variant": 0, "splits": 1, "tensor_core": 3 if i == 0 else -1}

    def set_layer_splits(self, s, i, n):
        if n > 1:
            raise binding.EEError(5, "one range")

    def set_layer_variant(self, s, i, lo, hi, v):
        assert i == 0
        for b in range(lo, hi + 1):
            self.variant[b] = v

    def plan(self, s, b):
        apart = bool(self.entries())
        return [{"launches": 1}, {"launches": int(apart)}]


class Timer:
    def __init__(self, m, spec):
        self.m = m

    def time(self, s, b):
        return self.m.cost(b, self.m.variant.get(b, 0), bool(self.m.entries()))


def tuned(monkeypatch, cost, batches=(1, 4, 16)):
    m = Model(cost)
    monkeypatch.setattr(binding, "EEModel", lambda spec, apply_tables: m)
    monkeypatch.setattr(autotune, "StageTimer", Timer)
    monkeypatch.setattr(torch.cuda, "Stream", lambda: None)
    monkeypatch.setattr(torch.cuda, "stream", lambda s: contextlib.nullcontext())
    layer = SimpleNamespace(kh=1, cin=16, cout=96, stride=1)
    spec = SimpleNamespace(stages=[SimpleNamespace(layers=[layer, layer])], max_batch=batches[-1])
    out, _ = autotune.tune(spec, list(batches), [1], verbose=False)
    return out[0]["variants"]


def test_an_entry_that_ends_a_shared_launch_counts_at_every_batch(monkeypatch):
    # variant 1 gains 10 % at batch 1; without the shared launch the larger batches lose 20 %
    def cost(b, v, apart):
        return 100.0 * b * (1.2 if apart and b > 1 else 1.0) * (0.9 if b == 1 and v == 1 else 1.0)

    assert tuned(monkeypatch, cost) == [0] * 16


def test_an_entry_that_gains_over_all_the_batches_it_touches_is_taken(monkeypatch):
    # variant 2 gains 30 % at batch 1, the others lose 1 % without the shared launch; from then on an entry touches its own batch only
    def cost(b, v, apart):
        return 100.0 * b * (1.01 if apart and b > 1 else 1.0) * (0.7 if b == 1 and v == 2 else 1.0) * (0.9 if b == 16 and v == 1 else 1.0)

    assert tuned(monkeypatch, cost) == [2, 0, 0, 0] + [1] * 12
