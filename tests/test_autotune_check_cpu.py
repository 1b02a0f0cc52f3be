"""The autotuner's last pass (no GPU): a table that is faster on the batches its
knobs were timed on, and slower on a batch of more than 2^27 keys, is given up."""

import pytest

torch = pytest.importorskip("torch")


class _FakeCtx:
    def __init__(self, device):
        self.knobs = {}

    def __enter__(self):
        return self

    def __exit__(self, *a):
        pass

    def set_tunable(self, name, v):
        self.knobs[name] = v

    def get_tunable(self, name):
        return {"target_bucket": 1536, "small_cap": 1024, "mid_cap": 2048,
                "rank_max": 64}.get(name, 0)


@pytest.mark.parametrize("loss,reverted", [(0.2, True), (-0.2, False)])
def test_table_that_loses_on_large_batches_is_reverted(monkeypatch, loss, reverted):
    from paper_1606_08766_gb300 import autotune

    def time_batches(ctx, batches, reps):
        # a batch is its key count and offsets; a smaller cap pays below 2^27 keys only
        cap = ctx.knobs.get("small_cap", 1024)
        return sum(10 + loss if n > 1 << 27 and cap != 1024 else
                   10 if n > 1 << 27 else 1 - (1024 - cap) / 10240 for n, _ in batches)

    monkeypatch.setattr(autotune, "Context", _FakeCtx)
    monkeypatch.setattr(autotune.torch.cuda, "device", lambda d: _FakeCtx(d))
    monkeypatch.setattr(autotune.torch.cuda, "empty_cache", lambda: None)
    monkeypatch.setattr(autotune, "segment_batch",
                        lambda lo, hi, total, seed, device: (total, torch.zeros(2)))
    monkeypatch.setattr(autotune, "_batches", lambda specs: list(specs))
    monkeypatch.setattr(autotune, "_time_batches", time_batches)
    monkeypatch.setattr(autotune, "DEFAULT_CLASSES", ())
    r = autotune.tune(0, classes=())
    assert r.reverted is reverted
    assert (r.tuned_ms > r.default_ms) is reverted
    assert r.table()["small_cap"] == (1024 if reverted else 256)
