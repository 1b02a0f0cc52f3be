"""Partitions whose chunks are long enough for ties to be placed by bands (8192 keys
and more, one segment), in every form of the classify that does so: uint64 and
float64 keys, 16-byte aligned and not; against the oracle."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SUBTILE, FINE_TILE, BAND_MIN = 4096, 6144, 8192


@pytest.fixture(scope="module")
def ctx():
    from paper_1606_08766_gb300 import Context
    c = Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def n():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    size = 6 * sms * FINE_TILE + 1      # odd: the last chunk is short
    # six chunks an SM from six scatter sub-tiles an SM on, in whole sub-tiles
    assert size > 5 * sms * FINE_TILE
    chunk = -(-(-(-size // (6 * sms))) // SUBTILE) * SUBTILE
    assert chunk >= BAND_MIN
    return size


def _keys(name, n):
    rng = np.random.default_rng(3)
    if name == "top":
        return np.full(n, 2**64 - 1, dtype=np.uint64)
    if name == "few":
        return rng.integers(0, 5, n).astype(np.uint64) << np.uint64(40)
    if name == "runs":
        return (np.repeat(rng.integers(0, 16, n // 999 + 1), 999)[:n].astype(np.uint64)
                << np.uint64(50))
    if name == "mix":
        keys = rng.integers(0, 2**63, n).astype(np.uint64)
        keys[rng.random(n) < 0.5] = 12345 << 40
        return keys
    # float64: a few values among distinct ones, or with the values floats have besides
    x = np.where(rng.random(n) < 0.3, rng.standard_normal(n), rng.integers(-3, 3, n) * 0.5)
    if name == "f64_special":
        for v in (0.0, -0.0, np.inf, -np.inf, np.nan):
            x[rng.random(n) < 0.1] = v
    return x


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("name,k", [("top", 64), ("few", 300), ("runs", 100), ("mix", 1000),
                                    ("f64", 300), ("f64_special", 100)])
def test_long_chunks_match_oracle(ctx, oracle_mod, n, name, k, shift):
    keys = _keys(name, n)
    kt = 1 if keys.dtype == np.float64 else 0
    ref = oracle_mod.partition_ex(keys, k, seed=6, key_type=kt, over=1)
    t = torch.empty(n + shift, dtype=torch.int64, device="cuda")[shift:]
    t.copy_(torch.from_numpy(keys.view(np.int64)))
    ko, po, off, _, _ = ctx.partition_ex(t, k, seed=6, key_type=kt)
    torch.cuda.synchronize()
    assert np.array_equal(off.cpu().numpy().astype(np.uint64), ref["offsets"])
    assert np.array_equal(po.cpu().numpy().view(np.uint32), ref["pos_out"])
    assert np.array_equal(ko.cpu().numpy().view(np.uint64), ref["keys_out"].view(np.uint64))
    ctx.check()
