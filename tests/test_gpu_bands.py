"""Partitions with long chunks whose keys tie with runs of splitters (ties placed
by the runs' bands in the chunk), against the oracle: one value, a few values in
random order (no band is constant) and in runs, a mix with distinct keys, float64,
keys that are not 16-byte aligned, and without tie-breaks."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# chunks of 8192 keys and more on 152 SMs; odd, so the last chunk is short
N = 2_700_001


@pytest.fixture(scope="module")
def ctx():
    from paper_1606_08766_gb300 import Context
    c = Context(0)
    yield c
    c.close()


def _keys(name):
    rng = np.random.default_rng(3)
    if name == "one":
        return np.full(N, 77, dtype=np.uint64)
    if name == "top":
        return np.full(N, 2**64 - 1, dtype=np.uint64)
    if name == "few":
        return rng.integers(0, 5, N).astype(np.uint64) << np.uint64(40)
    if name == "runs":
        return np.repeat(rng.integers(0, 16, N // 999 + 1), 999)[:N].astype(np.uint64) << np.uint64(50)
    keys = rng.integers(0, 2**63, N).astype(np.uint64)
    keys[rng.random(N) < 0.5] = 12345 << 40
    return keys


@pytest.mark.parametrize("tie_break", [True, False])
@pytest.mark.parametrize("k", [64, 1000])
@pytest.mark.parametrize("name", ["one", "top", "few", "runs", "mix"])
def test_bands_match_oracle(ctx, oracle_mod, name, k, tie_break):
    keys = _keys(name)
    ref = oracle_mod.partition_ex(keys, k, seed=6, tie_break=tie_break, over=1)
    t = torch.from_numpy(keys.view(np.int64).copy()).cuda()
    ko, po, off, _, _ = ctx.partition_ex(t, k, seed=6, tie_break=tie_break)
    torch.cuda.synchronize()
    assert np.array_equal(off.cpu().numpy().astype(np.uint64), ref["offsets"])
    assert np.array_equal(po.cpu().numpy().view(np.uint32), ref["pos_out"])
    assert np.array_equal(ko.cpu().numpy().view(np.uint64), ref["keys_out"])
    ctx.check()


@pytest.mark.parametrize("shift", [0, 1])
def test_bands_f64_and_unaligned_keys(ctx, oracle_mod, shift):
    rng = np.random.default_rng(4)
    vals = np.where(rng.random(N) < 0.3, rng.standard_normal(N), rng.integers(-3, 3, N) * 0.5)
    ref = oracle_mod.partition_ex(vals.view(np.uint64), 300, seed=4, key_type=oracle_mod.KEY_F64,
                                  tie_break=True, over=1)
    t = torch.empty(N + shift, dtype=torch.float64, device="cuda")[shift:]
    t.copy_(torch.from_numpy(vals))
    ko, po, off, _, _ = ctx.partition_ex(t, 300, seed=4)
    torch.cuda.synchronize()
    assert np.array_equal(off.cpu().numpy().astype(np.uint64), ref["offsets"])
    assert np.array_equal(po.cpu().numpy().view(np.uint32), ref["pos_out"])
    assert np.array_equal(ko.cpu().numpy().view(np.uint64), ref["keys_out"].view(np.uint64))
    ctx.check()
