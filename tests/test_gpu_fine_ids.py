"""Overpartitioned steps whose fine partition ids are stored once and mapped to
buckets, against the oracle: sizes on both sides of the rule that takes this
path (2048 elements a fine partition), odd chunk ends, runs of copies, with and
without tie-breaks, float64 and keys that are not 16-byte aligned."""

import numpy as np
import pytest
import torch

import instances

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1606_08766_gb300 import Context
    c = Context(0)
    yield c
    c.close()


def _compare(got, ref, what):
    ko, po, off, fine, first = got
    torch.cuda.synchronize()
    assert np.array_equal(off.cpu().numpy().astype(np.uint64), ref["offsets"]), what
    assert np.array_equal(fine.cpu().numpy().astype(np.uint64), ref["fine_sizes"]), what
    assert np.array_equal(first.cpu().numpy().astype(np.uint32), ref["group_first"]), what
    assert np.array_equal(po.cpu().numpy().view(np.uint32), ref["pos_out"]), what
    assert np.array_equal(ko.cpu().numpy().view(np.uint64), ref["keys_out"].view(np.uint64)), what


@pytest.mark.parametrize("name", ["uniform", "deter_dupl", "zero"])
@pytest.mark.parametrize("k,over", [(33, 2), (40, 5), (64, 10)])
def test_fine_ids_match_oracle(ctx, oracle_mod, name, k, over):
    for extra in (-1, 0, 1, 8191):
        n = 2048 * k * over + extra
        keys = instances.generate(name, n, p=1, seed=n)
        t = torch.from_numpy(np.ascontiguousarray(keys).view(np.int64)).cuda()
        for tb in (True, False):
            ref = oracle_mod.partition_ex(keys, k, seed=9, tie_break=tb, over=over)
            _compare(ctx.partition_ex(t, k, seed=9, tie_break=tb, overpartition=over), ref,
                     (n, tb))
    ctx.check()


@pytest.mark.parametrize("k,over", [(33, 2), (512, 10), (600, 10), (1024, 4)])
def test_small_steps_match_oracle(ctx, oracle_mod, k, over):
    for n in (1, 7, 9, 1023, 65551):
        keys = instances.generate("deter_dupl", n, p=1, seed=n)
        t = torch.from_numpy(np.ascontiguousarray(keys).view(np.int64)).cuda()
        ref = oracle_mod.partition_ex(keys, k, seed=9, tie_break=True, over=over)
        _compare(ctx.partition_ex(t, k, seed=9, overpartition=over), ref, n)
    ctx.check()


@pytest.mark.parametrize("shift", [0, 1])
def test_fine_ids_f64_and_unaligned_keys(ctx, oracle_mod, shift):
    n = 2048 * 160 + 3
    vals = np.random.default_rng(5).standard_normal(n)
    vals[::7] = vals[0]
    ref = oracle_mod.partition_ex(vals.view(np.uint64), 40, seed=4, key_type=oracle_mod.KEY_F64,
                                  over=4)
    t = torch.empty(n + shift, dtype=torch.float64, device="cuda")[shift:]
    t.copy_(torch.from_numpy(vals))
    _compare(ctx.partition_ex(t, 40, seed=4, overpartition=4), ref, shift)
    ctx.check()
