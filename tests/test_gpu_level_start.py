"""The start of a partition level: samples drawn and sorted by one launch,
sample chunks merged by ranges (two chunks and more, all samples of small
inputs, duplicates, sorted inputs), small and large histogram scans, and the
chunk sizes of small calls.  Partition layouts depend on every sample, so they
show a wrong one; sorts cover the deeper levels.
"""
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


def _dev(a):
    return torch.from_numpy(a.view(np.int64).copy()).cuda()


# 103 buckets: 11,536 samples in two chunks; 2048: 360,448 in 44
@pytest.mark.parametrize("n", [4097, 8193, 100_003, 262_145])
@pytest.mark.parametrize("k", [3, 16, 64, 102, 103, 700, 2048])
@pytest.mark.parametrize("name", ["uniform", "reverse", "rand_dupl", "zero"])
def test_partition_samples(ctx, oracle_mod, name, k, n):
    x = instances.generate(name, n, p=64, seed=n + k)
    ref = oracle_mod.partition(x, k, seed=k)
    ko, po, off = ctx.partition(_dev(x), k, seed=k)
    np.testing.assert_array_equal(off.cpu().numpy().astype(np.uint64), ref["offsets"])
    np.testing.assert_array_equal(po.cpu().numpy().view(np.uint32), ref["pos_out"])
    np.testing.assert_array_equal(ko.cpu().numpy().view(np.uint64), ref["keys_out"])
    ctx.check()


# one level with buckets above the target (four times the samples), the first
# sizes of two levels, and level-2 chunks of every size
@pytest.mark.parametrize("n,p", [(786_433, 1), (1_398_101, 1), (1_398_102, 1), (2_500_001, 1),
                                 (1 << 20, 16), (3_000_017, 600), (5_000_011, 2048)])
@pytest.mark.parametrize("name", ["uniform", "deter_dupl"])
def test_sort_levels(ctx, oracle_mod, name, n, p):
    x = instances.generate(name, n, p=64, seed=7)
    rk, rp = oracle_mod.sort(x)
    ko, po, st = ctx.sort(_dev(x), p=p, seed=5, stats=True)
    np.testing.assert_array_equal(po.cpu().numpy().view(np.uint32), rp)
    np.testing.assert_array_equal(ko.cpu().numpy().view(np.uint64), rk)
    assert sum(st.class_elems) == n
    if name == "uniform":
        assert st.class_elems[4] == 0   # no oversize bucket
    ctx.check()


def test_many_segments_in_one_level(ctx, oracle_mod):
    # more level-1 segments than the plan has threads, of sizes around the caps
    rng = np.random.default_rng(5)
    sizes = np.concatenate([rng.integers(4097, 9000, 1500), rng.integers(1, 200, 500),
                            [20_000, 70_000, 4096, 4097, 1, 0, 64, 65]])
    rng.shuffle(sizes)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    x = rng.standard_normal(int(off[-1]))
    ko, po = ctx.segmented(torch.from_numpy(x).cuda(), torch.from_numpy(off.view(np.int64)).cuda())
    rk, rp = oracle_mod.segmented(x, off, oracle_mod.KEY_F64)
    np.testing.assert_array_equal(po.cpu().numpy().view(np.uint32), rp)
    np.testing.assert_array_equal(ko.cpu().numpy().view(np.uint64), rk)
    ctx.check()
