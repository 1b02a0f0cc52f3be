"""Partitions of fewer elements than buckets, against the oracle: several
splitters are then one sample, and copies of a key tie with all of them."""

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


@pytest.mark.parametrize("name", ["deter_dupl", "zero", "uniform"])
@pytest.mark.parametrize("k", [64, 1000])
def test_fewer_elements_than_buckets(ctx, oracle_mod, name, k):
    for n in (2, 7, 31, 63, 500):
        keys = instances.generate(name, n, p=1, seed=n)
        ref = oracle_mod.partition_ex(keys, k, seed=9, tie_break=True, over=1)
        t = torch.from_numpy(np.ascontiguousarray(keys).view(np.int64)).cuda()
        ko, po, off, fine, first = ctx.partition_ex(t, k, seed=9)
        torch.cuda.synchronize()
        assert np.array_equal(off.cpu().numpy().astype(np.uint64), ref["offsets"]), n
        assert np.array_equal(po.cpu().numpy().view(np.uint32), ref["pos_out"]), n
    ctx.check()
