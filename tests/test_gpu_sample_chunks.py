"""Partitions whose samples lie on either side of the lines between one sample
chunk and several (5120 samples), chunks of 1024 and 2048 (8192) and of 2048 and
4096 (196,608), against the oracle: the sorted sample must not depend on them."""

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


# 16 k ceil(log2 k) samples: 5088, 5184, 6144, 8176, 8288, 196592, 196768
@pytest.mark.parametrize("k", [53, 54, 64, 73, 74, 1117, 1118])
@pytest.mark.parametrize("name", ["uniform", "deter_dupl"])
def test_sample_chunks_match_oracle(ctx, oracle_mod, name, k):
    n = 262_147
    keys = instances.generate(name, n, p=1, seed=k)
    ref = oracle_mod.partition_ex(keys, k, seed=2, tie_break=True, over=1)
    t = torch.from_numpy(np.ascontiguousarray(keys).view(np.int64)).cuda()
    ko, po, off, _, _ = ctx.partition_ex(t, k, seed=2)
    torch.cuda.synchronize()
    assert np.array_equal(off.cpu().numpy().astype(np.uint64), ref["offsets"])
    assert np.array_equal(po.cpu().numpy().view(np.uint32), ref["pos_out"])
    assert np.array_equal(ko.cpu().numpy().view(np.uint64), ref["keys_out"])
    ctx.check()
