"""The tree median across the edges of its kernels: one subtree of 4096 leaves
and just beyond, trees whose windows take two further launches, and a tree
most of whose subtrees are empty.  The chosen element is the oracle's.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1606_08766_gb300 import Context
    c = Context(0)
    yield c
    c.close()


def _check(ctx, oracle_mod, x, k, seeds):
    t = torch.from_numpy(x.view(np.int64).copy()).cuda()
    for seed in seeds:
        assert int(ctx.approx_median(t, k, seed).item()) == oracle_mod.tree_median(x, k, seed)
    ctx.check()


@pytest.mark.parametrize("n", [31, 4095, 4096, 4097, 8192, 8193, 131_072, 131_073])
@pytest.mark.parametrize("k", [2, 8, 32])
def test_subtree_edges(ctx, oracle_mod, n, k):
    rng = np.random.default_rng(n + k)
    _check(ctx, oracle_mod, rng.integers(0, 1 << 20, n, dtype=np.uint64), k, (1, 2))


@pytest.mark.parametrize("n,k", [((1 << 20) + 1, 16), ((1 << 20) + 1, 32), (1 << 22, 32)])
def test_three_launches(ctx, oracle_mod, n, k):
    rng = np.random.default_rng(n)
    _check(ctx, oracle_mod, rng.integers(0, 2**64, n, dtype=np.uint64), k, (3,))
