"""The tree median at the edges of its launches: the first launch's subtrees of 2048
leaves (one CTA that finishes, then two that hand their windows on), the groups of
windows of the next (4096 or 8192 entries of k), and a context's check after a
median as its only call.  The chosen element is the oracle's."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

LEAVES = 2048


def _group(k):
    return (8192 if k >= 16 else 4096) // k * LEAVES   # leaves of one group of windows


@pytest.fixture(scope="module")
def ctx():
    from paper_1606_08766_gb300 import Context
    c = Context(0)
    yield c
    c.close()


def _check(ctx, oracle_mod, x, k, seed):
    kt = 1 if x.dtype == np.float64 else 0
    t = torch.from_numpy(x.view(np.int64).copy()).cuda()
    got = int(ctx.approx_median(t, k, seed, key_type=kt).item())
    assert got == oracle_mod.tree_median(x, k, seed, key_type=kt)
    ctx.check()


@pytest.mark.parametrize("n", [1, LEAVES - 1, LEAVES, LEAVES + 1, 2 * LEAVES, 2 * LEAVES + 1])
@pytest.mark.parametrize("k", [2, 4, 8, 16, 32])
def test_first_launch(ctx, oracle_mod, n, k):
    rng = np.random.default_rng(n + k)
    _check(ctx, oracle_mod, rng.integers(0, 50, n, dtype=np.uint64), k, 1)
    _check(ctx, oracle_mod, rng.standard_normal(n), k, 2)


@pytest.mark.parametrize("k", [2, 4, 8, 16, 32])
def test_groups_of_windows(ctx, oracle_mod, k):
    for n in (_group(k) - 1, _group(k), _group(k) + 1):
        _check(ctx, oracle_mod, np.random.default_rng(n).integers(0, 2**64, n, dtype=np.uint64), k,
               3)


@pytest.mark.parametrize("n", [1, 5, 100])
def test_check_after_a_median_alone(oracle_mod, n):
    from paper_1606_08766_gb300 import Context
    with Context(0) as c:
        _check(c, oracle_mod, np.arange(n, dtype=np.uint64)[::-1].copy(), 2, 1)
