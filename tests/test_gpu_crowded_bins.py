"""Buckets whose equal-width bins are crowded: the bins are refined once to the
keys' density (smooth but uneven distributions, float64 above all), and what
is crowded still is sorted by the bitonic network in registers.  Sizes sit at
the edges of the in-SM size classes and of the network's shared-memory form;
results are the oracle's bit for bit.
"""
import numpy as np
import pytest
import torch

import instances

pytestmark = pytest.mark.gpu

BINS, BITONIC = 1, 2
SIZES = [65, 127, 128, 129, 256, 257, 1000, 1024, 1025, 2047, 2048, 2049, 4095, 4096]


@pytest.fixture(scope="module")
def ctx():
    from paper_1606_08766_gb300 import Context
    c = Context(0)
    yield c
    c.close()


def _keys(kind, n):
    rng = np.random.default_rng(n)
    if kind == "normal":
        return rng.standard_normal(n)
    if kind == "octaves":       # every float64 exponent, both signs
        return np.ldexp(rng.uniform(1, 2, n), rng.integers(-1074, 1023, n)) * rng.choice([-1, 1], n)
    if kind == "outlier":       # a narrow cluster and one far key
        x = rng.integers(1 << 40, (1 << 40) + 50 * n, n, dtype=np.uint64)
        x[n // 2] = np.uint64(2**64 - 1)
        return x
    if kind == "three":         # three values with the extremes among them
        return np.array([0, 1 << 33, 2**64 - 1], dtype=np.uint64)[rng.integers(0, 3, n)]
    x = rng.standard_normal(n)  # a third of the keys are copies of one value
    x[rng.random(n) < 0.33] = 0.25
    return x


def _sort(ctx, oracle_mod, x):
    f64 = x.dtype == np.float64
    rk, rp = oracle_mod.sort(x, oracle_mod.KEY_F64) if f64 else oracle_mod.sort(x)
    t = torch.from_numpy(x if f64 else x.view(np.int64).copy()).cuda()
    ko, po, st = ctx.sort(t, p=1, stats=True)
    np.testing.assert_array_equal(po.cpu().numpy().view(np.uint32), rp)
    np.testing.assert_array_equal(ko.cpu().numpy().view(np.uint64), rk)
    assert sum(st.algo_elems) + st.class_elems[0] == x.shape[0]
    ctx.check()
    return st


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", ["normal", "octaves", "outlier", "three", "copies"])
def test_one_bucket(ctx, oracle_mod, kind, n):
    st = _sort(ctx, oracle_mod, _keys(kind, n))
    if kind == "normal":
        assert st.algo_elems[BINS] == n
    if kind == "three":
        assert st.algo_elems[BITONIC] == n


@pytest.mark.parametrize("kind", ["normal", "copies"])
def test_sample_and_buckets(ctx, oracle_mod, kind):
    # the sample of level 1 (8192-pair chunks) and every final bucket
    _sort(ctx, oracle_mod, _keys(kind, 1_300_001))


@pytest.mark.parametrize("cls", ["sort_small", "sort_mid", "sort_medium"])
def test_bitonic_everywhere(oracle_mod, cls):
    from paper_1606_08766_gb300 import Context
    with Context(0) as c:
        c.set_tunable(cls, 2)
        for n in (65, 128, 129, 1024, 1025, 2048, 2049, 4096):
            _sort(c, oracle_mod, instances.generate("uniform", n, seed=n))
