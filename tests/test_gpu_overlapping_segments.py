"""Decreasing offsets, whose segments may overlap: reported as a device error, with
the segments above 4096 keys left alone, and the context goes on working."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

BIG = 4096


@pytest.fixture(scope="module")
def ctx():
    from paper_1606_08766_gb300 import Context
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("f64", [False, True])
@pytest.mark.parametrize("offsets", [
    [0, 400_000, 100_000, 300_000],                  # one large inside another
    [0, 400_000, 0, 400_000, 0, 200_000],            # the same one again
    [0, 3000, 2000, 2500, 100_000, 90_000, 390_000],  # small and large ones
    [390_000, 400_000, 0, 5000, 4000, 9000],
])
def test_decreasing_offsets(ctx, oracle_mod, offsets, f64):
    from paper_1606_08766_gb300 import RsortError
    rng = np.random.default_rng(len(offsets))
    n = 400_000
    keys = rng.standard_normal(n) if f64 else rng.integers(0, 2**64, n, dtype=np.uint64)
    bits = keys.view(np.int64)
    t = torch.from_numpy(bits.copy()).cuda()
    ko = torch.full_like(t, -7)
    po = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    off = torch.tensor(offsets, dtype=torch.int64, device="cuda")
    kt = 1 if f64 else 0
    ctx.segmented(t, off, keys_out=ko, perm_out=po, key_type=kt)
    with pytest.raises(RsortError) as e:
        ctx.check()
    assert e.value.status == -7
    # what no segment of at most 4096 keys covers is as it was
    got = ko.cpu().numpy()
    covered = np.zeros(n, bool)
    for a, b in zip(offsets[:-1], offsets[1:]):
        if a < b <= a + BIG:
            covered[a:b] = True
    assert (got[~covered] == -7).all()
    # a lone small segment is sorted all the same
    small = [(a, b) for a, b in zip(offsets[:-1], offsets[1:]) if a < b <= a + BIG]
    for a, b in small:
        if all(y <= a or x >= b for x, y in small if (x, y) != (a, b)):
            rk, _ = oracle_mod.sort(keys[a:b], kt)
            assert np.array_equal(got[a:b].view(np.uint64), rk)
    # and the context sorts on
    good = np.array([0, 5, 100_000, 300_000, n], np.int64)
    k2, p2 = ctx.segmented(t, torch.from_numpy(good).cuda(), key_type=kt)
    ctx.check()
    rk, rp = oracle_mod.segmented(keys, good.astype(np.uint64), key_type=kt)
    assert np.array_equal(k2.cpu().numpy().view(np.uint64), rk)
    assert np.array_equal(p2.cpu().numpy().view(np.uint32), rp)
