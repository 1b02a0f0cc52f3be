"""Calls under an HBM budget that just holds their scratch.

The budgets are what the library needed for these calls before its levels kept
key ranges and chunk maps; a program that set one of them must still be served,
whichever plan it takes.  Results against numpy and the oracle."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# the scratch of a call depends on the SM count through its chunk sizes
SMS = 152
# entry point, n, its parameters, bytes
CALLS = [
    ("sort", 200, (1,), 4096),
    ("sort", 4078, (1,), 11776),
    ("sort", 5063, (2,), 75264),
    ("sort", 1 << 22, (64,), 61923072),
    ("segmented", 768, (111,), 28928),
    ("segmented", 50_984, (1,), 737280),
    ("segmented", 1 << 20, (100_000,), 27480832),
    ("partition", 4566, (1, 1), 12800),
    ("partition", 7_709_767, (1, 1), 15703552),
    ("partition", 7_593_721, (3, 1), 15488768),
    ("partition", 1 << 22, (150, 1), 11445248),
    ("partition", 7_895_227, (3, 10), 16104192),
]


@pytest.fixture(autouse=True)
def sms():
    if torch.cuda.get_device_properties(0).multi_processor_count != SMS:
        pytest.skip(f"the budgets are of a GPU with {SMS} SMs")


def _keys(n, seed):
    return np.random.default_rng(seed).integers(0, 2**64, n, dtype=np.uint64)


def _sort_ok(keys, ko, po):
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(po.cpu().numpy().view(np.uint32), order)
    assert np.array_equal(ko.cpu().numpy().view(np.uint64), keys[order])


@pytest.mark.parametrize("call,n,args,budget", CALLS)
def test_call_fits_its_former_scratch(oracle_mod, call, n, args, budget):
    from paper_1606_08766_gb300 import Context
    keys = _keys(n, n)
    t = torch.from_numpy(keys.view(np.int64)).cuda()
    with Context(0, hbm_budget_bytes=budget) as ctx:
        if call == "sort":
            ko, po = ctx.sort(t, p=args[0], seed=3)
            ctx.check()
            _sort_ok(keys, ko, po)
        elif call == "segmented":
            off = np.linspace(0, n, args[0] + 1).astype(np.int64)
            ko, po = ctx.segmented(t, torch.from_numpy(off).cuda(), seed=3)
            ctx.check()
            ref_k, ref_p = oracle_mod.segmented(keys, off.astype(np.uint64))
            assert np.array_equal(ko.cpu().numpy().view(np.uint64), ref_k)
            assert np.array_equal(po.cpu().numpy().view(np.uint32), ref_p)
        else:
            k, over = args
            ko, po, offs, fine, first = ctx.partition_ex(t, k, seed=3, overpartition=over)
            ctx.check()
            ref = oracle_mod.partition_ex(keys, k, seed=3, over=over)
            assert np.array_equal(offs.cpu().numpy().astype(np.uint64), ref["offsets"])
            assert np.array_equal(po.cpu().numpy().view(np.uint32), ref["pos_out"])


@pytest.mark.parametrize("n,budget", [(100_000, 3459328), (300_000, 10384384),
                                      (1 << 20, 36316928)])
def test_request_fits_its_former_footprint(n, budget):
    """A request of the server, with its batch buffers."""
    from paper_1606_08766_gb300 import Context
    keys = _keys(n, n)
    t = torch.from_numpy(keys.view(np.int64)).cuda()
    ko = torch.empty_like(t)
    po = torch.empty(n, dtype=torch.int32, device="cuda")
    with Context(0, hbm_budget_bytes=budget) as ctx:
        for _ in range(2):
            assert ctx.wait(ctx.submit(t, ko, po)) == 0
        _sort_ok(keys, ko, po)


@pytest.mark.parametrize("beside", [745_000, 919_040, 20_000_000])
def test_a_call_next_to_another_workspace(beside):
    """A sort of 50,000 keys beside what a request of 100,000 left held: its finer
    plan (818,688 bytes) gives way to the least one (744,960) where only that fits."""
    from paper_1606_08766_gb300 import Context
    x = torch.from_numpy(_keys(100_000, 1).view(np.int64)).cuda()
    xo, xp = torch.empty_like(x), torch.empty(x.numel(), dtype=torch.int32, device="cuda")
    keys = _keys(50_000, 2)
    t = torch.from_numpy(keys.view(np.int64)).cuda()
    torch.cuda.synchronize()
    with Context(0, hbm_budget_bytes=3459328 + beside) as ctx:
        assert ctx.wait(ctx.submit(x, xo, xp)) == 0
        for _ in range(2):
            ko, po = ctx.sort(t)
        ctx.check()
        _sort_ok(keys, ko, po)
