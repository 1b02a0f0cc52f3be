"""A call whose input is the output of the call before it, with no wait between.

A call's launches are set up while the launch before them still runs, so the
kernels that can be the first of a call must not read the caller's arrays
through the read-only path (its data may not change while a kernel is resident).
That is shown on the source; the chains are then run against the oracle."""

import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1606_08766_gb300", "csrc")
READ_ONLY = re.compile(r"__ldg\b|\.nc\b|\bld_stream_|\bprefetch_l2_range\b")


def _body(file, name):
    """The definition of function `name` in a source file, comments removed."""
    text = open(os.path.join(CSRC, file)).read()
    text = re.sub(r"//[^\n]*", "", text)
    m = re.search(r"\b%s\s*\([^;{]*\)\s*(?:const\s*)?\{" % re.escape(name), text)
    assert m, f"{name} not found in {file}"
    depth, i = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[m.start():i]


@pytest.mark.parametrize("file,name", [
    ("splitters.cuh", "load_key"),              # the sample's keys
    ("partition_kernels.cu", "k_sample_sort"),  # first of a sort or partition
    ("partition_kernels.cu", "k_init_plain"),   # first of a batch
    ("partition_kernels.cu", "k_init_segments"),
    ("local_sort_kernels.cu", "load_elem"),     # k_direct_sort's keys
    ("local_sort_kernels.cu", "k_direct_sort"),
    ("median_kernels.cu", "k_tm_leaves"),
])
def test_first_launches_read_by_ordinary_loads(file, name):
    assert not READ_ONLY.search(_body(file, name))


@pytest.fixture(scope="module")
def ctx():
    from paper_1606_08766_gb300 import Context
    c = Context(0)
    yield c
    c.close()


# sizes: one launch, one level, two levels
@pytest.mark.gpu
@pytest.mark.parametrize("n", [1000, 70_001, 1_300_001])
@pytest.mark.parametrize("f64", [False, True])
def test_partition_of_a_sort_of_a_partition(ctx, oracle_mod, n, f64):
    import torch
    rng = np.random.default_rng(n)
    keys = rng.standard_normal(n) if f64 else rng.integers(0, 2**64, n, dtype=np.uint64)
    kt = 1 if f64 else 0
    bits = keys.view(np.uint64)
    t = torch.from_numpy(bits.view(np.int64).copy()).cuda()
    torch.cuda.synchronize()
    for seed in range(4):   # (other samples, so other orders, from round to round)
        ko, po, off = ctx.partition(t, 64, seed=seed, key_type=kt)
        so, sp = ctx.sort(ko, seed=5, key_type=kt)
        qo, qp, qoff = ctx.partition(so, 97, seed=7, key_type=kt)
        torch.cuda.synchronize()
        r1 = oracle_mod.partition(keys, 64, seed, key_type=kt)
        got = ko.cpu().numpy().view(np.uint64)
        assert np.array_equal(off.cpu().numpy().astype(np.uint64), r1["offsets"])
        assert np.array_equal(got, bits[r1["pos_out"]])
        order = np.argsort(got.view(keys.dtype), kind="stable")
        assert np.array_equal(sp.cpu().numpy().view(np.uint32), order)
        srt = so.cpu().numpy().view(np.uint64)
        assert np.array_equal(srt, got[order])
        r2 = oracle_mod.partition(srt.view(keys.dtype), 97, 7, key_type=kt)
        assert np.array_equal(qoff.cpu().numpy().astype(np.uint64), r2["offsets"])
        assert np.array_equal(qp.cpu().numpy().view(np.uint32), r2["pos_out"])
    ctx.check()
