"""Performance cases of the robust sample sort: what a program asks of the
library through its public entry points, over the range of sizes, key types and
key distributions it meets.

Entry points: Context.sort, Context.segmented, Context.partition,
Context.partition_ex (the no-tie-breaking and overpartitioning options),
Context.approx_median and the request server (submit / wait).  uint64 keys are
held in int64 tensors (bit patterns), float64 keys in float64 tensors.
"""
import math

import torch

from paper_1606_08766_gb300 import Context

DEVICE = "cuda:0"
TOP = -(1 << 63)      # the sign bit, as int64


def listed():
    return [
        # one small request sorted by itself: nothing but latency
        {"name": "sort_u64_200", "kind": "sort", "n": 200, "keys": "uniform", "p": 1},
        # the largest kind of input that one SM sorts, ragged, float64
        {"name": "sort_f64_3001", "kind": "sort", "n": 3001, "keys": "f64_dup", "p": 1},
        # an ordinary array of records, the fan-out left to the library
        {"name": "sort_gauss_100k", "kind": "sort", "n": 100_003, "keys": "gaussian", "p": 1},
        # the plain workload of 2^20 uniform keys over 64 virtual partitions
        {"name": "sort_u64_1m_p64", "kind": "sort", "n": 1 << 20, "keys": "uniform", "p": 64},
        # a column of 20 million measurements, a tenth of them repeated values
        {"name": "sort_f64_20m", "kind": "sort", "n": 20_000_003, "keys": "f64_dup", "p": 1},
        # the headline workload: 2^28 uniform keys over 1024 virtual partitions
        {"name": "sort_u64_268m_p1024", "kind": "sort", "n": 1 << 28, "keys": "uniform",
         "p": 1024},
        # duplicate-heavy keys (16 values in runs), the robustness workload
        {"name": "sort_runs_67m_p1024", "kind": "sort", "n": (1 << 26) + 5, "keys": "runs",
         "p": 1024},
        # the partition step alone: 1024 stable buckets for a program's own use
        {"name": "partition_u64_67m_k1024", "kind": "partition", "n": 1 << 26, "keys": "uniform",
         "k": 1024},
        # the overpartitioned step (b = 10: within 20 % of perfect balance)
        {"name": "partition_ams_17m_k256", "kind": "partition_ex", "n": (1 << 24) + 77,
         "keys": "gaussian", "k": 256, "over": 10, "ties": True},
        # the batched workload: 100,000 float64 segments of 1 to 2^15 keys
        {"name": "segmented_100k_2p15", "kind": "segmented", "segments": 100_000, "log2": 15},
        # pivot selection of a quicksort over a million keys
        {"name": "median_1m_k16", "kind": "median", "n": 1 << 20, "keys": "uniform", "k": 16},
        # a server's burst: requests of 2^4 to 2^22 keys of both types at once
        {"name": "serve_48_2p22", "kind": "serve", "requests": 48, "log2": 22},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sort", "sort", "sort", "partition", "partition_ex", "segmented", "median",
                       "serve"])
    c = {"kind": kind}
    if kind == "sort":
        c["n"] = _log_uniform(rng, 16, 1 << 27)
        c["keys"] = rng.choice(["uniform", "gaussian", "f64_dup", "runs"])
        # automatic, or partitions of about 256 keys, up to 1024 of them
        c["p"] = rng.choice([1, max(1, min(1024, -(-c["n"] // 256)))])
    elif kind in ("partition", "partition_ex"):
        c["n"] = _log_uniform(rng, 1 << 12, 1 << 27)
        c["keys"] = rng.choice(["uniform", "gaussian", "runs"])
        if kind == "partition":
            c["k"] = _log_uniform(rng, 2, 2048)
        else:
            c["k"] = _log_uniform(rng, 2, 1024)
            c["over"] = rng.choice([1, 4, 10])
            c["ties"] = rng.choice([True, False])
    elif kind == "segmented":
        c["log2"] = rng.randint(8, 20)
        most = min(100_000, int(1.5e8 / _mean_size(c["log2"])))
        c["segments"] = _log_uniform(rng, 50, max(51, most))
    elif kind == "median":
        c["n"] = _log_uniform(rng, 1 << 6, 1 << 20)
        c["keys"] = rng.choice(["uniform", "gaussian", "f64_dup"])
        c["k"] = rng.choice([4, 8, 16, 32])
    else:
        c["requests"] = rng.randint(12, 64)
        c["log2"] = rng.randint(14, 23)
    return c


def _mean_size(log2):
    return (2.0 ** log2 - 1) / (log2 * math.log(2.0))


def _sizes(count, log2, lo=0.0):
    """`count` sizes evenly spread over the logarithm of [2^lo, 2^log2]."""
    return [max(1, int(2.0 ** (lo + (log2 - lo) * (i + 0.5) / count))) for i in range(count)]


def _keys(kind, n, gen):
    """n keys: an int64 tensor of uint64 patterns, or a float64 tensor."""
    if kind == "uniform":
        return torch.randint(TOP, (1 << 63) - 1, (n,), dtype=torch.int64, device=DEVICE,
                             generator=gen)
    if kind == "gaussian":
        # mean 2^63, deviation 2^60 (uint64), as int64 patterns
        z = torch.randn(n, dtype=torch.float64, device=DEVICE, generator=gen)
        return (z.clamp_(-7.9, 7.9) * 2.0 ** 60).to(torch.int64) ^ TOP
    if kind == "runs":
        # runs of 1 to 4096 copies of one of 16 values
        r = max(1, n // 1024) + 16
        lengths = torch.randint(1, 4097, (r,), dtype=torch.int64, device=DEVICE, generator=gen)
        values = torch.randint(0, 16, (r,), dtype=torch.int64, device=DEVICE, generator=gen)
        x = torch.repeat_interleave(values, lengths)[:n]
        return torch.cat([x, values[:1].expand(n - x.numel())]).contiguous()
    if kind == "f64_dup":
        # normal values, about a tenth of them copies of another one
        x = torch.randn(n, dtype=torch.float64, device=DEVICE, generator=gen)
        m = n // 10
        to = torch.randint(0, n, (m,), dtype=torch.int64, device=DEVICE, generator=gen)
        x[to.unique()] = x[torch.randint(0, n, (to.unique().numel(),), dtype=torch.int64,
                                         device=DEVICE, generator=gen)]
        return x
    raise ValueError(kind)


def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _segmented_input(case, gen):
    sizes = torch.tensor(_sizes(case["segments"], case["log2"]), dtype=torch.int64, device=DEVICE)
    sizes = sizes[torch.randperm(sizes.numel(), device=DEVICE, generator=gen)]
    offsets = torch.zeros(sizes.numel() + 1, dtype=torch.int64, device=DEVICE)
    offsets[1:] = torch.cumsum(sizes, 0)
    n = int(offsets[-1])
    x = torch.randn(n, dtype=torch.float64, device=DEVICE, generator=gen)
    # a tenth of the positions take the value of another one of their segment
    at = torch.randint(0, n, (n // 10,), dtype=torch.int64, device=DEVICE, generator=gen).unique()
    seg = torch.searchsorted(offsets, at, right=True) - 1
    u = torch.rand(at.numel(), dtype=torch.float64, device=DEVICE, generator=gen)
    x[at] = x[offsets[seg] + (u * sizes[seg]).to(torch.int64)]
    return x, offsets


def _serve_input(case, gen):
    """One buffer of 8-byte keys cut into requests: (bits, [(offset, size, is_f64)])."""
    sizes = _sizes(case["requests"], case["log2"], lo=4.0)
    order = torch.randperm(len(sizes), device=DEVICE, generator=gen).tolist()
    parts, spans, at = [], [], 0
    for i, j in enumerate(order):
        kind = ("uniform", "f64_dup", "runs", "f64_dup", "gaussian", "f64_dup")[i % 6]
        x = _keys(kind, sizes[j], gen)
        parts.append(x.view(torch.int64))
        spans.append((at, sizes[j], kind == "f64_dup"))
        at += sizes[j]
    return torch.cat(parts), spans


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    s = {"case": case, "ctx": Context(0)}
    if kind == "segmented":
        s["keys"], s["offsets"] = _segmented_input(case, gen)
    elif kind == "serve":
        bits, spans = _serve_input(case, gen)
        s["out"] = torch.empty_like(bits)
        s["perm"] = torch.empty(bits.numel(), dtype=torch.int32, device=DEVICE)
        s["requests"] = []
        for at, m, f64 in spans:
            k, o = bits[at:at + m], s["out"][at:at + m]
            if f64:
                k, o = k.view(torch.float64), o.view(torch.float64)
            s["requests"].append((k, o, s["perm"][at:at + m]))
        torch.cuda.synchronize()   # the server reads the keys on streams of its own
        return s
    else:
        s["keys"] = _keys(case["keys"], case["n"], gen)
    if kind in ("sort", "segmented"):
        s["keys_out"] = torch.empty_like(s["keys"])
        s["perm_out"] = torch.empty(s["keys"].numel(), dtype=torch.int32, device=DEVICE)
    return s


def run(state):
    c, ctx = state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "sort":
        return ctx.sort(state["keys"], p=c["p"], seed=1, keys_out=state["keys_out"],
                        perm_out=state["perm_out"])
    if kind == "segmented":
        return ctx.segmented(state["keys"], state["offsets"], seed=1, keys_out=state["keys_out"],
                             perm_out=state["perm_out"])
    if kind == "partition":
        return ctx.partition(state["keys"], c["k"], seed=1)
    if kind == "partition_ex":
        return ctx.partition_ex(state["keys"], c["k"], seed=1, tie_break=c["ties"],
                                overpartition=c["over"])
    if kind == "median":
        return ctx.approx_median(state["keys"], k=c["k"], seed=1)
    tickets = [ctx.submit(k, o, p) for k, o, p in state["requests"]]
    for t in tickets:
        if ctx.wait(t) != 0:
            raise RuntimeError("a request failed")
    return state["out"], state["perm"]


def work(case):
    kind = case["kind"]
    if kind == "sort":          # read the keys; write keys and permutation
        return {"bytes": 20 * case["n"], "flops": 0}
    if kind == "segmented":
        n = sum(_sizes(case["segments"], case["log2"]))
        return {"bytes": 20 * n + 8 * (case["segments"] + 1), "flops": 0}
    if kind == "serve":
        return {"bytes": 20 * sum(_sizes(case["requests"], case["log2"], lo=4.0)), "flops": 0}
    if kind == "partition":
        return {"bytes": 20 * case["n"] + 8 * (case["k"] + 1), "flops": 0}
    if kind == "partition_ex":
        k, b = case["k"], case["over"]
        return {"bytes": 20 * case["n"] + 12 * (k + 1) + 8 * k * b, "flops": 0}
    return {"bytes": 8 * case["n"] + 8, "flops": 0}


def _ordered(bits, f64):
    """int64 values whose signed order is the order of the keys."""
    if f64:
        return torch.where(bits < 0, bits ^ ((1 << 63) - 1), bits)
    return bits ^ TOP


def _sorted(keys):
    bits = keys.view(torch.int64)
    perm = torch.sort(_ordered(bits, keys.dtype == torch.float64), stable=True).indices
    return keys[perm], perm.to(torch.int32)


def exact(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "sort":
        return _sorted(_keys(case["keys"], case["n"], gen))
    if kind == "segmented":
        x, offsets = _segmented_input(case, gen)
        o = torch.sort(_ordered(x.view(torch.int64), True), stable=True).indices
        seg = torch.searchsorted(offsets, o, right=True) - 1
        o = o[torch.sort(seg, stable=True).indices]
        first = torch.repeat_interleave(offsets[:-1], offsets[1:] - offsets[:-1])
        return x[o], (o - first).to(torch.int32)
    if kind == "serve":
        bits, spans = _serve_input(case, gen)
        out, perm = torch.empty_like(bits), torch.empty(bits.numel(), dtype=torch.int32,
                                                        device=DEVICE)
        for at, m, f64 in spans:
            k = bits[at:at + m]
            o = torch.sort(_ordered(k, f64), stable=True).indices
            out[at:at + m], perm[at:at + m] = k[o], o.to(torch.int32)
        return out, perm
    return None
