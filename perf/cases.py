"""The sorts whose speed this repository is measured by, each through the public entry points of
``paper_2505_18681_gb300``: lone arrays from a thousand keys to a billion, stable key/value sorts,
the mergesort, and batched segmented sorts, over the key types and the distributions that the
inputs module draws.

A case is a dict of plain values:

* ``op``          ``sort`` (keys into a second buffer), ``pairs`` (keys and uint32 values into second
                  buffers, the values an index: a stable argsort) or ``segments`` (a batch of arrays, in place)
* ``dtype``       key type
* ``n``           keys (``sort``, ``pairs``); a batch has ``segments`` arrays of log-uniform length
                  ``shortest``..``longest`` instead
* ``dist``        distribution of the keys (a name of the inputs module)
* ``algo``        ``auto`` (the library chooses), ``radix`` or ``merge``
* ``descending``  direction of the order
* ``table``       whether the program has loaded the tuned tables (the dispatcher then samples the keys)
"""
from __future__ import annotations

import glob
import os

import torch

import paper_2505_18681_gb300 as evo
from paper_2505_18681_gb300 import inputs

_TABLES = sorted(glob.glob(os.path.join(os.path.dirname(os.path.abspath(evo.__file__)), "tuned", "*.txt")))
_BYTES = {"int32": 4, "uint32": 4, "float32": 4, "int64": 8, "uint64": 8, "float64": 8}

_INT_DISTS = ("uniform", "uniform", "uniform", "uniform_paper", "gaussian", "zipf", "nearly_sorted", "sorted",
              "reverse", "distinct16", "uniform1000", "equal", "paper_normal", "paper_exponential",
              "paper_clustered", "paper_duplicates")


def _array(op, dtype, n, dist="uniform", algo="auto", descending=False, table=False, **more):
    return {"op": op, "dtype": dtype, "n": n, "dist": dist, "algo": algo, "descending": descending,
            "table": table, **more}


def _batch(dtype, segments, longest, shortest=16, table=False, **more):
    return {"op": "segments", "dtype": dtype, "segments": segments, "shortest": shortest, "longest": longest,
            "table": table, **more}


def listed():
    return [
        # a thousand keys: one bucket, one page of results, one request of a service; latency is all of it
        _array("sort", "int32", 1000, name="sort_1k_i32"),
        # scores of a few thousand candidates ranked best first, with the index of each
        _array("pairs", "float32", 3999, "float_mix", descending=True, name="argsort_4k_f32_desc"),
        # ten thousand keys, above what one thread block takes: several launches on a chip that is nearly idle
        _array("sort", "int32", 10_000, name="sort_10k_i32"),
        # a million keys by the plain radix sort, asked for by name: the benchmark's smallest configuration
        _array("sort", "int32", 1_000_000, algo="radix", name="sort_1m_i32_radix"),
        # measurements around zero, an odd number of them, with the tables loaded: few of the 64 bits vary
        _array("sort", "int64", 20_000_003, "gaussian", table=True, name="sort_20m_i64_gauss"),
        # the mergesort at the benchmark's size
        _array("sort", "int32", 100_000_000, algo="merge", name="merge_100m_i32"),
        # a billion random keys with the tables loaded: the benchmark's arrays, in both widths
        _array("sort", "int64", 1_000_000_000, table=True, name="sort_1b_i64"),
        _array("sort", "int32", 1_000_000_000, table=True, name="sort_1b_i32"),
        # heavy-tailed identifiers, as the benchmark's skewed array, with no table
        _array("sort", "int64", 500_000_000, "zipf", name="sort_500m_i64_zipf"),
        # the stable argsort of doubles with signed zeros and NaNs among them: the key/value configuration
        _array("pairs", "float64", 500_000_000, "float_mix", name="argsort_500m_f64"),
        # many arrays of very uneven length in one call: the segmented configuration
        _batch("int32", 10_000, 1_000_000, table=True, name="segments_10k_i32"),
        # short requests that a service packs into one call
        _batch("int64", 20_000, 8_000, name="segments_20k_short_i64"),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random())) | (1 if rng.random() < 0.5 else 0)


def draw(rng):
    """One more case: the operations and options of the listed ones over the whole range of sizes."""
    op = rng.choice(("sort", "sort", "sort", "pairs", "pairs", "merge", "segments", "segments"))
    if op == "segments":
        dtype = rng.choice(("int32", "int32", "int64", "float64", "uint32"))
        longest = _log(rng, 200, 1_000_000)
        # a log-uniform length averages about longest / ln(longest / 16) keys
        mean = max(16, longest // 8)
        return _batch(dtype, min(_log(rng, 50, 50_000), max(50, 600_000_000 // mean)), longest,
                      table=rng.random() < 0.5)
    dtype = rng.choice(("int32", "int32", "int64", "int64", "uint32", "uint64", "float32", "float64"))
    dist = rng.choice(("float_mix", "uniform")) if dtype.startswith("float") else rng.choice(_INT_DISTS)
    if dtype.startswith("uint") and dist.startswith(("gaussian", "uniform_paper", "paper_")):
        dist = "uniform"   # these draw signed values
    if op == "merge":
        return _array("sort", dtype, min(_log(rng, 300, 100_000_000), 50_000_000 if _BYTES[dtype] == 8 else 10 ** 9),
                      dist, algo="merge", descending=rng.random() < 0.2)
    n = _log(rng, 300, 300_000_000 if op == "pairs" else 800_000_000)
    return _array(op, dtype, n, dist, algo=rng.choice(("auto", "auto", "radix")), descending=rng.random() < 0.2,
                  table=rng.random() < 0.5)


def _lengths(case):
    """Lengths of a batch's arrays: the same for every seed, so that its outputs have one shape."""
    return inputs.segment_lengths(case["segments"], case["shortest"], case["longest"], seed=42)


def _zipf(n, dtype, seed):
    """Ranks 1..1e6 with P(k) proportional to k^-1.2, as the inputs module draws them; the cumulative
    shares are summed on the CPU, so that the same seed gives the same keys on every run."""
    share = torch.arange(1, 1_000_001, dtype=torch.float64) ** -1.2
    share = (torch.cumsum(share, 0) / share.sum()).cuda()
    state = inputs.stream_state(seed, 77)
    out = torch.empty(n, dtype=dtype, device="cuda")
    for start in range(0, n, 1 << 26):
        count = min(1 << 26, n - start)
        u = inputs.unit_double(inputs.raw64(state, start, count, "cuda"))
        _signed(out)[start:start + count] = \
            torch.searchsorted(share, u, right=True).clamp_(max=999_999).add_(1).to(_signed(out).dtype)
    return out


def _keys(case, seed):
    """The keys of a lone array, on the GPU."""
    dtype = getattr(torch, case["dtype"])
    if case["dist"] == "zipf":
        return _zipf(case["n"], dtype, seed)
    if case["dist"] in ("sorted", "reverse", "nearly_sorted"):
        # the ramps are the same for every seed: each key moves by less than a step, which keeps their order
        keys, n = inputs.generate(case["dist"], case["n"], dtype, seed=seed, device="cuda"), case["n"]
        step, state = (1 << 8 * _BYTES[case["dtype"]]) // n, inputs.stream_state(seed, 78)
        for start in range(0, n, 1 << 26):
            part = _signed(keys)[start:start + (1 << 26)]
            move = (inputs.raw64(state, start, part.numel(), "cuda") >> 1) & ((1 << 62) - 1)
            part.add_(move.remainder_(min(step, 1 << 62)).to(part.dtype))
        return keys
    if dtype == torch.float32 and case["dist"] != "float_mix":
        return inputs.generate(case["dist"], case["n"], torch.float64, seed=seed, device="cuda").to(dtype)
    return inputs.generate(case["dist"], case["n"], dtype, seed=seed, device="cuda")


def _signed(t):
    """The same memory as a type that every operation of torch takes."""
    return t.view({torch.uint32: torch.int32, torch.uint64: torch.int64}.get(t.dtype, t.dtype))


def prepare(case, seed):
    evo.table_clear()
    if case["table"]:
        for path in _TABLES:
            evo.table_load(path)
    if case["op"] == "segments":
        lengths = _lengths(case)
        name = {"float64": "int64", "float32": "int32"}.get(case["dtype"], case["dtype"])
        keys, offsets = inputs.segmented_keys(lengths, getattr(torch, name), seed=seed, device="cuda")
        if name != case["dtype"]:
            # the same ordering of values, as numbers of moderate size
            keys = keys.to(torch.float64).mul_(2.0 ** -40).to(getattr(torch, case["dtype"]))
        work = torch.empty_like(keys)
        return {"op": "segments", "keys": keys, "work": work, "shown": _signed(work), "offsets": offsets.cuda()}
    keys = _keys(case, seed)
    out = torch.empty_like(keys)
    options = {}
    if case["algo"] != "auto":
        options["algo"] = case["algo"]
    if case["algo"] == "merge":
        options["insertion_threshold"] = 32
    if case["descending"]:
        options["descending"] = True
    state = {"op": case["op"], "keys": keys, "out": out, "shown": _signed(out), "options": options}
    if case["op"] == "pairs":
        state["values"] = torch.arange(case["n"], dtype=torch.int32, device="cuda").view(torch.uint32)
        state["values_out"] = torch.empty_like(state["values"])
        state["values_shown"] = _signed(state["values_out"])
    return state


def run(state):
    if state["op"] == "sort":
        evo.sort(state["keys"], out=state["out"], **state["options"])
        return state["shown"]
    if state["op"] == "pairs":
        evo.sort_pairs(state["keys"], state["values"], state["out"], state["values_out"], **state["options"])
        return [state["shown"], state["values_shown"]]
    # the batch is sorted in place: the program keeps its input and sorts a copy
    state["work"].copy_(state["keys"])
    evo.segmented_sort(state["work"], state["offsets"])
    return state["shown"]


def work(case):
    if case["op"] == "segments":
        n = int(_lengths(case).sum())
    else:
        n = case["n"]
    # every key (and value) read once and written once; a sort computes nothing
    return {"bytes": 2.0 * n * (_BYTES[case["dtype"]] + (4 if case["op"] == "pairs" else 0)), "flops": 0.0}


def exact(case, seed):
    """The sorted keys of the floating types; whole numbers are moved, not computed."""
    if case["op"] == "segments" or not case["dtype"].startswith("float"):
        return None
    keys = _keys(case, seed).to(torch.float64)
    keys[torch.isnan(keys)] = float("nan")   # one sign: torch orders NaNs of both signs apart on the GPU
    keys = torch.sort(keys, descending=case["descending"])[0]
    return [keys, None] if case["op"] == "pairs" else keys
