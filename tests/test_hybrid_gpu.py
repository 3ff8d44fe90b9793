"""GPU parity of the partition sort (large lone arrays, keys only, the choice
left to the library) against the oracle: every key type, inputs that its
sample does not show (keys outside the sampled range, crowded stretches,
frequent values), both ways of asking for its verdict, and captured graphs."""
import glob
import os

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

N = (1 << 23) + 4099          # above the size where calls without a table try it
TABLES = glob.glob(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_18681_gb300",
                                "tuned", "*.txt"))


@pytest.fixture()
def evo():
    import paper_2505_18681_gb300 as evo
    evo.library()
    evo.table_clear()
    yield evo
    evo.table_clear()


def host(t):
    if t.dtype in (torch.uint32, torch.uint64):
        s = t.view(torch.int32 if t.dtype == torch.uint32 else torch.int64).cpu().numpy()
        return s.view(np.uint32 if t.dtype == torch.uint32 else np.uint64)
    return t.cpu().numpy()


def bits(t):
    a = host(t) if isinstance(t, torch.Tensor) else t
    return a.view(np.uint32 if a.dtype.itemsize == 4 else np.uint64)


def taken(evo, fn):
    """Whether the partition sort sorted the array, and whether radix passes ran."""
    evo.sync()
    evo.profile(True)
    fn()
    evo.sync()
    recs = evo.profile_read()
    evo.profile(False)
    return (any(r["kind"] == "hybrid" and r["active"] for r in recs),
            any(r["kind"] == "radix_onesweep" and r["active"] for r in recs))


def gen(name, n, dtype, seed=3):
    from paper_2505_18681_gb300 import inputs
    if name in ("uniform", "gaussian", "zipf", "float_mix", "paper_exponential", "paper_duplicates"):
        return inputs.generate(name, n, dtype, seed=seed, device="cuda")
    x = inputs.generate("uniform", n, torch.int64, seed=seed, device="cuda")
    if name == "outliers":      # a narrow range, with a few keys far outside it that no sample is likely to hold
        x = (x >> 34) + 5
        x[12345] = -(1 << 62)
        x[n // 2 + 1] = (1 << 62) + 7
    elif name == "crowded":     # one key in fifty in a stretch of 2^20 values of the whole range
        x = torch.where(x % 50 == 0, (x >> 44) + (1 << 40), x)
    elif name == "pressed":     # the same with one key in 120: the sample accepts it, a bucket is too long
        x = torch.where(x % 120 == 0, (x >> 44) + (1 << 40), x)
    elif name == "frequent":    # one value held by 15 % of the keys, the others spread over 2^20 values
        x = torch.where((x >> 8) % 100 < 15, torch.full_like(x, 77), (x >> 44) & 0xFFFFF)
    elif name == "powers":      # magnitudes spread over every binary order
        m = (inputs.generate("uniform", n, torch.int64, seed=seed + 1, device="cuda") & 63).clamp(max=62)
        x = (x & ((1 << 62) - 1)) >> m
    if dtype == torch.int64:
        return x
    if dtype == torch.float64:
        return x.to(torch.float64)
    return (x >> 32).to(dtype) if name in ("crowded", "powers") else x.to(dtype)


CASES = [("uniform", torch.int32, True), ("uniform", torch.int64, True), ("uniform", torch.uint32, True),
         ("uniform", torch.uint64, True), ("uniform", torch.float32, None), ("uniform", torch.float64, None),
         ("float_mix", torch.float64, None), ("zipf", torch.int64, None), ("gaussian", torch.int64, None),
         ("paper_exponential", torch.int32, None), ("paper_duplicates", torch.int32, True),
         ("outliers", torch.int64, None), ("crowded", torch.int64, None), ("frequent", torch.int64, None),
         ("powers", torch.int64, None), ("powers", torch.float64, None)]


@pytest.mark.parametrize("table", [False, True], ids=["async", "table"])
@pytest.mark.parametrize("name,dtype,expect", CASES, ids=lambda v: str(v))
def test_parity(evo, name, dtype, expect, table):
    """The oracle's order whichever path is taken; spread keys take this one."""
    x = gen(name, N, dtype)
    want = bits(oracle.radix_sort(host(x)))
    if table:
        for t in TABLES:
            evo.table_load(t)
    y = torch.empty_like(x)
    used, passes = taken(evo, lambda: evo.sort(x, out=y))
    assert np.array_equal(bits(y), want)
    assert used != passes
    if expect is not None:
        assert used == expect
    evo.sort(x, out=y, descending=True)
    z = x.clone()
    evo.sort(z)
    evo.sync()
    assert np.array_equal(bits(y), want[::-1]) and np.array_equal(bits(z), want)


@pytest.mark.parametrize("n,table", [((1 << 21) - 1, True), (1 << 21, True), ((1 << 23) - 1, False), (1 << 23, False)])
def test_size_threshold(evo, n, table):
    x = gen("uniform", n, torch.int64)
    if table:
        for t in TABLES:
            evo.table_load(t)
    y = torch.empty_like(x)
    used, _ = taken(evo, lambda: evo.sort(x, out=y))
    assert used == (n in (1 << 21, 1 << 23))
    assert np.array_equal(bits(y), bits(oracle.radix_sort(host(x))))


def test_explicit_parameters_and_pairs_keep_the_radix_passes(evo):
    x = gen("uniform", N, torch.int32)
    want = bits(oracle.radix_sort(host(x)))
    for kw in ({"algo": "radix"}, {"rank_mode": 3}, {"block_size": 1024, "keys_per_thread": 16}):
        y = torch.empty_like(x)
        assert taken(evo, lambda: evo.sort(x, out=y, **kw)) == (False, True), kw
        assert np.array_equal(bits(y), want)
    v = torch.arange(N, dtype=torch.int32, device="cuda").view(torch.uint32)
    k, w = torch.empty_like(x), torch.empty_like(v)
    assert taken(evo, lambda: evo.sort_pairs(x, v, k, w)) == (False, True)
    assert np.array_equal(bits(k), want)


def test_unaligned_view_and_caller_workspace(evo):
    x = gen("uniform", N + 3, torch.int32)[3:]
    want = bits(oracle.radix_sort(host(x)))
    y = torch.empty(N + 1, dtype=torch.int32, device="cuda")[1:]
    need = evo.workspace_bytes(N, torch.int32, algo=None)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    used, _ = taken(evo, lambda: evo.sort(x, out=y, workspace=ws))
    assert used and np.array_equal(bits(y), want)


def test_captured_graph_decides_anew_for_new_keys(evo):
    """One captured call, replayed on keys that take the path, keys that are
    refused by the sample and keys that are refused after the counts."""
    x = gen("uniform", N, torch.int64)
    y = torch.empty_like(x)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        evo.sort(x, out=y, stream=s)
        evo.sync(s)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            evo.sort(x, out=y, stream=s)
    for name in ("crowded", "uniform", "gaussian", "outliers", "frequent"):
        x.copy_(gen(name, N, torch.int64, seed=11))
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(bits(y), bits(oracle.radix_sort(host(x)))), name


def verdict(evo, fn):
    """"sorted" by the partition sort, "given up" after its counts, or "refused"
    by its sample (or not tried), with the radix passes where they had to run."""
    evo.sync()
    evo.profile(True)
    fn()
    evo.sync()
    recs = evo.profile_read()
    evo.profile(False)
    steps = {r["pass"] for r in recs if r["kind"] == "hybrid" and r["active"]}
    passes = any(r["kind"] == "radix_onesweep" and r["active"] for r in recs)
    got = {frozenset(range(10)): "sorted", frozenset(range(6)) | {9}: "given up", frozenset(): "refused"}[frozenset(steps)]
    assert passes == (got != "sorted")
    return got


VERDICTS = [("uniform", torch.int32, "sorted"), ("uniform", torch.float64, "sorted"), ("float_mix", torch.float64, "sorted"),
            ("zipf", torch.int64, "refused"), ("gaussian", torch.int64, "refused"),
            ("paper_exponential", torch.int32, "refused"), ("outliers", torch.int64, "sorted"),
            ("crowded", torch.int64, "refused"), ("pressed", torch.int64, "given up"), ("frequent", torch.int64, "refused"),
            ("powers", torch.int64, "refused"), ("powers", torch.float64, "refused")]


@pytest.mark.parametrize("table", [False, True], ids=["async", "table"])
@pytest.mark.parametrize("name,dtype,expect", VERDICTS, ids=lambda v: str(v))
def test_verdict(evo, name, dtype, expect, table):
    """How far each kind of keys gets, the same whether the verdict is read back or not."""
    x = gen(name, N, dtype)
    if table:
        for t in TABLES:
            evo.table_load(t)
    y = torch.empty_like(x)
    assert verdict(evo, lambda: evo.sort(x, out=y)) == expect
    assert np.array_equal(bits(y), bits(oracle.radix_sort(host(x))))


@pytest.mark.parametrize("table", [False, True], ids=["async", "table"])
@pytest.mark.parametrize("dtype", [torch.int64, torch.uint64], ids=str)
def test_given_up_after_the_counts(evo, dtype, table):
    """The sample accepts the keys and the counts refuse them: the radix passes
    sort them, in the scratch that the partition sort cleared, and sort other
    keys right after."""
    x = gen("pressed", N, torch.int64).view(dtype)
    want = bits(oracle.radix_sort(host(x)))
    if table:
        for t in TABLES:
            evo.table_load(t)
    y, z = torch.empty_like(x), x.clone()
    for _ in range(3):
        assert verdict(evo, lambda: evo.sort(x, out=y)) == "given up"
        assert np.array_equal(bits(y), want)
        y.zero_()
    evo.sort(z)
    evo.sort(x, out=y, descending=True)
    evo.sync()
    assert np.array_equal(bits(z), want) and np.array_equal(bits(y), want[::-1])


@pytest.mark.parametrize("copies", [10, 40, 300])
@pytest.mark.parametrize("dtype", [torch.int32, torch.int64, torch.float64], ids=str)
def test_repeated_values(evo, dtype, copies):
    """Some copies of every value, spread over the whole type: more of them than
    the local sorts' bins count, fewer than the sample takes for frequent."""
    values = gen("uniform", N // copies, torch.int64)
    pick = gen("uniform", N, torch.int64, seed=copies).remainder(N // copies)
    x = values[pick]
    x = (x >> 32).to(dtype) if dtype == torch.int32 else x.to(dtype)
    want = bits(oracle.radix_sort(host(x)))
    y = torch.empty_like(x)
    assert verdict(evo, lambda: evo.sort(x, out=y)) == "sorted"
    assert np.array_equal(bits(y), want)
    evo.sort(x, out=y, descending=True)
    evo.sync()
    assert np.array_equal(bits(y), want[::-1])
