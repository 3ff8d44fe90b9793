"""GPU parity of the one-launch radix sort of mid-sized arrays against the
oracle: sizes at the edges of its chunks and of its range, every key type,
keys and stable pairs, in place and not, and every shortcut it takes on its
own (order, reverse order, narrow and near-zero ranges, digits equal in all
keys)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

ALL = [torch.int32, torch.int64, torch.uint32, torch.uint64, torch.float32, torch.float64]


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


def largest(dtype, pairs):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return sms * 1024 * ((12 if pairs else 16) if dtype.itemsize == 4 else (8 if pairs else 12))


def gen(kind, n, dtype):
    from paper_2505_18681_gb300 import inputs
    if dtype.is_floating_point:
        return inputs.generate("float_mix", n, torch.float64, seed=n, device="cuda").to(dtype)
    if kind == "uniform" or dtype in (torch.uint32, torch.uint64):
        return inputs.generate("uniform", n, dtype, seed=n, device="cuda")
    r = inputs.generate("uniform", n, torch.int64, seed=n, device="cuda")
    x = {"near_zero": lambda: (r & 0xFFFFF) - (1 << 19), "narrow": lambda: (r & 0xFFF) - 77, "few": lambda: r % 5,
         "steps": lambda: (r & 0xFFFF) * 65536 - (1 << 30), "equal": lambda: torch.full_like(r, 3),
         "ramp": lambda: torch.arange(n, device="cuda") * 3 - n, "fall": lambda: n - torch.arange(n, device="cuda") * 2,
         "fall_dup": lambda: -(torch.arange(n, device="cuda") // 3),
         "one_off": lambda: torch.where(torch.arange(n, device="cuda") == n // 2, 0, torch.arange(n, device="cuda"))}[kind]()
    return x.to(dtype)


def launches(evo, fn):
    """Kernels launched, and the kinds of active records."""
    evo.sync()
    k0 = evo.kernel_launches()
    evo.profile(True)
    fn()
    evo.sync()
    recs = evo.profile_read()
    evo.profile(False)
    return evo.kernel_launches() - k0, [r["kind"] for r in recs]


def check(evo, x, **kw):
    want = bits(oracle.radix_sort(host(x)))
    n = x.numel()
    y, z = torch.empty_like(x), x.clone()
    evo.sort(x, out=y, **kw)
    evo.sort(z, **kw)
    d = torch.empty_like(x)
    evo.sort(x, out=d, descending=True, **kw)
    v = torch.arange(n, dtype=torch.int32, device="cuda").view(torch.uint32)
    wk, wv = oracle.radix_sort(host(x), np.arange(n, dtype=np.uint32))
    ko, vo, ki, vi = torch.empty_like(x), torch.empty_like(v), x.clone(), v.clone()
    evo.sort_pairs(x, v, ko, vo, **kw)
    evo.sort_pairs(ki, vi, **kw)
    evo.sync()
    assert np.array_equal(bits(y), want) and np.array_equal(bits(z), want) and np.array_equal(bits(d), want[::-1])
    assert np.array_equal(bits(ko), bits(wk)) and np.array_equal(host(vo), wv)
    assert np.array_equal(bits(ki), bits(wk)) and np.array_equal(host(vi), wv)


@pytest.mark.parametrize("dtype", ALL, ids=str)
@pytest.mark.parametrize("n", [2049, 4097, 5000, 10_000, 65_535, 155_648, 155_649, 1_000_003])
def test_sizes_and_types(evo, dtype, n):
    check(evo, gen("uniform", n, dtype), algo="radix")


@pytest.mark.parametrize("dtype,pairs", [(t, p) for t in (torch.int32, torch.int64) for p in (False, True)], ids=str)
def test_largest_size(evo, dtype, pairs):
    """The last size that goes into one launch, and the first that does not."""
    for n, one in ((largest(dtype, pairs), True), (largest(dtype, pairs) + 1, False)):
        x = gen("uniform", n, dtype)
        v = torch.arange(n, dtype=torch.int32, device="cuda").view(torch.uint32)
        ko, vo = torch.empty_like(x), torch.empty_like(v)
        fn = (lambda: evo.sort_pairs(x, v, ko, vo, algo="radix")) if pairs else (lambda: evo.sort(x, out=ko, algo="radix"))
        count, kinds = launches(evo, fn)
        assert (count == 1) == one and ("radix_fused" in kinds) == one
        wk, wv = oracle.radix_sort(host(x), np.arange(n, dtype=np.uint32))
        assert np.array_equal(bits(ko), bits(wk)) and (not pairs or np.array_equal(host(vo), wv))


@pytest.mark.parametrize("dtype", [torch.int32, torch.int64], ids=str)
@pytest.mark.parametrize("kind", ["near_zero", "narrow", "few", "steps", "equal", "ramp", "fall", "fall_dup", "one_off"])
@pytest.mark.parametrize("n", [3001, 200_003])
def test_shortcuts(evo, dtype, kind, n):
    check(evo, gen(kind, n, dtype), algo="radix")


def test_automatic_calls_and_explicit_tiles(evo):
    x = gen("uniform", 30_000, torch.int32)
    y = torch.empty_like(x)
    want = bits(oracle.radix_sort(host(x)))
    assert launches(evo, lambda: evo.sort(x, out=y))[0] == 1
    assert np.array_equal(bits(y), want)
    for kw in ({"rank_mode": 3}, {"pass_kernel": 1}, {"block_size": 512, "keys_per_thread": 16}, {"digit_bits": 6}):
        assert launches(evo, lambda: evo.sort(x, out=y, algo="radix", **kw))[0] > 1, kw
        assert np.array_equal(bits(y), want)


def test_captured_graph_and_unaligned_views(evo):
    n = 123_457
    x = gen("uniform", n + 1, torch.int64)[1:]
    y = torch.empty(n + 1, dtype=torch.int64, device="cuda")[1:]
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        evo.sort(x, out=y, stream=s)
        evo.sync(s)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            evo.sort(x, out=y, stream=s)
    for kind in ("uniform", "near_zero", "ramp", "narrow"):
        x.copy_(gen(kind, n, torch.int64))
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(bits(y), bits(oracle.radix_sort(host(x)))), kind


def test_two_streams_at_once(evo):
    """Two sorts enqueued on two streams: each waits for all its own CTAs to be
    resident, whatever the other holds."""
    xs = [gen("uniform", 900_001 + i, torch.int32) for i in range(6)]
    ys = [torch.empty_like(x) for x in xs]
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for i, (x, y) in enumerate(zip(xs, ys)):
        evo.sort(x, out=y, algo="radix", stream=streams[i % 2])
    for s in streams:
        evo.sync(s)
    for x, y in zip(xs, ys):
        assert np.array_equal(bits(y), bits(oracle.radix_sort(host(x))))


@pytest.mark.parametrize("pairs", [False, True], ids=["keys", "pairs"])
@pytest.mark.parametrize("dtype,n", [(torch.int32, 1_000_003), (torch.int64, 20_000), (torch.float64, 700_001)], ids=str)
def test_barrier_wait_times_out_and_recovers(evo, dtype, n, pairs):
    """With the poll limit cut to one, the first barrier over the grid runs out:
    the kernel returns, evosort_sync reports ERR_TIMEOUT, and the next sorts with
    the default limit match the oracle."""
    x = gen("uniform", n, dtype)
    v = torch.arange(n, dtype=torch.int32, device="cuda").view(torch.uint32)
    y, w = torch.empty_like(x), torch.empty_like(v)
    sort = (lambda: evo.sort_pairs(x, v, y, w, algo="radix")) if pairs else (lambda: evo.sort(x, out=y, algo="radix"))
    count, kinds = launches(evo, sort)
    assert count == 1 and "radix_fused" in kinds
    evo.set_wait_limit(1)
    try:
        sort()
        with pytest.raises(evo.EvoSortError) as ei:
            evo.sync()
        assert ei.value.status == "ERR_TIMEOUT"
    finally:
        evo.set_wait_limit(0)
    evo.sync()   # the status word was cleared when it was reported
    check(evo, x, algo="radix")


def test_a_named_digit_width_gives_way_to_the_table(evo):
    """With a table loaded an AUTO sort takes the table's digits whatever width
    the call names, below the size of the data-dependent paths too."""
    import os
    tuned = os.path.join(os.path.dirname(evo.__file__), "tuned", "gb300_int32.txt")
    x = gen("uniform", 30_000, torch.int32)
    want = bits(oracle.radix_sort(host(x)))
    y = torch.empty_like(x)
    evo.table_load(tuned)
    for d in (4, 8, 11):
        assert "radix_fused" in launches(evo, lambda: evo.sort(x, out=y, digit_bits=d))[1], d
        assert np.array_equal(bits(y), want)
    evo.table_clear()
    assert "radix_fused" not in launches(evo, lambda: evo.sort(x, out=y, digit_bits=4))[1]
    assert np.array_equal(bits(y), want)
