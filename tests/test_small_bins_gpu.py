"""GPU parity of the one-CTA small sort against the oracle on keys that its
bins separate well, badly or not at all: sizes at the edges of its compiled
shapes, frequent values, and floats whose positions are taken from their
values (infinities, NaNs of both signs, zeros of both signs, denormals, the
widest and the narrowest ranges)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

SIZES = [2, 3, 33, 511, 1000, 1023, 1024, 1025, 2049, 4095, 4096, 4097, 8191, 8192]


@pytest.fixture(scope="module")
def evo():
    import paper_2505_18681_gb300 as evo
    evo.library()
    evo.table_clear()
    return evo


def bits(a):
    a = a.cpu().numpy() if isinstance(a, torch.Tensor) else a
    return a.view(np.uint32 if a.dtype.itemsize == 4 else np.uint64)


def ints(kind, n, dtype):
    r = np.random.default_rng(n)
    lo, hi = np.iinfo(dtype).min, np.iinfo(dtype).max
    return {"spread": lambda: r.integers(lo, hi, n, dtype=dtype, endpoint=True),
            "few": lambda: r.integers(0, 5, n).astype(dtype), "equal": lambda: np.full(n, -7, dtype),
            "pairs": lambda: (r.integers(0, n, n) // 2).astype(dtype),
            "clump": lambda: np.where(r.random(n) < 0.5, r.integers(0, 40, n), r.integers(lo // 2, hi // 2, n)).astype(dtype),
            "late": lambda: np.where((np.arange(n) < 512) | (r.random(n) < 0.5), hi, r.integers(lo, lo + 99, n)).astype(dtype),
            "ends": lambda: np.where(r.random(n) < 0.5, lo, hi).astype(dtype)}[kind]()


def floats(kind, n, dtype):
    r = np.random.default_rng(n)
    info = np.finfo(dtype)
    x = {"uniform": lambda: r.uniform(-1e6, 1e6, n), "normal": lambda: r.normal(0, 1, n),
         "orders": lambda: np.ldexp(r.uniform(-1, 1, n), r.integers(-100, 100, n)),
         "specials": lambda: r.uniform(-1, 1, n), "tiny": lambda: r.integers(0, 50, n) * float(info.smallest_subnormal),
         "wide": lambda: np.where(r.random(n) < 0.5, -1.0, 1.0) * float(info.max) * r.uniform(0.4, 1, n),
         "close": lambda: 1.0 + r.integers(0, 3 * n, n) * float(info.eps), "infinite": lambda: np.full(n, np.inf)}[kind]()
    x = x.astype(dtype)
    if kind in ("specials", "infinite"):
        neg_nan = np.copysign(np.array([np.nan], dtype), dtype(-1))
        pick = r.integers(0, 12, n)
        for i, v in enumerate((np.inf, -np.inf, np.nan, -0.0, 0.0)):
            x[pick == i] = v
        x[pick == 5] = neg_nan[0]
    return x


def check(evo, a):
    n = a.size
    x = torch.from_numpy(a.copy()).cuda()
    v = torch.arange(n, dtype=torch.int32, device="cuda").view(torch.uint32)
    want = bits(oracle.radix_sort(a))
    wk, wv = oracle.radix_sort(a, np.arange(n, dtype=np.uint32))
    y, z, d = torch.empty_like(x), x.clone(), torch.empty_like(x)
    ko, vo, ki, vi = torch.empty_like(x), torch.empty_like(v), x.clone(), v.clone()
    kd, vd = torch.empty_like(x), torch.empty_like(v)
    k0 = evo.kernel_launches()
    evo.sort(x, out=y, small_cap=8192)
    evo.sort(z, small_cap=8192)
    evo.sort(x, out=d, small_cap=8192, descending=True)
    evo.sort_pairs(x, v, ko, vo, small_cap=8192)
    evo.sort_pairs(ki, vi, small_cap=8192)
    evo.sort_pairs(x, v, kd, vd, small_cap=8192, descending=True)
    evo.sync()
    assert evo.kernel_launches() - k0 == 6
    assert np.array_equal(bits(y), want) and np.array_equal(bits(z), want) and np.array_equal(bits(d), want[::-1])
    for k, w in ((ko, vo), (ki, vi)):
        assert np.array_equal(bits(k), bits(wk)) and np.array_equal(w.view(torch.int32).cpu().numpy().view(np.uint32), wv)
    # descending and stable: equal keys in input order
    assert np.array_equal(bits(kd), want[::-1])
    w = vd.view(torch.int32).cpu().numpy()
    assert np.array_equal(bits(a)[w], want[::-1])
    same = want[::-1][1:] == want[::-1][:-1]
    assert np.all(np.diff(w)[same] > 0)


@pytest.mark.parametrize("dtype", [np.int32, np.int64], ids=["int32", "int64"])
@pytest.mark.parametrize("kind", ["spread", "few", "equal", "pairs", "clump", "ends", "late"])
def test_integers(evo, dtype, kind):
    for n in SIZES:
        check(evo, ints(kind, n, dtype))


@pytest.mark.parametrize("dtype", [np.float32, np.float64], ids=["float32", "float64"])
@pytest.mark.parametrize("kind", ["uniform", "normal", "orders", "specials", "tiny", "wide", "close", "infinite"])
def test_floats(evo, dtype, kind):
    for n in SIZES:
        check(evo, floats(kind, n, dtype))


@pytest.mark.parametrize("dtype", [np.int32, np.float32, np.int64], ids=["int32", "float32", "int64"])
@pytest.mark.parametrize("kind", ["spread", "few", "clump", "late", "ends", "normal", "specials"])
def test_arrays_the_dispatcher_gives_to_one_cta(evo, dtype, kind):
    """Above the default cut-over, with the choice left to the library: the
    last size of each width that one CTA takes and the first that it does not."""
    if (dtype == np.float32) != (kind in ("normal", "specials")):
        pytest.skip("a kind of the other key types")
    for n in (4097, 8191, 8192, 8193, 12289, 15359, 15360, 15361):
        a = floats(kind, n, dtype) if dtype == np.float32 else ints(kind, n, dtype)
        x = torch.from_numpy(a.copy()).cuda()
        y, d = torch.empty_like(x), torch.empty_like(x)
        evo.sync()
        evo.profile(True)
        try:
            evo.sort(x, out=y)
            evo.sync()
            kinds = [r["kind"] for r in evo.profile_read()]
        finally:
            evo.profile(False)
        evo.sort(x, out=d, descending=True)
        evo.sync()
        want = oracle.radix_sort(a)
        assert np.array_equal(bits(y), bits(want)) and np.array_equal(bits(d), bits(want)[::-1]), n
        assert (kinds == ["small"]) == (n <= (15360 if a.itemsize == 4 else 8192)), n


def uneven(kind, n, r):
    x = r.integers(-2**62, 2**62, n)
    return {"powers": lambda: np.abs(x) >> r.integers(0, 62, n), "zipf": lambda: np.minimum(r.random(n) ** -2.0, 1e6).astype(np.int64),
            "half": lambda: np.where(r.random(n) < 0.5, 0, x >> 31), "clumps": lambda: (x >> 50 << 50) + r.integers(0, 9, n),
            "outliers": lambda: np.where(r.random(n) < 0.02, x, np.arange(n) // 3)}[kind]()


@pytest.mark.parametrize("dtype", [np.int32, np.int64, np.float32, np.float64], ids=lambda t: t.__name__)
@pytest.mark.parametrize("kind", ["powers", "zipf", "half", "clumps", "outliers"])
def test_keys_that_crowd_together(evo, kind, dtype):
    """Words of many keys, which the size limits, and the bitonic runs and merge
    rounds behind them, at the sizes where they change."""
    for n in (3, 12, 13, 50, 128, 129, 300, 512, 513, 1024, 1025, 2048, 2049, 3000, 4096, 4097, 8192):
        x = uneven(kind, n, np.random.default_rng(n))
        if dtype in (np.float32, np.float64):
            x = x / 2**20
        elif dtype == np.int32 and np.abs(x).max() >= 2**31:
            x = x >> 31
        check(evo, x.astype(dtype))
