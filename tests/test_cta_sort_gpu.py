"""GPU parity of the one-CTA sorts of the batched segmented sort (the bin sort
of a short run, the cuts of a long one and the radix passes behind them)
against the oracle: lengths at the edges of each, keys that their range
separates well, badly or not at all."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def evo():
    import paper_2505_18681_gb300 as evo
    evo.library()
    evo.table_clear()
    return evo


def host(t):
    if t.dtype in (torch.uint32, torch.uint64):
        s = t.view(torch.int32 if t.dtype == torch.uint32 else torch.int64).cpu().numpy()
        return s.view(np.uint32 if t.dtype == torch.uint32 else np.uint64)
    return t.cpu().numpy()


def bits(t):
    a = host(t) if isinstance(t, torch.Tensor) else t
    return a.view(np.uint32 if a.dtype.itemsize == 4 else np.uint64)


def powers(n, seed):
    """Magnitudes spread over every binary order."""
    from paper_2505_18681_gb300 import inputs
    x = inputs.generate("uniform", n, torch.int64, seed=seed, device="cuda")
    m = (inputs.generate("uniform", n, torch.int64, seed=seed + 1, device="cuda") & 63).clamp(max=62)
    return (x & ((1 << 62) - 1)) >> m


@pytest.mark.parametrize("dtype", [torch.int32, torch.int64, torch.float64], ids=str)
@pytest.mark.parametrize("kind", ["uniform", "equal", "few", "sparse", "powers", "clusters", "ramp"])
def test_segments_of_every_shape(evo, dtype, kind):
    """Segments at the edges of the one-CTA sorts (a short run, a full local
    sort, one key more, several cuts) whose keys their range separates well,
    badly or not at all."""
    lengths = torch.tensor([2, 31, 255, 256, 257, 1535, 1536, 1537, 4096, 4097, 6143, 6144, 6145, 8191, 8192, 8193,
                            12289, 65536, 100_003, 700_001], dtype=torch.int64)
    offs = torch.zeros(lengths.numel() + 1, dtype=torch.int64)
    offs[1:] = torch.cumsum(lengths, 0)
    n = int(offs[-1])
    from paper_2505_18681_gb300 import inputs
    x = inputs.generate("uniform", n, torch.int64, seed=5, device="cuda")
    if kind == "equal":
        x = torch.full_like(x, -9)
    elif kind == "few":
        x = x % 7
    elif kind == "sparse":
        x = torch.where(x % 10 == 0, x >> 33, torch.zeros_like(x))
    elif kind == "powers":
        x = powers(n, 6)
    elif kind == "clusters":    # half of the keys in 300 values far from the rest
        x = torch.where(x % 2 == 0, (x >> 8) % 300, x)
    elif kind == "ramp":
        x = torch.arange(n, dtype=torch.int64, device="cuda") * 5 - n
    k = x.to(dtype) if dtype != torch.int32 else (x >> (32 if kind in ("uniform", "powers", "clusters") else 0)).to(dtype)
    want = oracle.segmented_sort(host(k), offs.numpy().astype(np.uint64))
    evo.segmented_sort(k, offs.cuda())
    evo.sync()
    assert np.array_equal(bits(k), bits(want))


@pytest.mark.parametrize("dtype", [np.float32, np.float64], ids=["float32", "float64"])
@pytest.mark.parametrize("kind", ["normal", "specials", "orders", "infinite"])
def test_float_segments_cut_by_value(evo, dtype, kind):
    """Float keys are cut by their values: infinities, NaNs and zeros of both
    signs, values whose range is not finite, and ranges that values cut badly."""
    lengths = np.array([0, 1, 255, 257, 1536, 1537, 6144, 6145, 8192, 8193, 50_001, 300_007])
    offs = np.concatenate([[0], np.cumsum(lengths)]).astype(np.uint64)
    r = np.random.default_rng(11)
    n = int(offs[-1])
    x = r.normal(0, 1, n)
    if kind == "orders":
        x = np.ldexp(x, r.integers(-100, 100, n))
    elif kind == "specials":
        x = np.choose(r.integers(0, 12, n), [x * (np.finfo(dtype).max / 64), np.inf, -np.inf, np.nan, -np.nan, 0.0, -0.0] + [x] * 5)
    elif kind == "infinite":
        x = np.where(r.random(n) < 0.5, np.inf, -np.inf)
    x = x.astype(dtype)
    want = oracle.segmented_sort(x, offs)
    k = torch.from_numpy(x.copy()).cuda()
    evo.segmented_sort(k, torch.from_numpy(offs.astype(np.int64)).cuda())
    evo.sync()
    assert np.array_equal(bits(k), bits(want))


def uneven(kind, n, r):
    """int64 keys that bins over the range, or parts of it, separate badly."""
    x = r.integers(-2**62, 2**62, n)
    return {"half": lambda: np.where(r.random(n) < 0.5, 0, x >> 31), "most": lambda: np.where(r.random(n) < 0.995, 7, x),
            "beside": lambda: np.where(r.random(n) < 0.9, 10**9, np.where(r.random(n) < 0.02, 10**9 + r.integers(-3, 4, n), x)),
            "ends": lambda: np.where(r.random(n) < 0.5, 5, np.where(r.random(n) < 0.9, 6, x)),
            "zipf": lambda: np.minimum(r.random(n) ** -2.0, 1e6).astype(np.int64), "hundred": lambda: x % 100,
            "thousand": lambda: x % 1000, "words": lambda: r.integers(-2**62, 2**62, 16)[x % 16],
            "kinds": lambda: r.integers(-2**62, 2**62, 1000)[x % 1000], "powers": lambda: np.abs(x) >> r.integers(0, 62, n),
            "outliers": lambda: np.where(r.random(n) < 0.01, x, np.arange(n)), "short": lambda: x % 40_000}[kind]()


@pytest.mark.parametrize("descending", [False, True], ids=["ascending", "descending"])
@pytest.mark.parametrize("dtype", [np.int32, np.int64, np.float32, np.float64], ids=lambda t: t.__name__)
@pytest.mark.parametrize("kind", ["half", "most", "beside", "ends", "zipf", "hundred", "thousand", "words", "kinds",
                                  "powers", "outliers", "short"])
def test_segments_that_their_range_separates_badly(evo, kind, dtype, descending):
    """Frequent values among others, values that repeat, magnitudes and outliers:
    the ways that take over where bins and cuts do not separate the keys, at the
    sizes where they change, in both directions (floats are cut by value)."""
    lengths = np.array([40, 300, 512, 513, 1500, 1537, 2048, 2049, 4096, 6144, 8192, 8193, 12_000, 40_003, 300_007])
    offs = np.concatenate([[0], np.cumsum(lengths)]).astype(np.uint64)
    r = np.random.default_rng(17)
    x = uneven(kind, int(offs[-1]), r)
    if dtype in (np.float32, np.float64):
        x = x / 2**20
    elif dtype == np.int32 and np.abs(x).max() >= 2**31:
        x = x >> 31
    x = x.astype(dtype)
    want = oracle.segmented_sort(x, offs)
    k = torch.from_numpy(x.copy()).cuda()
    evo.segmented_sort(k, torch.from_numpy(offs.astype(np.int64)).cuda(), descending=descending)
    evo.sync()
    if descending:
        want = np.concatenate([want[int(a):int(b)][::-1] for a, b in zip(offs[:-1], offs[1:])])
    assert np.array_equal(bits(k), bits(want))
