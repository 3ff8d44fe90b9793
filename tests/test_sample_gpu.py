"""GPU parity of the dispatcher's sample: the class that the device reads off an
array against the class that the host reads off a copy of it, at the edges of
the sample's size, for every key type and kind of order and repetition."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = [2, 3, 31, 33, 1025, 4095, 4096, 4097, 8191, 100_003]
DTYPES = {"int32": torch.int32, "uint32": torch.uint32, "float32": torch.float32,
          "int64": torch.int64, "uint64": torch.uint64, "float64": torch.float64}


@pytest.fixture(scope="module")
def evo():
    import paper_2505_18681_gb300 as evo
    evo.library()
    evo.table_clear()
    evo.table_set(torch.int32, 20, "random", {"algo": "radix"})   # (the host classifies with a table only)
    yield evo
    evo.table_clear()


def keys(kind, n, r):
    u = r.integers(-2**63, 2**63 - 1, n, endpoint=True)
    i = np.arange(n)
    return {"uniform": lambda: u, "equal": lambda: u * 0 - 3, "sorted": lambda: np.sort(u),
            "reverse": lambda: np.sort(u)[::-1].copy(), "sorted_but_one": lambda: np.where(i == n // 2, u, np.sort(u)),
            "few64": lambda: (i * 2654435761 % 64 - 9) * 2**50, "few65": lambda: (i * 2654435761 % 65 - 9) * 2**50,
            "threes": lambda: (i // 3 * 40503 % 65536) * 2**40, "narrow16": lambda: u % 50_000, "narrow": lambda: u % 2**30,
            "quarter": lambda: np.where(i % 4 == 0, 7, u), "zeros": lambda: np.where(r.random(n) < 0.9, 0, u)}[kind]()


@pytest.mark.parametrize("name", list(DTYPES))
@pytest.mark.parametrize("kind", ["uniform", "equal", "sorted", "reverse", "sorted_but_one", "few64", "few65", "threes",
                                  "narrow16", "narrow", "quarter", "zeros"])
def test_device_class_is_the_hosts(evo, name, kind):
    for n in SIZES:
        x = keys(kind, n, np.random.default_rng(n))
        if name.endswith("32") and kind not in ("narrow16", "narrow"):
            x = x >> 32
        x = x.view(np.uint64).astype(name) if name.startswith("uint") else x.astype(name)
        host = torch.from_numpy(x.view(name.replace("uint", "int"))).view(DTYPES[name])
        assert evo.classify(host.cuda()) == evo.plan_host(host)[1], n
