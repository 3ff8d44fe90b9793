"""Lengths of one segment around the 32-bit limits of the one-CTA tiers: the
counters of the cut (csrc/cta_sort.cuh) restated on the CPU, and one segment
past the limit on the GPU."""
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_18681_gb300", "csrc")
# what the loops of the cut and of its radix passes add to a counter: threads,
# unrolled reads, tiles of both key widths
STEPS = [512, 4 * 512, 8 * 512, 16 * 512, 12 * 512]


@pytest.fixture(scope="module")
def cut_keys(tmp_path_factory):
    """Longest segment that goes to the 32-bit counters (seg_tiers.h)."""
    d = tmp_path_factory.mktemp("tiers")
    (d / "t.cpp").write_text('#include <cstdio>\n#include "seg_tiers.h"\n'
                             'int main() { std::printf("%llu %d\\n", (unsigned long long)evosort::kSegCutKeys,'
                             ' evosort::kSegLongLog2); }\n')
    subprocess.run([shutil.which("g++") or "c++", "-std=c++17", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")],
                   check=True)
    keys, log2 = map(int, subprocess.run([str(d / "t")], check=True, capture_output=True, text=True).stdout.split())
    assert keys == (1 << log2) - 1   # the work list falls by floor(log2) of the length
    return keys


def ends(length, step):
    """Whether `for (uint32_t i = 0; i < length; i += step)` ends: the first
    multiple of step that is not below length, as 32 bits hold it."""
    past = -(-length // step) * step
    return past < 1 << 32


def test_no_counter_of_the_cut_wraps(cut_keys):
    for step in STEPS:
        assert all(ends(length, step) for length in (1, step, step + 1, cut_keys - 1, cut_keys))
        assert cut_keys + step < 1 << 32      # (and a thread's first key is not 0)
    assert not ends((1 << 32) - 1, 8192)      # what the limit keeps out


def test_no_length_is_truncated(cut_keys):
    for length in (cut_keys, cut_keys + 1, (1 << 32) - 1, 1 << 32, (1 << 32) + 5):
        assert length > cut_keys or np.uint32(length & 0xFFFFFFFF) == length


@pytest.mark.gpu
def test_segment_past_the_limit_among_short_ones():
    """2^31 + 77 int32 keys in one segment that no device-wide sort takes: the
    64-bit counters' passes (two digits vary), beside the other tiers."""
    import paper_2505_18681_gb300 as evo
    evo.library()
    evo.table_clear()
    lens = [100, 5000, (1 << 31) + 77, 70_000, 3]
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    n = int(offs[-1])
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 60 GB of device memory")
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    x = torch.randint(600, (n,), dtype=torch.int32, device="cuda", generator=g)
    counts = [sum(torch.bincount(p, minlength=600) for p in x[a:b].split(1 << 28)) for a, b in zip(offs[:-1], offs[1:])]
    evo.segmented_sort(x, torch.from_numpy(offs).cuda(), seg_giant=-1)
    evo.sync()
    for a, b, c in zip(offs[:-1], offs[1:], counts):
        at = torch.cat([c.new_zeros(1), torch.cumsum(c, 0)])
        for v in range(600):   # value v of the segment, where its count says
            assert bool((x[a + int(at[v]):a + int(at[v + 1])] == v).all())
