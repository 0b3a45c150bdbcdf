"""Host-side index and size arithmetic of the CUDA sources, compiled with
nvcc and run on the CPU (nothing in it touches a GPU)."""
import os
import shutil
import subprocess

import pytest

import paper_2404_19634_gb300 as dfl

CSRC = os.path.join(os.path.dirname(dfl.__file__), "csrc")


def run_host(tmp_path, body):
    """The words that main(), with `body` as its text, prints."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "host.cu"
    src.write_text('#include <cstdio>\n#include <cinttypes>\n#include "common.cuh"\n'
                   "using namespace dfl;\nint main() {\n" + body + "\n}\n")
    exe = str(tmp_path / "host")
    out = subprocess.run([nvcc, *dfl.NVCC_FLAGS, "-I", CSRC, str(src), "-o", exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    return [int(x) for x in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()]


@pytest.mark.parametrize("n", [10, 2**32 // 6 + 1, 2**31 - 1])
@pytest.mark.parametrize("k", [1, 4, 8])
def test_frontier_segments_do_not_overlap(tmp_path, n, k):
    """Every (class, bin) segment follows the one before, up to the largest n
    that dfl_create takes."""
    counts = [n // k + (s < n % k) for s in range(k)] + [0] * (8 - k)
    got = run_host(tmp_path, """
  const uint64_t counts[kMaxSubsteps] = {%s};
  Segs seg;
  layout_segs(seg, counts, %d);
  std::printf("%%d\\n", kBins);
  for (uint32_t q = 0; q < kMaxSubsteps * kBins; ++q)
    std::printf("%%" PRIu64 " %%u\\n", uint64_t(seg.off[q]), seg.cap[q]);
""" % (", ".join("%dull" % c for c in counts), k))
    bins, off, cap = got[0], got[1::2], got[2::2]
    at = 0
    for s in range(8):
        for b in range(bins):
            assert off[s * bins + b] == at and cap[s * bins + b] == counts[s]
            at += counts[s]
    assert at == bins * n  # what the list buffers hold


@pytest.mark.parametrize("lim,rows", [
    (4096, [(4097, 1024)] * 4098),                       # every row as full of tombstones as a row can be
    (4096, [(4097, 0), (9000, 2250), (131_073, 7)]),
    (32, [(33, 8), (40, 10), (35, 8)] * 50),
    (31, [(32, 8), (33, 8)] * 9),
    (0, [(9, 8), (1, 1), (8, 8), (30, 8)] * 20),         # short rows: tombstones alone, or nearly
])
def test_slots_bound_covers_tombstones(tmp_path, lim, rows):
    """Buffers sized for the degrees (slots in use) of the rows above a limit
    hold them when the rows carry tombstones, which the live arcs leave out."""
    assert all(d > lim and t <= max(8, d // 4) for d, t in rows)
    slots, tombs = sum(d for d, _ in rows), sum(t for _, t in rows)
    exact, loose = run_host(tmp_path, """
  std::printf("%%" PRIu64 " %%" PRIu64 "\\n", slots_bound(%dull, %dull, %du), slots_bound(%dull, %dull, %du));
""" % (slots - tombs, tombs, lim, slots - tombs, tombs * 1000, lim))
    assert exact >= slots  # the tombstones are known exactly ...
    if lim >= 32:          # ... or only by a bound far above them
        assert slots <= loose <= slots * 4 // 3
