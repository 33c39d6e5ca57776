"""Directory entries on their way to the device: where they go in large contexts, and more of them than one launch carries."""
import os
import shutil
import subprocess

import pytest

import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <sys/mman.h>
#include "spin_dev.cuh"
// An entry of a directory region of n words (reserved, never touched): does its index lead back to it?
int main() {
  const size_t words = 6ull << 30;
  void *p = mmap(nullptr, words * 4, PROT_NONE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (p == MAP_FAILED) return 2;
  const int32_t *dirs = (const int32_t *)p;
  for (size_t at : {(size_t)0, (size_t)77, ((size_t)1 << 31) - 1, (size_t)1 << 31, (size_t)2684354560ull, ((size_t)1 << 32) + 5, words - 1}) {
    const spin::DirUpdate u = spin::dir_update(dirs, dirs + at, 9);
    if (dirs + u.at != dirs + at || u.value != 9) { printf("entry %zu goes to %lld\n", at, (long long)u.at); return 1; }
  }
  return 0;
}
"""


def test_entries_beyond_two_to_the_31_words(tmp_path):
    import paper_2604_26837_b200 as P
    from paper_2604_26837_b200 import build
    # accepted, and with more words of directories than 31 bits count: 256 requests, 80 layers, 8 kv heads,
    # a million tokens each, segments of 16 entries
    cfg = P.make_config(device=0, num_layers=80, num_q_heads=64, num_kv_heads=8, max_requests=256, max_context_tokens=1 << 20,
                        partition_kind=P.PART_PAGE_MINMAX, topk=64, segment_entries=16, gpu_cache_pages=70000, host_pages=70000)
    dev, _ = P.spin_required_bytes(cfg)
    n_sets, pages = 256 * 80 * 8, (1 << 16) + 1
    before_sums = n_sets * 4 * ((pages + 15) // 16)       # metadata, offsets, GPU slots, CPU pages
    assert before_sums > 1 << 31 and before_sums * 4 < dev < 180e9
    src, exe = tmp_path / "dirs.cu", tmp_path / "dirs"
    src.write_text(HARNESS)
    nvcc = build._nvcc() if os.path.exists(build._nvcc()) else shutil.which("nvcc")
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-DSPIN_FILE_ID=0", "-I", build.CSRC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("kind,pages", [(W.PART_PAGE_MINMAX, 1400), (W.PART_TOKEN_DOT, 700)])
def test_more_entries_than_one_launch_carries(kind, pages):
    # an append of 1400 pages to 2 heads maps 2 x (3 x 88 + 11) segments of 16 entries, 700 pages of
    # single tokens 2 x (3 x 44 + 44); scores, page lists, residency and counts of every partition against the oracle
    from test_gpu_parity import _wl, run_parity
    w = _wl(kind, num_layers=1, batch=1, num_q_heads=4, num_kv_heads=2, context=16 * pages + 5, topk=300, slots_per_set=320, steps=3)
    assert run_parity(w, segment_entries=16, check_bytes=False)["stats"]["error_bits"] == 0
