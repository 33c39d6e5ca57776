"""What a call marks to leave L2 first: steps and lists that L2 holds until they are read again are not spoiled."""
import subprocess

import pytest

HARNESS = r"""
#include <cstdio>
#include "spin_dev.cuh"
using namespace spin;
int main() {
  int kind;
  double summaries, pages;
  while (scanf("%d %lf %lf", &kind, &summaries, &pages) == 3) printf("%d\n", kind < 0 ? lists_read_once(pages) : step_reads_once(kind, summaries, pages));
}
"""
LISTS, PAGE, TOKEN, CLUSTER, MEAN = -1, 0, 1, 2, 3
SUMMARIES, PAGES = 1, 2


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    from paper_2604_26837_b200 import build
    d = tmp_path_factory.mktemp("once")
    (d / "once.cu").write_text(HARNESS)
    subprocess.check_call([build._nvcc(), "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-DSPIN_FILE_ID=0", "-I", build.CSRC, str(d / "once.cu"), "-o", str(d / "once")])

    def run(kind, summaries, pages):
        return int(subprocess.run([str(d / "once")], input="%d %f %f\n" % (kind, summaries, pages), capture_output=True, text=True, check=True).stdout)
    return run


def test_plain_lists(ask):
    mb = 8192 / 1e6
    for sets, pages, want in ((444, 10, 0), (1024, 8, 0), (256, 40, 0), (222, 48, PAGES), (148, 80, PAGES), (256, 56, PAGES)):
        assert ask(LISTS, 0, sets * pages * mb * 1e6) == want, (sets, pages)


def test_decode_steps(ask):
    assert ask(PAGE, 8.4e6, 8.5e6) == 0
    assert ask(PAGE, 17e6, 34e6) == PAGES and ask(MEAN, 8.7e6, 68e6) == PAGES and ask(CLUSTER, 4e6, 60e6) == PAGES
    assert ask(PAGE, 25e6, 67e6) == PAGES and ask(PAGE, 67e6, 67e6) == PAGES | SUMMARIES
    assert ask(TOKEN, 67e6, 10e6) == PAGES | SUMMARIES and ask(TOKEN, 10e6, 10e6) == 0
