"""How a launch of attention deals sets to CTAs, as the host decides it: which lists go to clusters of which size, to CTAs that merge
through memory, to CTAs that count."""
import os
import subprocess

import pytest

from test_gpu_cluster_merge import SHAPES

HERE = os.path.dirname(os.path.abspath(__file__))
WARP, COUNTED, ROWS = 0, 1, 2


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    from paper_2604_26837_b200 import build
    exe = str(tmp_path_factory.mktemp("plan") / "plan")
    subprocess.check_call([build._nvcc(), "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", build.CSRC,
                           os.path.join(HERE, "attention_plan.cu"), "-o", exe])

    def ask(*args, beside=0):
        text = "".join("%d %d %d %d %d\n" % (decode, beside, sets, pages, (pages + 7) // 8) for decode, sets, pages in args)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    ask.exe = exe
    return ask


def test_every_plan(plans):
    r = subprocess.run([plans.exe, "all"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_clusters_leave_a_margin(plans):
    # as many sets as the runtime says that clusters fit, and the most that are there at once
    got = plans((0, 142, 24), (0, 138, 24), (0, 104, 24), (0, 101, 24), (0, 82, 40), (0, 80, 40), (0, 71, 40), (0, 69, 40), (0, 57, 28), (0, 56, 28),
                (0, 222, 40), (0, 49, 29), (0, 48, 29))
    assert [g[2] for g in got] == [0, 3, 3, 4, 0, 5, 5, 6, 6, 7, 2, 7, 8]


def test_plain_lists(plans):
    got = plans((0, 1, 4), (0, 16000, 1), (0, 256, 56), (0, 72, 354), (0, 148, 33), (0, 8, 80))
    assert got == [(ROWS, 1, 0), (WARP, 1, 0), (ROWS, 1, 0), (COUNTED, 720, 0), (ROWS, 3, 0), (ROWS, 10, 0)]


def test_decode_steps_beside_a_scoring_grid(plans):
    # single CTAs find room there before clusters do
    steps = (1, 64, 65), (1, 64, 129), (1, 32, 33), (1, 8, 17)
    assert [g[1:] for g in plans(*steps)] == [(6, 6), (6, 6), (8, 8), (5, 5)]
    assert [g[1:] for g in plans(*steps, beside=1)] == [(6, 0), (6, 0), (5, 0), (3, 0)]


def test_what_the_cluster_tests_run(plans):
    assert [g[2] for g in plans(*((0, sets, pages) for sets, _, pages, _ in SHAPES))] == [cluster for *_, cluster in SHAPES]
    assert {cluster for *_, cluster in SHAPES} == {0, 2, 3, 4, 5, 6, 7, 8}
    # its decode steps: five requests of 8, 4 and 2 kv heads
    assert [g[2] for g in plans((1, 40, 41), (1, 20, 61), (1, 10, 41))] == [8, 8, 8]
