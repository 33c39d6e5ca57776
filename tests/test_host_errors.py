"""The host runtime on a stand-in for the CUDA runtime (tests/cuda_stand_in.c): launches that fail, errors that other calls
have left behind, and the device on which calls without a stream work."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = r"""
import ctypes as C
import sys
sys.path.insert(0, %r)
import paper_2604_26837_b200.binding as B
cuda, lib = C.CDLL(%r), B.load()

def context(**kw):
    cfg = B.make_config(**dict(dict(device=0, num_layers=2, num_q_heads=2, num_kv_heads=2, max_requests=4, max_context_tokens=4096,
                                    partition_kind=B.PART_PAGE_MINMAX, topk=8, segment_entries=16, gpu_cache_pages=4 * 64, host_pages=64), **kw))
    cfg.hbm_pool, cfg.hbm_pool_bytes = 1 << 40, B.spin_required_bytes(cfg)[0]       # an address range, never touched
    h = C.c_void_p()
    assert lib.spin_create(C.byref(cfg), C.byref(h)) == 0
    return h

def opened(h, slots):
    r = C.c_int32(-1)
    return lib.spin_request_open(h, slots, C.byref(r)), r.value

def in_use(h):
    s = B.spin_stats_t()
    s.struct_size = C.sizeof(B.spin_stats_t)
    assert lib.spin_stats(h, C.byref(s)) == 0
    return s.gpu_pages_in_use, s.gpu_meta_bytes
"""

OK, CUDA = 0, 6


@pytest.fixture(scope="module")
def stand_in(tmp_path_factory):
    so = tmp_path_factory.mktemp("cuda") / "stand_in.so"
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-O1", os.path.join(HERE, "cuda_stand_in.c"), "-o", str(so)])

    def run(body):
        r = subprocess.run([sys.executable, "-c", PRELUDE % (ROOT, str(so)) + body], capture_output=True, text=True,
                           env=dict(os.environ, LD_PRELOAD=str(so)))
        assert r.returncode == 0, r.stdout + r.stderr
    return run


def test_an_error_left_behind_by_others(stand_in):
    # neither opening nor closing takes it for its own, nor takes it away
    stand_in("""
h = context()
cuda.stand_in_stale(101)
assert opened(h, 64) == (0, 0) and in_use(h)[0] == 4 * 64
assert lib.spin_request_close(h, 0) == 0 and in_use(h) == (0, 0)
assert cuda.cudaGetLastError() == 101
""")


def test_open_that_fails_holds_nothing(stand_in):
    # any of its copies, segments together or (every second one taken) in pieces
    stand_in("""
for turn in range(3):
    h = context()
    cuda.stand_in_fail(turn)
    assert opened(h, 64)[0] == 6 and in_use(h) == (0, 0)
    assert opened(h, 64) == (0, 0) and in_use(h)[0] == 4 * 64      # the whole budget is there
    assert opened(h, 1)[0] == 5                                     # ... and no more
h = context(num_layers=1, num_kv_heads=1, num_q_heads=1, gpu_cache_pages=128)
for r in range(4):
    assert opened(h, 16) == (0, r)
assert lib.spin_request_close(h, 0) == 0 and lib.spin_request_close(h, 2) == 0
held = in_use(h)
for turn in range(4):
    cuda.stand_in_fail(turn)
    assert opened(h, 48)[0] == 6 and in_use(h) == held
assert opened(h, 48) == (0, 0)
""")


def test_close_that_fails_has_closed(stand_in):
    stand_in("""
h = context()
assert opened(h, 64) == (0, 0)
cuda.stand_in_fail(0)
assert lib.spin_request_close(h, 0) == 6 and in_use(h) == (0, 0)
assert lib.spin_request_close(h, 0) == 2                           # not open any more
assert opened(h, 64) == (0, 0)
""")


def test_calls_without_a_stream_work_on_the_contexts_device(stand_in):
    # a context of the second device, the first one current
    stand_in("""
h = context(device=1)
cuda.cudaSetDevice(0)
before = cuda.stand_in_launches(1)
assert opened(h, 64) == (0, 0)
for slots in (32, 48):                                             # a kernel reclaims what a smaller budget gives up
    assert lib.spin_set_budget(h, 0, slots) == 0
assert in_use(h)[0] == 4 * 48
page = (C.c_uint8 * 8192)()
assert lib.spin_debug_read_page(h, 0, 0, 0, 0, 0, 0, page) == 0
assert lib.spin_profile(h, 0) == 0
assert lib.spin_request_close(h, 0) == 0 and lib.spin_destroy(h) == 0
d = C.c_int(-1)
cuda.cudaGetDevice(C.byref(d))
assert d.value == 0 and cuda.stand_in_launches(0) == 0 and cuda.stand_in_launches(1) - before == 1
assert cuda.stand_in_synced(0) == 0 and cuda.stand_in_synced(1) > 0
""")
