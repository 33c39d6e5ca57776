"""Attention whose flags, turns on the host link or pages do not come: every wait ends, says so, leaves no turn open and
no copy behind, and the outputs are written, or left as they were where a set's first flag does not come to all its rows."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("defines", [[], ["-DSPIN_LANDED_POLLS=0"]])
def test_waits_that_run_out(defines, tmp_path):
    from paper_2604_26837_b200 import build
    exe = tmp_path / "waits"
    flags = [f for f in build.NVCC_FLAGS if f != "-lineinfo"]
    subprocess.check_call([build._nvcc()] + flags + defines + ["-I", build.CSRC, os.path.join(HERE, "attention_waits.cu"), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
