"""The host's writes to the pinned mirrors of a tile wait for the copies that read them: run_queue over a model of the
tile whose stream runs as late as its order allows (tests/native/queue_uploads.cu), on the CPU."""

import os
import subprocess

import pytest

from paper_2212_04430_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("queue") / "queue_uploads")
    cmd = [build.nvcc()] + build.ARCH + ["-std=c++17", "-O1", "-cudart", "none", "-I" + build.INCLUDE,
                                         "-I" + build.CSRC, os.path.join(HERE, "native", "queue_uploads.cu"),
                                         os.path.join(build.CSRC, "fs_driver.cu"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return out


@pytest.mark.parametrize("kind", ["staged", "single", "chain"])
def test_every_row_is_right_on_the_latest_stream(program, kind):
    r = subprocess.run([program, kind], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
