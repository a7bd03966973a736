"""One process with contexts on two devices: every launch of a solve and of a contraction has its shared-memory opt-in
on the device it runs on (the library's objects over a model of the CUDA runtime, tests/native/device_setup.cu)."""

import os
import subprocess

from paper_2212_04430_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_launches_are_opted_in_on_both_devices(tmp_path):
    build.build()
    out = str(tmp_path / "device_setup")
    objs = [os.path.join(build.BUILD, s[:-3] + ".o") for s in build.sources()]
    cmd = [build.nvcc()] + build.ARCH + ["-std=c++17", "-O1", "-cudart", "none", "-I" + build.INCLUDE, "-I" + build.CSRC,
                                         "-Xlinker", "--unresolved-symbols=ignore-all",
                                         os.path.join(HERE, "native", "device_setup.cu")] + objs + ["-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([out], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
