"""What the launchers set up once (kernel attributes, the cluster size, occupancy) is per device:
the compiled launchers run on the CPU against a stand-in for the CUDA runtime that keeps
attributes per device, as the runtime does, and refuses a launch whose shared memory or
cluster size was not allowed on the current one.  Every launcher must work on a second
device as on the first, the cluster must have the size that each device can place, and a
device that can place none must be reported as such and not be launched on."""
import os
import shutil
import subprocess

import pytest

from paper_0905_3409_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
UNITS = ["step2d_small", "step2d", "step2d_vortex", "step2d_fourier", "step2d_linear", "step2d_waves", "step3d", "batch2d",
         "mlp_train_tile", "mlp_infer"]


def test_launch_state_is_per_device(tmp_path):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("no nvcc")
    build.build()
    objs = [os.path.join(build.BUILD, u + ".o") for u in UNITS]
    src, exe, rt = os.path.join(HERE, "native"), str(tmp_path / "device_state"), str(tmp_path / "fake_cudart.o")
    inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    for cmd in (["g++", "-std=c++17", "-I", inc, "-c", os.path.join(src, "fake_cudart.cpp"), "-o", rt],
                [build.nvcc()] + build.ARCH + ["-std=c++17", "-cudart", "none", "-I", build.CSRC,
                                               os.path.join(src, "device_state.cu"), rt, "-o", exe] + objs):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-1000:]
