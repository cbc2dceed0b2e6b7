"""Launches prepare the device that is current.  Shared-memory and cluster
attributes and occupancy answers belong to one device: the library's own
objects, linked with a stand-in runtime that keeps attributes by device, launch
on every one of several devices, and fall back where one takes no cluster."""
import os
import shutil
import subprocess

import pytest

from paper_1406_2686_gb300 import build_lib

HERE = os.path.dirname(os.path.abspath(__file__))
UNITS = ("lbm_small", "lbm_kernels", "lbm_mrt", "fd_kernels", "nn_gemm", "nn_conv")


@pytest.mark.slow
def test_attributes_are_set_on_every_device(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    build_lib.build()
    objs = [os.path.join(build_lib.OUT_DIR, u + ".o") for u in UNITS]
    if not all(os.path.exists(o) for o in objs):
        build_lib.build(force=True)
    main, fake, exe = (str(tmp_path / n) for n in ("main.o", "fake.o", "sites"))
    include = ["-I", build_lib.INCLUDE, "-I", build_lib.CSRC]
    for cmd in ([build_lib.nvcc(), "-c", os.path.join(HERE, "launch_sites.cu"), "-o", main, "-std=c++17",
                 "--expt-relaxed-constexpr"] + build_lib.ARCH + include,
                ["g++", "-c", "-std=c++17", "-O1", os.path.join(HERE, "fake_cudart.cpp"), "-o", fake],
                ["g++", "-o", exe, main, fake] + objs):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-2000:] + r.stderr
