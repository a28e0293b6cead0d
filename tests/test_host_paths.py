"""The host side of the copies and pools, against a fake of the CUDA runtime (host_paths.cu)."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("host_paths") / "host_paths")
    subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "none", "-o", out,
                    os.path.join(HERE, "host_paths.cu"), os.path.join(HERE, "host_paths_fake.cpp"), "-lpthread"], check=True, capture_output=True, text=True)
    return out


@pytest.mark.parametrize("scenario", ["copies", "launch fails in workers", "launch fails", "device pointer", "no host memory",
                                      "asking for free memory"])
def test_host_path(program, scenario):
    p = subprocess.run([program, scenario], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, p.stdout + p.stderr
