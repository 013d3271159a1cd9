"""The library's host code (csrc/api.cu) on a fake CUDA runtime: several
devices, error words of recycled plans, side streams, scratch in use.  Needs
nvcc, no GPU; every check is a process of its own (process-wide pools)."""
from __future__ import annotations

import concurrent.futures as cf
import os
import re
import subprocess

import pytest

from paper_2606_20855_gb300 import build

HERE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host_runtime")
CHECKS = re.findall(r'^ +\{"(\w+)",', open(os.path.join(HERE, "checks.cu")).read(), re.M)


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    out = tmp_path_factory.mktemp("host_runtime")
    flags = ["-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-I", build.INCLUDE, "-I", build.CSRC, "-I", HERE]

    def run(*args):
        res = subprocess.run([build.nvcc(), *build.ARCH, *args], capture_output=True, text=True)
        assert res.returncode == 0, res.stdout + res.stderr

    srcs = [os.path.join(build.CSRC, "api.cu"), os.path.join(HERE, "checks.cu"),
            os.path.join(HERE, "fake_runtime.cpp")]
    objs = [str(out / (os.path.splitext(os.path.basename(s))[0] + ".o")) for s in srcs]
    with cf.ThreadPoolExecutor(len(srcs)) as ex:
        list(ex.map(lambda so: run(*flags, "-c", so[0], "-o", so[1]), zip(srcs, objs)))
    exe = str(out / "checks")
    run("-cudart", "none", *objs, "-o", exe)
    return exe


@pytest.mark.parametrize("name", CHECKS)
def test_host_runtime(program, name):
    res = subprocess.run([program, name], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout + res.stderr
