"""Host: what the runtime enqueues and keeps, checked without a GPU
(tests/host/runtime_check.cpp: pcs_runtime.cpp over a stand-in CUDA runtime,
built here with g++).

upload_order  descriptors written by k_upload are complete before the first
              kernel of the call may read them, over calls of every kind and
              around the sizes where descriptors stop travelling with a launch;
              calls on an idle stream, or that wait for their end, copy them
fork_tables   a block made by forks keeps the section tables of its own
              snapshots only, in a loop of forks too
failed_call   the pinned slot of a call that failed half-way is not given back
              by a later call
"""
import os
import shutil
import subprocess

import pytest

from paper_2607_21686_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    gxx = shutil.which("g++")
    cuda = os.path.join(build._cuda_home(), "include")
    if not gxx or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no g++ or no CUDA headers")
    exe = str(tmp_path_factory.mktemp("runtime") / "runtime_check")
    subprocess.run([gxx, "-O1", "-std=c++17", "-Wno-subobject-linkage", "-I", build.CSRC, "-I", build.INCLUDE, "-I", cuda,
                    os.path.join(ROOT, "tests", "host", "runtime_check.cpp"), "-o", exe, "-ldl"],
                   check=True)
    return exe


@pytest.mark.parametrize("check", ["upload_order", "fork_tables", "failed_call"])
def test_runtime(checker, check):
    out = subprocess.run([checker, check], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
