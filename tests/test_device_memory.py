"""Allocation of device memory when there is little of it (csrc/dev_mem.h over a fake device): what a
handle can do without gives way, and a failed allocation is reported once, by the call that made it."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2101_02959_gb300", "csrc")


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cxx = shutil.which("g++")
    cuda = "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are not available")
    out = str(tmp_path_factory.mktemp("mem") / "dev_mem")
    src = os.path.join(ROOT, "tests", "native", "dev_mem_harness.cpp")
    r = subprocess.run([cxx, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", cuda, src, "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def answers(*commands):
        r = subprocess.run([out], input="\n".join(commands) + "\n", capture_output=True, text=True, check=True)
        return r.stdout.split("\n")[:-1]
    return answers


def test_optional_memory_keeps_the_spare(run):
    assert run("device 1000", "alloc 300", "optional 500 200", "optional 1 200", "optional 1 199") == \
        ["ok", "700", "200", "none", "199"]


def test_workspace_shrinks_to_what_there_is(run):
    # as wanted; halved until the spare is left; the least whatever it leaves; refused below that
    assert run("device 1000", "between 100 600 200") == ["ok", "600 400"]
    assert run("device 1000", "between 100 900 200") == ["ok", "450 550"]
    assert run("device 1000", "alloc 750", "between 100 800 200") == ["ok", "250", "100 150"]
    assert run("device 1000", "alloc 950", "between 100 800 200", "error") == ["ok", "50", "nomem", "0"]
    assert run("device 1000", "between 100 100 950") == ["ok", "100 900"]


def test_failed_allocation_leaves_no_error_behind(run):
    assert run("device 100", "alloc 200", "error", "alloc 60", "drop") == ["ok", "nomem", "0", "40", "100"]


def test_released_memory_comes_back_once(run):
    assert run("device 100", "alloc 30", "alloc 50", "release", "drop") == ["ok", "70", "20", "70", "100"]
