"""The library's host code without a GPU: its own objects linked with a stand-in for the CUDA runtime
(tests/host), which records the launches and refuses what the runtime would refuse."""
import glob
import os
import re
import subprocess

import pytest


@pytest.fixture(scope="module")
def program(repo_root, tmp_path_factory):
    import __graft_entry__ as g
    g.build()
    from paper_2607_17715_gb300 import build as b
    host = os.path.join(repo_root, "tests", "host")
    exe = str(tmp_path_factory.mktemp("host") / "host_paths")
    cuda = os.path.join(os.path.dirname(os.path.dirname(b._nvcc())), "include")
    cmd = ["g++", "-std=c++17", "-O1", "-I", b.INCLUDE, "-I", host, "-I", cuda, "-o", exe,
           os.path.join(host, "fake_cudart.cpp"), os.path.join(host, "host_paths.cpp"),
           *sorted(glob.glob(os.path.join(b.BUILD_DIR, "*.o")))]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-4000:]
    return exe


def _run(program, *args):
    res = subprocess.run([program, *args], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0, res.stdout + res.stderr
    return res.stdout


def test_register_splits_are_guarded(program):
    kernels = [k for k in _run(program, "kernels").split() if re.search(r"\d(attn_tc\d*_(decode_|sif_)?kernel)", k)]
    assert len(kernels) == 8
    for k in kernels:
        _run(program, "registers", k)


@pytest.mark.parametrize("scenario", ["second_device", "no_partials", "no_queries", "few_rows", "short64"])
def test_scenario(program, scenario):
    _run(program, scenario)
