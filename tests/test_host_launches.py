"""The library's host code (plans, block sizes, launch configurations) against
a stand-in for the CUDA runtime: no GPU is needed and no kernel runs."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_0812_0244_gb300 import build
    build.build()
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    exe = str(tmp_path_factory.mktemp("fake") / "fake_cuda")
    cmd = [shutil.which("g++") or "c++", "-std=c++17", "-O1", "-I", inc, os.path.join(HERE, "fake_cuda.cpp"), *objs,
           "-lpthread", "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return exe


def run(exe, *args):
    r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, (r.returncode, r.stdout[-3000:])


@pytest.mark.parametrize("Nq", [8, 20])
def test_block_sizes_of_many_small_planes(fake, Nq):
    """More than 32 planes per SM still leave each block at least one warp."""
    run(fake, "planes", Nq)


def test_batch_workspaces_are_cleared_before_vdw_plan_batch_returns(fake):
    """The caller's stream need not wait for the default stream."""
    run(fake, "batch")


def test_learned_parameters_are_laid_out_after_their_memory_is_cleared(fake):
    run(fake, "learned")
