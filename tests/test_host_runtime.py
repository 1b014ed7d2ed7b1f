"""The host runtime on a CUDA runtime that only keeps books (host_runtime.cpp): lifetimes of
the buffers that captures use, order of the work on a plan's streams, and what a call that
fails leaves behind.  No GPU and no libbbp.so: the runtime's sources, compiled with g++."""

import concurrent.futures
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1008_3171_gb300", "csrc")
SOURCES = ["bbp_runtime.cu", "bbp_prime_run.cu", "bbp_batch.cu", "bbp_serve.cu", "bbp_planner.cpp", "bbp_primes.cpp",
           "bbp_tune.cpp"]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    out = str(tmp_path_factory.mktemp("host_runtime"))
    flags = ["-O1", "-std=c++17", "-pthread", "-I", include, "-I", os.path.join(ROOT, "include"), "-I", CSRC]

    def compile_one(path):
        obj = os.path.join(out, os.path.basename(path) + ".o")
        r = subprocess.run(["g++"] + flags + ["-x", "c++", "-c", path, "-o", obj], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        return obj

    paths = [os.path.join(CSRC, s) for s in SOURCES] + [os.path.join(ROOT, "tests", "host_runtime.cpp")]
    with concurrent.futures.ThreadPoolExecutor() as ex:
        objs = list(ex.map(compile_one, paths))
    exe = os.path.join(out, "host_runtime")
    r = subprocess.run(["g++", "-pthread", "-o", exe] + objs, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("case", ["captured_lists_stay", "sum_quotients", "largest_positions", "no_plan_no_primes",
                                  "failed_batch_leaves_nothing", "unplanned_query_fails",
                                  "failed_iteration_leaves_nothing", "beside_a_capture",
                                  "runs_follow_one_another", "short_ranges_stay_whole",
                                  "short_47_bit_ranges", "one_launch_by_size", "small_groups_spread"])
def test_case(program, case):
    r = subprocess.run([program, case], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
