"""Host-side ordering and memory of the library, without a GPU: its objects linked to a
CUDA runtime that runs nothing and records the calls (host_cuda/)."""
import os
import shutil
import subprocess

import pytest

import __graft_entry__ as entry

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA_INCLUDE = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    """program(name): host_cuda/<name>.cpp linked to the library's objects and the stand-in runtime."""
    gxx = shutil.which("g++")
    if gxx is None or not os.path.isdir(CUDA_INCLUDE):
        pytest.skip("needs g++ and the CUDA headers")
    entry.build()
    from paper_1805_04791_gb300 import build as b

    objs = [os.path.join(b.BUILD, s.replace(".cu", ".o")) for s in b.SOURCES]
    out = tmp_path_factory.mktemp("host_cuda")

    def make(name):
        exe = str(out / name)
        src = [os.path.join(HERE, "host_cuda", f) for f in (f"{name}.cpp", "fake_cuda.cpp")]
        subprocess.run([gxx, "-std=c++17", "-O1", "-I", CUDA_INCLUDE, "-I", os.path.join(ROOT, "include"), *src, *objs,
                        "-o", exe, "-lpthread"], check=True)
        return exe

    return make


def test_problem_bytes_is_what_a_problem_holds(program):
    """At least the most that create, a mixed solve and the scattered field hold together,
    and at most 5 % and 256 KiB (small buffers) more."""
    r = subprocess.run([program("problem_bytes")], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, "\n".join(v for v in r.stdout.splitlines() if v.startswith("BAD"))


def test_kept_memory_is_bounded_and_given_back(program):
    r = subprocess.run([program("pool_limits")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:]


def test_calls_work_after_a_refused_allocation(program):
    r = subprocess.run([program("refused_memory")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:]


def test_solve_that_ends_early_leaves_nothing_running(program):
    r = subprocess.run([program("early_end")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:]
