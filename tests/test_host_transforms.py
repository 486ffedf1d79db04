"""The device code of the line transforms, run on the host (host_cuda/transforms.cpp):
every codelet and every two-step length against the definition of the DFT, and the error
of the double-word arithmetic against that of the published algorithms."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA_INCLUDE = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def transforms(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.isdir(CUDA_INCLUDE):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("host_cuda") / "transforms")
    csrc = os.path.join(ROOT, "paper_1805_04791_gb300", "csrc")
    subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off", "-fpermissive", "-w", "-I", CUDA_INCLUDE, "-I", csrc,
                    os.path.join(HERE, "host_cuda", "transforms.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("part", ["codelets", "double_word"])
def test_transforms(transforms, part):
    """codelets: 16 and 32 roundings of the norm.  double_word: no bound is needed, the
    published operations are the measure: same transforms, same data, no larger an error."""
    r = subprocess.run([transforms, part], capture_output=True, text=True, timeout=600)
    print(r.stdout)
    assert r.returncode == 0, r.stdout[-3000:]
