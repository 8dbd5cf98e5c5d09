"""CPU tests of the serving loop's failure paths: csrc/server.cu compiled
against a CUDA runtime made of host memory (fake_cuda_server.cpp), whose calls
fail on demand."""
import os
import shutil
import subprocess

import pytest

import paper_2310_16298_gb300 as sx

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")


@pytest.fixture(scope="module")
def serve(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path_factory.mktemp("server") / "serve")
    csrc = os.path.join(ROOT, "paper_2310_16298_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-I", csrc, "-I", os.path.join(ROOT, "include"), "-I", CUDA,
                    "-x", "c++", os.path.join(csrc, "server.cu"), os.path.join(HERE, "fake_cuda_server.cpp"),
                    "-lpthread", "-o", exe], check=True)

    def run(what):
        res = subprocess.run([exe, what], capture_output=True, text=True, timeout=60)
        assert res.returncode == 0, (res.returncode, res.stdout, res.stderr)
        return res.stdout.split()
    return run


def test_requests_without_failures(serve):
    assert serve("none") == [str(sx.OK), "17"]


@pytest.mark.parametrize("call", ["copy", "record"])
def test_a_failed_result_copy_fails_the_request(serve, call):
    """Not OK with the result that an earlier request left in the kept buffer."""
    assert serve(call) == [str(sx.ECUDA)]


def test_kept_buffers_make_room_for_a_result(serve):
    """Pinned memory runs out while the server keeps a buffer that is too small."""
    assert serve("pinned") == [str(sx.OK), "17"]
