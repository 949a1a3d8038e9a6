"""Device memory of the library's objects (memory.cu) and the server's admission
by it (server.cu) compiled by the host compiler against a stand-in for the CUDA runtime: two devices, threads without
a context, addresses that come back.  No GPU needed."""

import os
import shutil
import subprocess

import pytest

from paper_2310_11186_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b.nvcc()))), "include")
    exe = str(tmp_path_factory.mktemp("blocks") / "blocks")
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-I", b.INCLUDE, "-I", b.CSRC, "-isystem", cuda, "-x", "c++",
                        os.path.join(b.CSRC, "memory.cu"), os.path.join(b.CSRC, "server.cu"), os.path.join(HERE, "cuda_memory_stub.cpp"), "-pthread",
                        "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("scenario", ["other_device", "fresh_thread", "two_devices", "idle_bound", "account", "limit",
                                      "per_thread_stream", "server_admission"])
def test_blocks(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
