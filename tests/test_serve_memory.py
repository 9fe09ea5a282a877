"""The server on a fake device (tests/fake_cuda/serve_memory.cpp): what it keeps for later requests
is given back when an allocation fails, and when it has nothing to do."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if not shutil.which("g++") or not os.path.exists(f"{cuda}/include/cuda_runtime.h"):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("fake") / "serve_memory")
    csrc = os.path.join(ROOT, "paper_2506_16045_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-pthread", f"-I{cuda}/include",
                    f"-I{ROOT}/include", f"-I{csrc}", f"{HERE}/fake_cuda/serve_memory.cpp",
                    "-x", "c++", f"{csrc}/sgn_serve.cu", "-o", exe], check=True)
    return lambda what: subprocess.run([exe, what], check=True, timeout=60, capture_output=True,
                                       text=True).stdout.split("\n")


@pytest.mark.parametrize("what", ["submit", "state", "solve1d", "pack1d", "run1d", "multistep1d"])
def test_a_failed_allocation_takes_what_is_kept(fake, what):
    assert fake(what)[0].startswith("status 0 ")


def test_what_does_not_fit_is_still_refused(fake):
    assert fake("too_large")[0].startswith("status 3 ")


def test_an_idle_server_gives_its_memory_back(fake):
    out = fake("idle")
    assert out[0] == "status 0 iters 0" and out[1] == "left 0 blocks"


def test_a_layout_without_a_solve_graph_is_not_kept(fake):
    """Its solves are host-driven (report 2 here): later requests must not inherit that."""
    assert fake("graph")[0] == "status 0 iters 1"
