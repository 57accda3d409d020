"""The host side of a decode (csrc/api.cu against a pretended CUDA runtime): what
it enqueues on which stream, and that a call that fails leaves nothing running
on the context's side stream, whose scratch the next call may use elsewhere."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("decode") / "decode_host")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["g++", "-std=c++17", "-O0", "-w", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2609_10264_gb300", "csrc"), "-I", cuda, "-x", "c++",
                    os.path.join(ROOT, "tests", "decode_host.cpp"), "-Wl,--unresolved-symbols=ignore-all", "-o", out],
                   check=True)
    return lambda *calls: subprocess.run([out, *calls], check=True, capture_output=True, text=True).stdout.split("\n")[:-1]


EARLY = ["challenges side", "record fork caller", "wait fork side", "check side", "decrypt caller", "record join side",
         "wait join caller", "status 0"]
LATE = ["record fork caller", "wait fork side", "challenges side", *EARLY[3:]]


def test_where_the_challenges_run(run):
    """Beside the caller's stream without waiting for it, unless the scratch was
    last used on the caller's stream or a graph may use it."""
    in_place = ["challenges caller", "check caller", "decrypt caller", "status 0"]
    assert run("side", "side") == EARLY + EARLY
    assert run("caller", "side", "side") == ["decode caller", "status 0"] + LATE + EARLY
    assert run("inplace", "side", "side") == in_place + LATE + EARLY
    assert run("captured", "side") == LATE + LATE


@pytest.mark.parametrize("before", [[], ["caller"]])
@pytest.mark.parametrize("fail", range(7))
def test_a_failed_call_leaves_the_side_stream_idle(run, before, fail):
    log = run(*before, f"side:{fail}", "caller")
    log = log[2 * len(before):]
    end = log.index("status -4")
    assert log[end + 1:] == ["decode caller", "status 0"]
    side = [i for i, line in enumerate(log[:end]) if line.endswith("side")]
    if side:
        assert "synchronize" in log[side[-1]], log
