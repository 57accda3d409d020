"""The library's scratch on the host (csrc/scratch.cu against a pretended CUDA
runtime): what a growing buffer holds, and that a buffer which a captured graph
may use is never given back, also where memory runs short."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MIB = 1 << 20
OOM = 2  # cudaErrorMemoryAllocation


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("scratch") / "scratch_host.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I",
                    os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2609_10264_gb300", "csrc"), "-I", cuda, "-x", "c++",
                    os.path.join(ROOT, "tests", "scratch_host.cpp"), "-o", out], check=True)
    h = ctypes.CDLL(out)
    h.host_reset.argtypes = [ctypes.c_size_t]
    h.host_used.restype = ctypes.c_size_t
    h.host_live.argtypes = [ctypes.c_void_p]
    h.host_scratch.argtypes = [ctypes.c_size_t, ctypes.POINTER(ctypes.c_void_p)]
    return h


def _get(lib, need):
    p = ctypes.c_void_p()
    return lib.host_scratch(need, ctypes.byref(p)), p.value


def _captured(lib, need):
    lib.host_capturing(1)
    e, p = _get(lib, need)
    lib.host_capturing(0)
    assert e == 0
    return p


def test_captured_buffer_survives_memory_running_short(lib):
    lib.host_reset(100 * MIB)
    assert _get(lib, 40 * MIB)[0] == 0
    graph = _captured(lib, 30 * MIB)
    # 70 MiB beside the 40 do not fit: refused, and the graph's buffer stays
    assert _get(lib, 70 * MIB)[0] == OOM
    assert lib.host_live(graph)
    assert _get(lib, 35 * MIB) == (0, graph)
    # 50 MiB do; later growth keeps both the graph's and one captured since
    e, p = _get(lib, 50 * MIB)
    assert e == 0 and lib.host_live(graph)
    second = _captured(lib, 50 * MIB)
    assert second == p
    assert _get(lib, 60 * MIB)[0] == OOM
    assert lib.host_live(graph) and lib.host_live(second)


def test_bytes_held_by_a_growing_sequence(lib):
    """A stream that was never captured holds one buffer, little more than what is
    needed; one whose every buffer a graph uses, those and at most as much again."""
    lib.host_reset(1 << 40)
    for need in (1, 1000, MIB, 5 * MIB, 40 * MIB, 1000 * MIB, 1100 * MIB):
        assert _get(lib, need)[0] == 0
        assert lib.host_used() <= min(2 * need, need + 32 * MIB)
    lib.host_reset(1 << 40)
    graphs = []
    for need in (MIB, 2 * MIB, 3 * MIB, 100 * MIB, 110 * MIB, 111 * MIB):
        assert _get(lib, need)[0] == 0
        graphs.append(_captured(lib, need))
        assert all(lib.host_live(g) for g in graphs)
        assert lib.host_used() < 4 * need


def test_a_buffer_no_capture_has_seen_makes_room(lib):
    lib.host_reset(100 * MIB)
    assert _get(lib, 60 * MIB)[0] == 0
    assert _get(lib, 90 * MIB)[0] == 0
    assert lib.host_used() < 150 * MIB and lib.host_syncs() >= 1  # the first one went, the stream drained


def test_growth_under_capture_is_refused(lib):
    lib.host_reset(100 * MIB)
    assert _get(lib, 10 * MIB)[0] == 0
    lib.host_capturing(1)
    assert _get(lib, 20 * MIB)[0] not in (0, OOM)
    lib.host_capturing(0)
    assert lib.host_used() == 10 * MIB and _get(lib, 20 * MIB)[0] == 0
