"""Device arrays of a caller are read by a kernel only where that kernel may
dereference them; the memory of a second GPU and pinned host memory go through
a staging area and the copy engine (no GPU needed: the rule and the room)."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))
UNREGISTERED, HOST, DEVICE, MANAGED = 0, 1, 2, 3   # cudaMemoryType


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "libreach.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", os.path.join(cuda, "include"), "-I",
                    os.path.join(ROOT, "paper_2606_17772_gb300", "csrc"), "-o", out,
                    os.path.join(HERE, "array_reach_probe.cpp"), "-L", os.path.join(cuda, "lib64"), "-lcudart"],
                   check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("kind,where,here,direct", [
    (DEVICE, 0, 0, 1), (DEVICE, 3, 3, 1), (DEVICE, 1, 0, 0), (DEVICE, 0, 1, 0), (MANAGED, 0, 0, 1), (MANAGED, 1, 0, 1),
    (HOST, 0, 0, 0), (UNREGISTERED, 0, 0, 0), (UNREGISTERED, -2, 0, 0)])
def test_only_own_and_managed_memory_is_read_directly(probe, kind, where, here, direct):
    assert probe.probe_kernel_reaches(kind, where, here) == direct


@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 3), (29, 5), (33, 33), (1, 4000), (4000, 1), (1024, 1024)])
@pytest.mark.parametrize("bounded", [0, 1])
@pytest.mark.parametrize("mixed", [0, 1])
def test_point_buffer_has_room_for_the_state(probe, nx, ny, bounded, mixed):
    need, have = ctypes.c_long(), ctypes.c_long()
    probe.probe_staging(nx, ny, bounded, mixed, ctypes.byref(need), ctypes.byref(have))
    assert need.value <= have.value
