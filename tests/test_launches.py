"""What the library's launchers ask of the CUDA runtime, shown on the CPU with
a stand-in for its launch calls.

Kernel attributes (dynamic shared-memory limit, shared-memory split) belong to
one device.  The FP64 node update needs more than the default limit, so a
process that steps meshes on a second device has to set them there too (also
run on two GPUs where there are two)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture
def native(tmp_path):
    """Builds tests/native/<name>.cpp against the library and runs it: its output."""
    def run(name):
        from paper_2509_01827_gb300 import build
        lib = build.build()
        exe = str(tmp_path / name)
        subprocess.run(["g++", "-std=c++17", "-O1", "-rdynamic", os.path.join(ROOT, "tests", "native", name + ".cpp"),
                        "-I", os.path.join(ROOT, "paper_2509_01827_gb300", "csrc"),
                        "-I", os.path.join(CUDA, "include"), "-o", exe, lib,
                        "-L", os.path.join(CUDA, "lib64"), "-lcudart", "-Wl,-rpath," + os.path.dirname(lib),
                        "-Wl,-rpath," + os.path.join(CUDA, "lib64")], check=True)
        r = subprocess.run([exe], capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr
        return r.stdout
    if shutil.which("g++") is None:
        pytest.skip("needs a host compiler")
    return run


def test_attributes_on_each_device(native):
    native("device_attributes")


def test_batch_grids_fill_the_gpu(native):
    """Kernels that take the work items of all members one block each: with more
    items than fit at once, at least one full load of threads (the piece forces' blocks of
    64 threads as many more blocks)."""
    launches = [tuple(int(v) for v in line.split()) for line in native("batch_grids").splitlines()]
    pieces = [(block, grid) for block, grid in launches if block == 64]
    assert len(pieces) == 1
    assert pieces[0][0] * pieces[0][1] >= 152 * 2048
    for block, grid in launches:
        if block in (128, 256) and grid > 64:  # evaluation, phantom and node updates
            assert grid >= 1216


@pytest.mark.parametrize("side,blocks", [(1024, 1216), (1440, 1216), (2048, 304)])
def test_piece_blocks_and_evaluation_split(native, monkeypatch, side, blocks):
    """Plates with hundreds of thousands of split elements: the piece forces have as
    many blocks as the SMs hold (meshes whose node update sets the step: two an SM),
    and the evaluation beside them leaves the SMs their L1."""
    monkeypatch.setenv("MESH_SIDE", str(side))
    lines = native("step_grids").splitlines()
    assert lines[0] == "0" or side == 2048
    launches = [tuple(int(v) for v in line.split()) for line in lines[1:]]
    assert max(grid for block, grid in launches if block == 256 and grid > 1) == blocks


@pytest.mark.gpu
def test_two_devices_in_one_process():
    import torch
    if torch.cuda.device_count() < 2:
        pytest.skip("one GPU visible")
    from paper_2509_01827_gb300 import build, inputs
    from paper_2509_01827_gb300.cem import Batch, Solver
    build.build()
    p = inputs.notched_plate(400, 160, traction=2.5e6, phantom_cap=40000, crack_cap=16000)
    got = []
    for dev in (0, 1):
        s, m = Solver(p, device=dev), Solver(p, device=dev)
        s.step(20)
        b = Batch([m])
        b.step(20)
        got += [s.nodes()["uy"], m.nodes()["uy"]]
        b.close()
    for g in got[1:]:
        np.testing.assert_array_equal(g, got[0])
