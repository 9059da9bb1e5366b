"""The serving loop's grid barrier when a block stays away: the waits of the others
run out after their limit, the failure is recorded, and a block that comes late
fails too, however many blocks gave up before it."""
import ctypes as C
import os
import subprocess

import pytest

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.path.join(HERE, "cuda")


@pytest.fixture(scope="module")
def probe():
    from paper_2504_18211_gb300 import build
    os.makedirs(os.path.join(CUDA, "_build"), exist_ok=True)
    lib = os.path.join(CUDA, "_build", "libbarrier_probe.so")
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.INCLUDE,
                    "-I", build.CSRC, os.path.join(CUDA, "ouro_barrier_probe.cu"), "-o", lib], check=True)
    fn = C.CDLL(lib).barrier_probe
    fn.argtypes = [C.c_void_p, C.c_uint, C.c_uint, C.c_uint, C.c_void_p]
    return fn


@pytest.mark.parametrize("waiting", [1, 2, 3, 4, 5, 7, 8, 16, 100])
def test_a_block_that_stays_away(probe, waiting):
    torch = torch_cuda()
    ctl = torch.zeros(11, dtype=torch.int64, device="cuda")
    passed = torch.full((waiting,), -1, dtype=torch.int32, device="cuda")
    assert probe(ctl.data_ptr(), waiting + 1, waiting, 2000, passed.data_ptr()) == 0
    assert passed.tolist() == [0] * waiting and int(ctl[4]) == 1
    late = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    assert probe(ctl.data_ptr(), waiting + 1, 1, 2000, late.data_ptr()) == 0
    assert late.tolist() == [0]


def test_all_blocks_come(probe):
    torch = torch_cuda()
    ctl = torch.zeros(11, dtype=torch.int64, device="cuda")
    passed = torch.full((100,), -1, dtype=torch.int32, device="cuda")
    assert probe(ctl.data_ptr(), 100, 100, 1 << 20, passed.data_ptr()) == 0
    assert passed.tolist() == [1] * 100 and ctl[:5].tolist() == [100, 0, 0, 0, 0]
