"""The tile exchange of the resident kernel (csrc/tile_exchange.cuh): a block whose neighbour's
values never arrive gives up after its poll limit, reports it and leaves as a whole; with every
value there it receives them all, also over an earlier period's values in the slots."""
import ctypes
import os
import shutil
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = os.path.join(HERE, "native", "_build", "libexchangecheck.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17",
                           "-Xcompiler", "-fPIC", "-shared", os.path.join(HERE, "native", "exchange_check.cu"),
                           "-o", out])
    l = ctypes.CDLL(out)
    l.run_receive_check.argtypes = [ctypes.c_int] * 3 + [ctypes.c_uint] * 2 + [ctypes.POINTER(ctypes.c_int)]
    l.run_entry_check.argtypes = [ctypes.c_int] * 2 + [ctypes.POINTER(ctypes.c_int)]
    return l


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("count", [1, 64, 255, 256, 257, 600])
def test_block_leaves_when_a_value_never_arrives(lib, bits, count):
    out = (ctypes.c_int * 3)()
    assert lib.run_receive_check(bits, count, 1, 7, 1000, out) == 0
    assert list(out) == [2, 64, 0]  # status bit 1, all 64 threads, nothing compared
    assert lib.run_receive_check(bits, count, 0, 7, 1 << 20, out) == 0
    assert list(out) == [0, 0, 0]
    # period numbers past 2^31 and at the wrap
    for seq in (1 << 31, 0xffffffff, 0, 1):
        assert lib.run_receive_check(bits, count, 0, seq, 1 << 20, out) == 0
        assert list(out) == [0, 0, 0]


@pytest.mark.parametrize("status,left", [(0, 0), (2, 512)])
def test_whole_block_agrees_on_the_status(lib, status, left):
    out = ctypes.c_int(-1)
    assert lib.run_entry_check(status, 512, ctypes.byref(out)) == 0
    assert out.value == left
