"""The convolution kernels' index arithmetic (csrc/conv_index.cuh), compiled for the host,
against Python's integers: offsets in rows of more than 2^31 elements, which every accepted
width reaches with enough channels.  CPU only."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "native", "conv_index_host_check.cpp")
HDR = os.path.join(os.path.dirname(HERE), "paper_2607_01735_gb300", "csrc", "conv_index.cuh")
OUT = os.path.join(HERE, "native", "_build", "libconvindexcheck.so")


def _cuda_include():
    for d in (os.environ.get("CUDA_HOME", ""), "/usr/local/cuda"):
        if d and os.path.exists(os.path.join(d, "include", "cuda_runtime.h")):
            return os.path.join(d, "include")
    pytest.skip("CUDA headers not found")


@pytest.fixture(scope="module")
def lib():
    os.makedirs(os.path.dirname(OUT), exist_ok=True)
    if not os.path.exists(OUT) or os.path.getmtime(OUT) < max(os.path.getmtime(p) for p in (SRC, HDR)):
        tmp = OUT + f".tmp{os.getpid()}"
        subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", _cuda_include(), SRC, "-o", tmp])
        os.replace(tmp, OUT)
    l = ctypes.CDLL(OUT)
    l.check_tap_offset.argtypes = [ctypes.c_int] * 5
    l.check_tap_offset.restype = ctypes.c_long
    l.check_offsets_fit_int.argtypes = [ctypes.c_int] * 2
    return l


@pytest.mark.parametrize("W,C", [(1, 8), (264, 96), (32767, 2048), (32767, 65528), (32767, 65536), (32767, 65544), (32767, 1 << 20),
                                 (161, 1 << 24), (2, (1 << 31) - 8)])
def test_tap_offsets_of_rows_beyond_32_bits(lib, W, C):
    """Every tap of a 3x3 layer, forward and mirrored, at W = 32767 with 65536 channels (2^31
    elements a row, the first size whose element offset leaves 32 bits) and beyond."""
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            for ch in (0, 8, C - 8):
                assert lib.check_tap_offset(dy, dx, W, C, ch) == (dy * W + dx) * C + ch


@pytest.mark.parametrize("seg", [16, 144, 160])
def test_offsets_of_a_staged_row_fit_an_int(lib, seg):
    """seg + 2 pixels of C channels, at the largest C that fits and the next one accepted."""
    most = (2 ** 31 - 1) // (seg + 2) // 8 * 8
    assert lib.check_offsets_fit_int(seg, most) and not lib.check_offsets_fit_int(seg, most + 8)


def test_tap_row_weight_gradient_leaves_rows_that_its_offsets_do_not_hold():
    """The tap-row kernel keeps its copies' offsets within a segment of a row in 32 bits: from
    2^31 / 18 channels no segment fits, and the gather kernel, whose offsets are 64-bit, runs."""
    from paper_2607_01735_gb300 import build, unet as un
    build.build_library()
    un.rbgs_conv_set_wgrad_kernel(un.RBGS_WGRAD_TAPROW)
    try:
        assert un.rbgs_conv_wgrad_kernel_for(1, 1, 161, 1 << 23, 8) == un.RBGS_WGRAD_TAPROW
        assert un.rbgs_conv_wgrad_kernel_for(1, 1, 161, 1 << 27, 8) == un.RBGS_WGRAD_GATHER
        assert un.rbgs_conv_wgrad_kernel_for(1, 1, 161, 8, 12) == -1
    finally:
        un.rbgs_conv_set_wgrad_kernel(un.RBGS_WGRAD_AUTO)
