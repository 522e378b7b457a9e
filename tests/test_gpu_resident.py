"""The resident kernel (all sweeps of a small grid in one cooperative launch, tiles in shared
memory, halo values exchanged between neighbouring tiles once per period of several sweeps):
the default of the bit-exact and the fused FP64 sweeps and of the refinement's inner FP32
sweeps on small grids.  Bit for bit the oracle's sequential loops: single tiles, tiles of
uneven sizes, sweep counts below, at and past the period, several calls in a row (the
exchange's period numbers continue), a replayed capture, and the largest grids it takes."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_01735_gb300 as rb
import synth

from test_gpu_parity import _assert_bits, _problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_01735_gb300 import build
    build.build_library()
    rb.load_library()


def _ref(u, f, h2, k, fma):
    (oracle.sweeps_fused if fma else oracle.sweeps)(u, f, h2, k)


@pytest.mark.parametrize("fma", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 3, 13, 23, 24, 37, 64, 97, 100, 127, 255, 256, 401])
def test_resident_sweeps_bit_exact(n, fma):
    f, u0 = _problem(n, 900 + n)
    h2 = synth.h_squared(n)
    ref = u0.copy()
    out = torch.empty((n + 2, n + 2), dtype=torch.float64, device="cuda")
    with rb.Solver(n, h2, torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(), fma=fma) as s:
        for k in (2, 1, 3, 7, 4, 40):
            s.sweep(k)
            _ref(ref, f, h2, k, fma)
            s.get_solution(out)
            _assert_bits(out.cpu().numpy(), ref)


@pytest.mark.parametrize("n,fma", [(1023, 0), (1023, 1), (1190, 0), (1191, 1)])
def test_resident_largest_grids_equal_one_launch_per_colour(n, fma):
    f, u0 = _problem(n, 5)
    h2 = synth.h_squared(n)
    outs = []
    for kernel in (rb.RBGS_KERNEL_AUTO, rb.RBGS_KERNEL_COLOUR):
        out = torch.empty((n + 2, n + 2), dtype=torch.float64, device="cuda")
        with rb.Solver(n, h2, torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(), fma=fma, kernel=kernel) as s:
            s.sweep(23)
            s.get_solution(out)
        outs.append(out.cpu().numpy())
    _assert_bits(outs[0], outs[1])


@pytest.mark.parametrize("n", [5, 31, 70, 255, 511, 700])
def test_resident_inner_sweeps_of_the_refinement(n):
    """Two corrections of 25 FP32 sweeps: the same bits as one launch per colour."""
    f, u0 = _problem(n, 61)
    h2 = synth.h_squared(n)
    outs = []
    for kernel in (rb.RBGS_KERNEL_AUTO, rb.RBGS_KERNEL_COLOUR):
        out = torch.empty((n + 2, n + 2), dtype=torch.float64, device="cuda")
        with rb.Solver(n, h2, torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(), kernel=kernel,
                       precision=rb.RBGS_FP32_REFINE, inner_sweeps=25, max_sweeps=50) as s:
            s.solve(0.0, allow_not_converged=True)
            s.get_solution(out)
        outs.append(out.cpu().numpy())
    _assert_bits(outs[0], outs[1])


def test_resident_sweeps_replay_in_a_captured_graph():
    """A captured rbgs_sweep replays: the exchange's period numbers live on the device."""
    n, k, replays = 127, 9, 5
    f, u0 = _problem(n, 3)
    h2 = synth.h_squared(n)
    st = torch.cuda.Stream()
    out = torch.empty((n + 2, n + 2), dtype=torch.float64, device="cuda")
    with torch.cuda.stream(st):
        with rb.Solver(n, h2, torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(), stream=st.cuda_stream) as s:
            s.sweep(k)
            st.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st):
                s.sweep(k)
            for _ in range(replays):
                g.replay()
            s.get_solution(out)
            st.synchronize()
    ref = u0.copy()
    oracle.sweeps(ref, f, h2, k * (1 + replays))
    _assert_bits(out.cpu().numpy(), ref)
