"""The kernels at the sizes where the automatic choice takes them up and leaves them (152 SMs;
tests/test_host_dispatch.py checks the choice itself): the fused wavefront passes from 1369^2, the
tiles' largest grids, the refinement's tiles and passes about 1000^2, and the fused graphs of
launches per colour."""
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


def _run(n, f, u0, calls, **opts):
    out = torch.empty((n + 2, n + 2), dtype=torch.float64, device="cuda")
    with rb.Solver(n, synth.h_squared(n), torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(), **opts) as s:
        for k in calls:
            s.sweep(k)
        s.get_solution(out)
    return out.cpu().numpy()


@pytest.mark.parametrize("sweeps", [4, 5, 6, 7, 8, 9])
@pytest.mark.parametrize("n", [1369, 1437, 1439, 1453, 1455, 1500])
def test_fused_wavefront_passes_match_the_oracle(n, sweeps):
    """Every split of a sweep count into passes of 2 and 3 sweeps (first and last pass of either
    depth), at the smallest grid that takes them and at grids that end at and one value past a whole
    number of strips (60 stored values at depth 2, 56 at depth 3)."""
    f, u0 = _problem(n, 31 + n)
    ref = u0.copy()
    oracle.sweeps_fused(ref, f, synth.h_squared(n), sweeps)
    _assert_bits(_run(n, f, u0, [sweeps], fma=1), ref)


def test_fused_wavefront_blocks_of_sweeps():
    """Blocks of 1024 sweeps, a rest of passes and one of fewer sweeps than a pass takes: the bits
    of one launch per colour."""
    n = 1400
    f, u0 = _problem(n, 8)
    calls = [1024 + 7, 3, 2048 + 2]
    _assert_bits(_run(n, f, u0, calls, fma=1), _run(n, f, u0, calls, fma=1, kernel=rb.RBGS_KERNEL_COLOUR))


@pytest.mark.parametrize("sweeps", [4, 6, 9])
@pytest.mark.parametrize("what", ["f", "u", "ring"])
def test_fused_wavefront_reports_non_finite_values(what, sweeps):
    """No valid scale: the last pass, of either depth, writes NaN to every point it updates."""
    n = 1400
    f, u0 = _problem(n, 9)
    if what == "f":
        f[700, 3] = np.inf
    else:
        u0[(5, 9) if what == "u" else (0, 9)] = np.nan
    with rb.Solver(n, synth.h_squared(n), torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(), fma=1) as s:
        s.sweep(sweeps)
        with pytest.raises(rb.RbgsError) as e:
            s.residual()
        out = torch.empty((n + 2, n + 2), dtype=torch.float64, device="cuda")
        s.get_solution(out)
    assert e.value.status == rb.RBGS_ENONFINITE
    assert bool(torch.isnan(out[1:-1, 1:-1]).all())


@pytest.mark.parametrize("fma", [0, 1])
@pytest.mark.parametrize("n", [1192, 1300, 1367, 1368])
def test_fullest_tiles_equal_one_launch_per_colour(n, fma):
    """The largest grids that fit in tiles, where shared memory and the halo's list are all but
    used up, in calls below, at and past a period."""
    f, u0 = _problem(n, 15)
    calls = [2, 3, 20, 1, 7]
    _assert_bits(_run(n, f, u0, calls, fma=fma), _run(n, f, u0, calls, fma=fma, kernel=rb.RBGS_KERNEL_COLOUR))


@pytest.mark.parametrize("n", [900, 999, 1000, 1001, 1002])
def test_refinement_where_tiles_give_way_to_passes(n):
    f, u0 = _problem(n, 62)
    outs = []
    for kernel in (rb.RBGS_KERNEL_AUTO, rb.RBGS_KERNEL_COLOUR):
        out = torch.empty((n + 2, n + 2), dtype=torch.float64, device="cuda")
        with rb.Solver(n, synth.h_squared(n), torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(), kernel=kernel,
                       precision=rb.RBGS_FP32_REFINE, inner_sweeps=27, max_sweeps=54) as s:
            s.solve(0.0, allow_not_converged=True)
            s.get_solution(out)
        outs.append(out.cpu().numpy())
    _assert_bits(outs[0], outs[1])


def test_fused_graphs_of_launches_per_colour():
    """Cached graphs of 32 fused sweeps, replayed across blocks of 1024 with other scales."""
    n = 63
    f, u0 = _problem(n, 4)
    ref = u0.copy()
    calls = [40, 1024 + 33, 32]
    for k in calls:
        oracle.sweeps_fused(ref, f, synth.h_squared(n), min(k, 1024))
        if k > 1024:
            oracle.sweeps_fused(ref, f, synth.h_squared(n), k - 1024)
    _assert_bits(_run(n, f, u0, calls, fma=1, kernel=rb.RBGS_KERNEL_COLOUR), ref)
