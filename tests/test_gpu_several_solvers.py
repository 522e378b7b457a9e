"""Several small solvers at once, each on a stream of its own: the same bits as alone, and their
work overlaps (include/rbgs.h: separate contexts may be used from separate threads)."""
import threading
import time

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


def _solvers(n, count, **opts):
    out = []
    for q in range(count):
        f, u0 = _problem(n, 40 + q)
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            s = rb.Solver(n, synth.h_squared(n), torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(),
                          stream=st.cuda_stream, **opts)
        out.append((s, f, u0, st))
    torch.cuda.synchronize()
    return out


def _solution(s, n, st):
    out = torch.empty((n + 2, n + 2), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    s.get_solution(out)
    st.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("fma", [0, 1])
@pytest.mark.parametrize("n,count", [(31, 16), (127, 2), (127, 8), (255, 5), (511, 3), (1023, 2), (1400, 4)])
def test_several_contexts_match_the_oracle(n, count, fma):
    """Bursts of calls on every stream, then single ones: each context's launches change between
    whole and shared plans of the device, and its period numbers continue across them."""
    ks = (30, 7, 2, 25) if n < 500 else (9, 2, 5)
    solvers = _solvers(n, count, fma=fma)
    for k in ks:
        for s, *_ in solvers:
            s.sweep(k)
    torch.cuda.synchronize()
    solvers[0][0].sweep(11)
    for q, (s, f, u0, st) in enumerate(solvers):
        ref = u0.copy()
        for k in ks + ((11,) if q == 0 else ()):  # a fused call chooses its own scale
            (oracle.sweeps_fused if fma else oracle.sweeps)(ref, f, synth.h_squared(n), k)
        _assert_bits(_solution(s, n, st), ref)
        s.close()


@pytest.mark.parametrize("n,count", [(255, 6), (720, 8), (999, 6), (1100, 8)])
def test_several_threads_refine_with_the_bits_of_one(n, count):
    """Tiles of a part of the device, and wavefront passes of a part from about 700^2 on."""
    opts = dict(precision=rb.RBGS_FP32_REFINE, inner_sweeps=25, max_sweeps=100)
    alone = []
    for s, _, _, st in _solvers(n, count, **opts):
        s.solve(0.0, allow_not_converged=True)
        alone.append(_solution(s, n, st))
        s.close()
    solvers = _solvers(n, count, **opts)
    threads = [threading.Thread(target=s.solve, args=(0.0, True)) for s, *_ in solvers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for (s, _, _, st), ref in zip(solvers, alone):
        _assert_bits(_solution(s, n, st), ref)
        s.close()


def test_small_solvers_overlap():
    """Eight 127^2 contexts on eight streams take less than 0.6 of eight calls one after another
    (0.2 when small grids ran as launches of a few blocks, 0.9 when each call took the whole GPU)."""
    solvers = _solvers(127, 8)

    def burst():
        torch.cuda.synchronize()
        t = time.perf_counter()
        for s, *_ in solvers:
            s.sweep(400)
        torch.cuda.synchronize()
        return time.perf_counter() - t

    def in_turn():
        torch.cuda.synchronize()
        t = time.perf_counter()
        for s, *_ in solvers:
            s.sweep(400)
            torch.cuda.synchronize()
        return time.perf_counter() - t

    for _ in range(3):
        burst(), in_turn()
    assert min(burst() for _ in range(7)) <= 0.6 * min(in_turn() for _ in range(7))
    for s, *_ in solvers:
        s.close()
