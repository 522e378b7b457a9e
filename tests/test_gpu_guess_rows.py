"""The interpolating kernels around the network at every number of rows per block (1 on small grids
to 16 on large ones) and at grids that end within a block, against the formula in numpy."""
import numpy as np
import pytest
import torch

import paper_2607_01735_gb300 as rb
from paper_2607_01735_gb300.unet import boundary_blend, guess_assemble, guess_target, network_input

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_01735_gb300 import build
    build.build_library()
    rb.load_library()


def _blend(u):
    g = u.shape[0]
    t = np.arange(g) / (g - 1)
    x, y = t[:, None], t[None, :]
    edges = (1 - x) * u[0][None] + x * u[-1][None] + (1 - y) * u[:, :1] + y * u[:, -1:]
    corners = (1 - x) * (1 - y) * u[0, 0] + (1 - x) * y * u[0, -1] + x * (1 - y) * u[-1, 0] + x * y * u[-1, -1]
    return edges - corners


@pytest.mark.parametrize("n", [1, 2, 31, 127, 150, 201, 300, 383, 600, 767, 1100])
def test_blend_input_target_and_assembly(n):
    """Values of order 1: about ten roundings of terms below 8, so 1e-14 in binary64, and one
    binary32 rounding (2^-24 of at most 8) where the output is binary32."""
    rng = np.random.default_rng(n)
    u = rng.uniform(-1, 1, (n + 2, n + 2))
    f, sol = rng.uniform(-1, 1, (n, n)), rng.uniform(-1, 1, (n + 2, n + 2))
    size = (n + 2 + 7) // 8 * 8 + 8
    ud, fd, sd = (torch.from_numpy(a).cuda() for a in (u, f, sol))
    want = _blend(u)
    assert np.abs(boundary_blend(ud).cpu().numpy() - want).max() <= 1e-14
    x = network_input(fd, ud, size).cpu().numpy()
    ring = np.ones((n + 2, n + 2), bool)
    ring[1:-1, 1:-1] = False
    full = np.zeros((size, size, 4))
    full[:n + 2, :n + 2, 1] = ring
    full[:n + 2, :n + 2, 2] = np.where(ring, u, 0)
    full[1:n + 1, 1:n + 1, 0] = f
    full[:n + 2, :n + 2, 3] = want
    assert np.abs(x - full).max() <= 5e-7 and np.array_equal(x[..., 1], full[..., 1])
    t = guess_target(sd, ud, size).cpu().numpy()
    assert np.abs(t[:n + 2, :n + 2] - (sol - want)).max() <= 5e-7
    assert not t[n + 2:].any() and not t[:, n + 2:].any()
    pred = rng.uniform(-1, 1, (size, size)).astype(np.float32)
    u0 = guess_assemble(ud, torch.from_numpy(pred).cuda()).cpu().numpy()
    assert np.array_equal(u0[ring], u[ring])
    assert np.abs(u0 - np.where(ring, u, want + pred[:n + 2, :n + 2])).max() <= 1e-14
