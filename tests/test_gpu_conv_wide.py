"""A 3x3 layer whose image rows hold 2^31 elements: the forward product's offsets between rows
leave 32 bits (csrc/conv_index.cuh)."""
import pytest
import torch

import paper_2607_01735_gb300 as rb
from paper_2607_01735_gb300 import unet as un

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_01735_gb300 import build
    build.build_library()
    rb.load_library()


def test_forward_of_rows_beyond_32_bits():
    """Two rows of 32767 pixels of 65536 channels (8.6 GB), 8 outputs of about unit size, at
    pixels of both rows (each reads the row above or below) against 64-bit sums.  The 9 x 65536
    products are added in FP32 16 at a time: 36864 additions that may each be off by 2^-23 of a
    partial sum of at most about 4, so 0.018 in all."""
    W, C, N = 32767, 65536, 8
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.empty((1, 2, W, C), dtype=torch.bfloat16, device="cuda").normal_(generator=g)
    w = (torch.randn((N, 3, 3, C), device="cuda", generator=g) / (9 * C) ** 0.5).bfloat16()
    y = torch.full((1, 2, W, N), 7.0, device="cuda")
    un.rbgs_conv_forward(x, w, None, y, relu=False)
    un.rbgs_conv_check()
    wd = w.double()
    for r in (0, 1):
        for c in (0, 1, 127, 128, 16000, W - 2, W - 1):
            ref = torch.zeros(N, dtype=torch.float64, device="cuda")
            for ty in range(3):
                for tx in range(3):
                    yy, xx = r + ty - 1, c + tx - 1
                    if 0 <= yy < 2 and 0 <= xx < W:
                        ref += wd[:, ty, tx] @ x[0, yy, xx].double()
            assert float((y[0, r, c].double() - ref).abs().max()) <= 0.018, (r, c)
    del x
    torch.cuda.empty_cache()
