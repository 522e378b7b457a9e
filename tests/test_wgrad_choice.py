"""The automatic choice of the weight-gradient kernel (host code over a stand-in runtime of 152
SMs) against measured times.  CPU only."""
import pytest

import fake_runtime

RING, TAPROW, GATHER = 1, 2, 3

# us on GB300 of the gather and the tap-row kernel for W^2 images, batch B, Cin -> Cout
MEASURED = {
    (66, 64, 128): {2: (16.5, 18.6), 4: (18.5, 21.8), 8: (29.6, 29.7), 10: (31.9, 32.4), 12: (35.4, 32.0),
                    14: (39.1, 40.2), 16: (47.2, 43.7)},
    (66, 128, 128): {2: (18.4, 28.4), 4: (26.1, 32.4), 8: (41.0, 46.7), 10: (49.5, 48.7), 12: (56.9, 48.1),
                     14: (64.5, 63.3), 16: (72.1, 69.3)},
    (66, 384, 128): {2: (36.5, 36.9), 4: (69.7, 44.6), 5: (84.1, 59.0), 8: (128.2, 77.4), 10: (160.0, 85.5),
                     12: (184.4, 94.1), 14: (216.3, 104.0), 16: (248.4, 112.3)},
    (132, 64, 64): {4: (35.6, 26.9), 5: (36.6, 30.6), 8: (61.9, 43.0), 10: (75.4, 54.7), 12: (88.3, 54.7),
                    14: (101.9, 60.9), 16: (115.0, 73.7)},
    (132, 192, 64): {4: (91.7, 53.3), 8: (186.1, 89.0), 16: (363.3, 168.1)},
    (264, 96, 32): {2: (75.8, 42.5), 4: (165.8, 63.6), 8: (322.9, 116.9), 16: (638.4, 215.1)},
    (33, 128, 256): {2: (15.0, 26.7), 8: (26.5, 40.4), 16: (38.7, 56.9)},
    (33, 256, 256): {2: (20.5, 27.9), 8: (39.7, 56.3), 16: (63.4, 67.0)},
}


@pytest.fixture(scope="module")
def lib():
    return fake_runtime.load()


@pytest.mark.parametrize("layer", MEASURED)
def test_choice_is_within_5_percent_of_the_faster_kernel(lib, layer):
    W, Cin, Cout = layer
    for B, (gather, taprow) in MEASURED[layer].items():
        chosen = lib.rbgs_conv_wgrad_kernel_for(B, W, W, Cin, Cout, 3)
        assert chosen in (TAPROW, GATHER)
        t = taprow if chosen == TAPROW else gather
        assert t <= 1.05 * min(gather, taprow), (layer, B, chosen)


def test_narrow_layers_take_the_ring_and_other_sizes_of_tap_the_gather_kernel(lib):
    for W, Cin, Cout in ((264, 16, 32), (264, 32, 32), (132, 32, 64)):
        assert lib.rbgs_conv_wgrad_kernel_for(16, W, W, Cin, Cout, 3) == RING
    assert lib.rbgs_conv_wgrad_kernel_for(16, 264, 264, 32, 8, 1) == GATHER
