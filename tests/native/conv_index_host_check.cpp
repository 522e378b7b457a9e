// Host build of the convolution kernels' index arithmetic (csrc/conv_index.cuh).
// Test infrastructure only.
#include "../../paper_2607_01735_gb300/csrc/conv_index.cuh"

// The offset as the forward product forms it.
extern "C" long check_tap_offset(int dy, int dx, int W, int C, int ch) {
    return rbgs::offsets_fit_int(W, C) ? rbgs::tap_offset<int>(dy, dx, W, C, ch)
                                       : rbgs::tap_offset<long>(dy, dx, W, C, ch);
}

extern "C" int check_offsets_fit_int(int W, int C) { return rbgs::offsets_fit_int(W, C); }
