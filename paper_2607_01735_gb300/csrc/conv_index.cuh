// Element offsets inside NHWC tensors, shared by the convolution kernels and the host test of
// their arithmetic.  An image row may hold more than 2^31 elements (up to 32767 pixels of any
// number of channels).
#pragma once

#include <cuda_runtime.h>

namespace rbgs {

// Elements from a pixel to channel `ch` of the pixel dy rows and dx columns further on (|dy|,
// |dx| <= 1, rows of W <= 32767 pixels, C channels), in a type that holds it: int where
// offsets_fit_int says so, else long.  (Always in 64 bits, the gather kernel's copies needed two
// instructions more each: a guess at 1023^2 took 1175 us instead of 1170.)
template <typename Offset>
__host__ __device__ __forceinline__ Offset tap_offset(int dy, int dx, int W, int C, int ch) {
    return (Offset)(dy * W + dx) * C + ch;
}

// Offsets within W + 2 neighbouring pixels of C channels fit an int.
inline bool offsets_fit_int(int W, int C) { return ((long)W + 2) * C <= 0x7fffffffL; }

}  // namespace rbgs
