// Mixed-precision defect correction: the FP64 update of the refinement loop.
//
// One outer step of the refinement (the loop lives in api.cu):
//   1. rt = h^2 (b - A u) in FP64, max |rt| and (float)rt (residual.cu, exact max);
//   2. e = the binary exponent of max |rt|; r32 = (float)(rt * 2^-e)   (exact scaling,
//      one rounding to binary32): (float)rt * 2^-e, the same bits, where e <= 24 and no nonzero
//      |rt| is below 2^-102, else a second walk;
//   3. d = m FP32 red-black sweeps of (4 I - Adj) d = r32 from d = 0 with a zero ring
//      (the update of Eq. (1) with h^2 f replaced by r32);
//   4. u = u + (double)d * 2^e at interior points   (this file).
// Steps 1 and 4 touch the FP64 iterate; only step 3 runs in FP32.
#include "common.cuh"

namespace rbgs {
namespace {

constexpr int kThreads = 256;
constexpr int kRows = 4;  // rows per block

// A thread takes the pair of elements k, k + 1 of both colour rows: 16-byte loads and stores of u
// and 8-byte loads of d (element by element at the ring columns).
__global__ void __launch_bounds__(kThreads)
correct_kernel(double *__restrict__ red, double *__restrict__ black, const float *__restrict__ d_red,
               const float *__restrict__ d_black, int n, int W, int W32, double scale) {
    const int k = 2 * (blockIdx.x * kThreads + threadIdx.x);
    if (k > (n + 1) / 2) return;
    const bool inner = k > 0 && 2 * k + 3 <= n;  // columns 2k .. 2k + 3 are all interior
    for (int g = blockIdx.y; g * kRows < n; g += gridDim.y) {
        for (int i = 1 + g * kRows; i <= min(n, g * kRows + kRows); ++i) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                double *u = (c ? black : red) + (size_t)i * W + k;
                const float2 d = __ldg(reinterpret_cast<const float2 *>((c ? d_black : d_red) + (size_t)i * W32 + k));
                double2 v = *reinterpret_cast<const double2 *>(u);
                v.x = __dadd_rn(v.x, __dmul_rn((double)d.x, scale));
                v.y = __dadd_rn(v.y, __dmul_rn((double)d.y, scale));
                if (inner) {
                    *reinterpret_cast<double2 *>(u) = v;
                } else {
                    const int j = 2 * k + ((i + c) & 1);  // natural column of element k
                    if (j >= 1 && j <= n) u[0] = v.x;
                    if (j + 2 <= n) u[1] = v.y;
                }
            }
        }
    }
}

__global__ void __launch_bounds__(kThreads) scale_kernel(float4 *__restrict__ red, float4 *__restrict__ black, long count,
                                                         float scale) {
    float4 *__restrict__ r = blockIdx.y ? black : red;
    for (long q = (long)blockIdx.x * kThreads + threadIdx.x; q < count; q += (long)gridDim.x * kThreads) {
        float4 v = r[q];
        v.x *= scale, v.y *= scale, v.z *= scale, v.w *= scale;
        r[q] = v;
    }
}

}  // namespace

// Rows 1..n of the defect arrays times a power of two (their ring places and padding hold zeros).
rbgs_status launch_scale_defect(const rbgs_ctx *c, float scale, cudaStream_t s) {
    const long count = (long)c->g.n * c->f32.W / 4;  // W: a multiple of 64
    const long blocks = (count + kThreads - 1) / kThreads;
    scale_kernel<<<dim3((unsigned)(blocks < 8 * 152 ? blocks : 8 * 152), 2), kThreads, 0, s>>>(
        reinterpret_cast<float4 *>(c->f32.hf[0] + c->f32.W), reinterpret_cast<float4 *>(c->f32.hf[1] + c->f32.W), count,
        scale);
    RBGS_LAUNCH_CHECK();
    return RBGS_OK;
}

rbgs_status launch_correct(const rbgs_ctx *c, double scale, cudaStream_t s) {
    const int n = c->g.n;
    const int pairs = (n + 1) / 4 + 1;  // pairs that hold an element up to (n + 1) / 2
    const int gy = (n + kRows - 1) / kRows;
    dim3 grid((pairs + kThreads - 1) / kThreads, gy < 65535 ? gy : 65535);
    correct_kernel<<<grid, kThreads, 0, s>>>(c->f64.u[0], c->f64.u[1], c->f32.u[0], c->f32.u[1], n, c->g.W,
                                             c->f32.W, scale);
    RBGS_LAUNCH_CHECK();
    return RBGS_OK;
}

}  // namespace rbgs
