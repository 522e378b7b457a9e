// The learned initial guess: a 4-level U-Net trained and run by the library's own
// kernels (conv.cu for the convolutions; pooling, upsampling, concatenation, loss and
// Adam here).  Layer order, shapes and the parameter layout are fixed:
//
//   level 0 (H x W):      e0a 16->32, e0b 32->32                       -> skip0
//   level 1 (H/2 x W/2):  e1a 32->64, e1b 64->64                       -> skip1
//   level 2 (H/4 x W/4):  e2a 64->128, e2b 128->128                    -> skip2
//   level 3 (H/8 x W/8):  b3a 128->256, b3b 256->256
//   level 2: concat(up(b3b), skip2) 384 -> d2a 384->128, d2b 128->128
//   level 1: concat(up(d2b), skip1) 192 -> d1a 192->64, d1b 64->64
//   level 0: concat(up(d1b), skip0)  96 -> d0a 96->32, d0b 32->32
//   out: 1x1 conv 32->8 (channel 0 is the prediction), no activation
// 3x3 convolutions with ReLU; 2x2 average pooling; nearest-neighbour upsampling.
// Parameters (FP32, in this order per layer): weights [Cout][k][k][Cin], then bias[Cout].
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "common.cuh"
#include "../../include/rbgs_unet.h"

namespace rbgs {

rbgs_status conv_forward(const uint16_t *X, const uint16_t *Wt, const float *bias, void *Y, int B, int H,
                         int W, int Cin, int Cout, int ks, int relu, int y_fp32, cudaStream_t s);
rbgs_status umma_conv_check(cudaStream_t s);
rbgs_status conv_backward_layer(const uint16_t *X, const uint16_t *G, float *dX, uint16_t *Gin, float *dW, float *db,
                                const uint16_t *Wtt, int B, int H, int W, int Cin, int Cout, int ks, cudaStream_t s);

namespace {

struct Layer {
    int cin, cout, ks, relu, level;
    long w_off, b_off;  // offsets into the parameter vector
};

constexpr int kInCh = 16;  // f, mask, g, boundary interpolation, zero padding
constexpr int kXCh = 4;    // channels of the caller's input
const int kSpec[15][5] = {
    // cin, cout, ks, relu, level
    {16, 32, 3, 1, 0},   {32, 32, 3, 1, 0},   {32, 64, 3, 1, 1},   {64, 64, 3, 1, 1},
    {64, 128, 3, 1, 2},  {128, 128, 3, 1, 2}, {128, 256, 3, 1, 3}, {256, 256, 3, 1, 3},
    {384, 128, 3, 1, 2}, {128, 128, 3, 1, 2}, {192, 64, 3, 1, 1},  {64, 64, 3, 1, 1},
    {96, 32, 3, 1, 0},   {32, 32, 3, 1, 0},   {32, 8, 1, 0, 0}};

// ------------------------------------------------------------------ elementwise kernels
// All of them move 16-byte vectors (8 bf16 or 4 FP32 channels), one image row per blockIdx.y
// step, with the channel counts of the network as template parameters, so that a vector's place
// costs one division by a constant.  HBM bounds them.  At 16 x 264^2, before (one channel per
// thread, 64-bit divisions) and now: up_concat 900 -> 100 us over the three levels, avgpool 106 ->
// 25, pack_input 100 -> 10.

constexpr int kEw = 256;  // threads per block

__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t bf_pack(float lo, float hi) {
    const __nv_bfloat16 a = __float2bfloat16_rn(lo), b = __float2bfloat16_rn(hi);
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}
// v where the activation y is positive, else 0 (a pair of channels; y as bf16 bits)
__device__ __forceinline__ uint32_t relu_grad2(float lo, float hi, uint32_t y) {
    return bf_pack(bf_lo(y) > 0.f ? lo : 0.f, bf_hi(y) > 0.f ? hi : 0.f);
}

// VEC: x is 16-byte aligned (the caller's pointer need not be)
template <bool VEC>
__global__ void pack_input_kernel(const float *__restrict__ x, uint4 *__restrict__ out, long P) {
    static_assert(kInCh == 16 && kXCh == 4, "one 16-byte load, two 16-byte stores per pixel");
    for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < P; p += (long)gridDim.x * blockDim.x) {
        const float4 v = VEC ? *reinterpret_cast<const float4 *>(x + 4 * p)
                             : make_float4(x[4 * p], x[4 * p + 1], x[4 * p + 2], x[4 * p + 3]);
        out[2 * p] = make_uint4(bf_pack(v.x, v.y), bf_pack(v.z, v.w), 0u, 0u);
        out[2 * p + 1] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// 2x2 average pooling: in [rows][W][C] -> out [rows/2][W/2][C] (rows = B H, H even)
template <int C>
__global__ void __launch_bounds__(kEw) avgpool_kernel(const uint4 *__restrict__ in, uint4 *__restrict__ out,
                                                      long orows, int W) {
    constexpr int C8 = C / 8;
    const int w = W / 2, q = blockIdx.x * kEw + threadIdx.x;
    if (q >= w * C8) return;
    const int x = q / C8, c = q - x * C8;
    for (long r = blockIdx.y; r < orows; r += gridDim.y) {
        const uint4 *p = in + ((2 * r) * W + 2 * x) * C8 + c;
        const uint4 v[4] = {p[0], p[C8], p[(long)W * C8], p[(long)W * C8 + C8]};
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float lo = 0.f, hi = 0.f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t t = e == 0 ? v[k].x : e == 1 ? v[k].y : e == 2 ? v[k].z : v[k].w;
                lo = k ? lo + bf_lo(t) : bf_lo(t);
                hi = k ? hi + bf_hi(t) : bf_hi(t);
            }
            o[e] = bf_pack(0.25f * lo, 0.25f * hi);
        }
        out[(r * w + x) * C8 + c] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// concat(up(lo), skip): out [rows][W][CLO + CS]
template <int CLO, int CS>
__global__ void __launch_bounds__(kEw) up_concat_kernel(const uint4 *__restrict__ lo, const uint4 *__restrict__ skip,
                                                        uint4 *__restrict__ out, long rows, int W) {
    constexpr int L8 = CLO / 8, S8 = CS / 8, T8 = L8 + S8;
    const int q = blockIdx.x * kEw + threadIdx.x;
    if (q >= W * T8) return;
    const int x = q / T8, c = q - x * T8;
    for (long r = blockIdx.y; r < rows; r += gridDim.y)  // H is even: row r / 2 of lo is the same image's
        out[r * W * T8 + q] = c < L8 ? lo[((r >> 1) * (W / 2) + x / 2) * L8 + c] : skip[(r * W + x) * S8 + (c - L8)];
}

// Gradient of a decoder tensor that was upsampled into a concatenation, through its ReLU: the sum
// of dCat[.., :CLO] over each 2x2 block, where y (the tensor itself) is positive, as bf16.
template <int CLO, int CS>
__global__ void __launch_bounds__(kEw) up_grad_kernel(const float4 *__restrict__ dCat, const uint2 *__restrict__ y,
                                                      uint2 *__restrict__ G, long lrows, int W) {
    constexpr int L4 = CLO / 4, T4 = (CLO + CS) / 4;
    const int w = W / 2, q = blockIdx.x * kEw + threadIdx.x;
    if (q >= w * L4) return;
    const int x = q / L4, c = q - x * L4;
    for (long r = blockIdx.y; r < lrows; r += gridDim.y) {
        const float4 *p = dCat + ((2 * r) * W + 2 * x) * T4 + c;
        const float4 a = p[0], b = p[T4], d = p[(long)W * T4], e = p[(long)W * T4 + T4];
        const uint2 m = y[r * w * L4 + q];
        G[r * w * L4 + q] = make_uint2(relu_grad2(a.x + b.x + d.x + e.x, a.y + b.y + d.y + e.y, m.x),
                                       relu_grad2(a.z + b.z + d.z + e.z, a.w + b.w + d.w + e.w, m.y));
    }
}

// Gradient of an encoder tensor that went into a concatenation and into a pooling, through its
// ReLU: dCat[.., CLO:] + dPool / 4, where y (the tensor itself) is positive, as bf16.
template <int CLO, int CS>
__global__ void __launch_bounds__(kEw) skip_grad_kernel(const float4 *__restrict__ dCat,
                                                        const float4 *__restrict__ dPool,
                                                        const uint2 *__restrict__ y, uint2 *__restrict__ G, long rows,
                                                        int W) {
    constexpr int L4 = CLO / 4, S4 = CS / 4, T4 = L4 + S4;
    const int q = blockIdx.x * kEw + threadIdx.x;
    if (q >= W * S4) return;
    const int x = q / S4, c = q - x * S4;
    for (long r = blockIdx.y; r < rows; r += gridDim.y) {
        const float4 a = dCat[(r * W + x) * T4 + L4 + c], d = dPool[((r >> 1) * (W / 2) + x / 2) * S4 + c];
        const uint2 m = y[r * W * S4 + q];
        G[r * W * S4 + q] =
            make_uint2(relu_grad2(__fmaf_rn(0.25f, d.x, a.x), __fmaf_rn(0.25f, d.y, a.y), m.x),
                       relu_grad2(__fmaf_rn(0.25f, d.z, a.z), __fmaf_rn(0.25f, d.w, a.w), m.y));
    }
}

// The transposed weights Wt_t[t][c][o] of every layer's Wt[o][t][c], in one launch (blockIdx.y:
// the layer).
struct TransposeTable {
    long off[15];
    int cin[15], cout[15], taps[15];
};

__global__ void transpose_all_kernel(const uint16_t *__restrict__ wb, uint16_t *__restrict__ wtt,
                                     const TransposeTable t) {
    const int li = blockIdx.y, ci = t.cin[li], co = t.cout[li], taps = t.taps[li];
    const uint16_t *src = wb + t.off[li];
    uint16_t *dst = wtt + t.off[li];
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < ci * co * taps; q += gridDim.x * blockDim.x) {
        const int o = q % co, r = q / co;  // r = tap * cin + c
        dst[q] = src[(long)o * taps * ci + r];
    }
}

__global__ void mask_sum_kernel(const float *__restrict__ mask, float *__restrict__ count, long P) {
    __shared__ float sm[32];
    float acc = 0.f;
    for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < P; p += (long)gridDim.x * blockDim.x)
        acc += mask[p];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        float t = threadIdx.x < blockDim.x / 32 ? sm[threadIdx.x] : 0.f;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) atomicAdd(count, t);
    }
}

// prediction (channel 0 of the 8-channel output) and masked MSE: loss partials, and the output
// layer's gradient as bf16 (the other seven channels are zero)
__global__ void loss_kernel(const float *__restrict__ out8, const float *__restrict__ target,
                            const float *__restrict__ mask, const float *__restrict__ count,
                            uint4 *__restrict__ G8, float *__restrict__ loss, long P) {
    __shared__ float sm[32];
    const float inv_count = *count > 0.f ? 1.f / *count : 0.f;
    float acc = 0.f;
    for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < P; p += (long)gridDim.x * blockDim.x) {
        const float d = out8[p * 8] - target[p];
        const float m = mask[p];
        acc += m * d * d;
        G8[p] = make_uint4(bf_pack(2.f * m * d * inv_count, 0.f), 0u, 0u, 0u);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        float t = threadIdx.x < blockDim.x / 32 ? sm[threadIdx.x] : 0.f;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) atomicAdd(loss, t * inv_count);
    }
}

__global__ void extract_pred_kernel(const float *__restrict__ out8, float *__restrict__ y, long P) {
    for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < P; p += (long)gridDim.x * blockDim.x)
        y[p] = out8[p * 8];
}

__global__ void adam_kernel(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, __nv_bfloat16 *__restrict__ wb, long n, float lr, float b1,
                            float b2, float c1, float c2, float eps) {
    for (long q = (long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x) {
        const float gq = g[q];
        const float mq = b1 * m[q] + (1.f - b1) * gq;
        const float vq = b2 * v[q] + (1.f - b2) * gq * gq;
        m[q] = mq;
        v[q] = vq;
        const float wq = w[q] - lr * (mq * c1) / (sqrtf(vq * c2) + eps);
        w[q] = wq;
        wb[q] = __float2bfloat16_rn(wq);
    }
}

__global__ void to_bf16_kernel(const float *__restrict__ w, __nv_bfloat16 *__restrict__ wb, long n) {
    for (long q = (long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x)
        wb[q] = __float2bfloat16_rn(w[q]);
}

int nblocks(long n) {
    long b = (n + 255) / 256;
    return (int)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

uint64_t splitmix(uint64_t &s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

}  // namespace
}  // namespace rbgs

using namespace rbgs;

struct rbgs_unet {
    cudaStream_t stream;
    std::vector<Layer> layers;
    long nparams;
    float *w, *grad, *m, *v;   // FP32 master weights, gradient, Adam moments
    uint16_t *wb;               // bf16 copy used by the forward and backward
    uint16_t *wtt;              // transposed weights of every layer (at the weights' offsets)
    long step;
    // activation / gradient buffers for one (B, H, W); the gradients' from the first training step on
    int B, H, W;
    std::vector<void *> bufs;
    uint16_t *act[22];          // bf16 activations (see forward for the order)
    float *gr[22];              // FP32 gradients of the concatenations and the pooled tensors
    uint16_t *gbf[2];           // bf16 pre-activation gradients: a layer's and the next one's (NULL: none yet)
    float *scratch;             // FP32 data gradient of the mma.sync engine (NULL: none yet)
    float *out8, *dloss, *hloss;
};

namespace {

// activation tensors: index, channels, level
enum {
    A_IN = 0, A_E0A, A_S0, A_P0, A_E1A, A_S1, A_P1, A_E2A, A_S2, A_P2, A_B3A, A_B3B,
    A_C2, A_D2A, A_D2B, A_C1, A_D1A, A_D1B, A_C0, A_D0A, A_D0B, A_COUNT
};
const int kActCh[A_COUNT] = {16, 32, 32, 32, 64, 64, 64, 128, 128, 128, 256, 256, 384, 128, 128, 192, 64, 64, 96, 32, 32};
const int kActLv[A_COUNT] = {0, 0, 0, 1, 1, 1, 2, 2, 2, 3, 3, 3, 2, 2, 2, 1, 1, 1, 0, 0, 0};

size_t act_elems(const rbgs_unet *net, int a) {
    return (size_t)net->B * (net->H >> kActLv[a]) * (net->W >> kActLv[a]) * kActCh[a];
}

// A buffer for the network's current (B, H, W), freed with the others of that size.
bool alloc_buffer(rbgs_unet *net, size_t bytes, void **p) {
    if (cudaMalloc(p, bytes) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return false;
    }
    net->bufs.push_back(*p);
    return true;
}

void free_buffers(rbgs_unet *net) {
    for (void *p : net->bufs) cudaFree(p);
    net->bufs.clear();
    net->B = net->H = net->W = 0;
    net->gbf[0] = net->gbf[1] = nullptr;
    net->scratch = nullptr;
}

// What a forward pass needs.
rbgs_status ensure_buffers(rbgs_unet *net, int B, int H, int W) {
    if (net->B == B && net->H == H && net->W == W) return RBGS_OK;
    free_buffers(net);
    net->B = B, net->H = H, net->W = W;
    bool ok = alloc_buffer(net, (size_t)B * H * W * 8 * 4, (void **)&net->out8) &&
              alloc_buffer(net, 8, (void **)&net->dloss);
    for (int a = 0; a < A_COUNT && ok; ++a) ok = alloc_buffer(net, act_elems(net, a) * 2, (void **)&net->act[a]);
    if (!ok) {
        free_buffers(net);
        set_error("U-Net buffers: out of device memory");
        return RBGS_ENOMEM;
    }
    return RBGS_OK;
}

// What a backward pass needs besides: FP32 gradients where one kernel forms a sum of several
// (concatenations and poolings), the bf16 ones that a layer hands to the next, as large as the
// largest output of a layer, and with the mma.sync engine that layer's FP32 data gradient.
rbgs_status ensure_gradients(rbgs_unet *net) {
    size_t most = 0;
    bool ok = true;
    const bool first = !net->gbf[1];
    for (int a = 1; a < A_COUNT; ++a) {
        const bool summed = a == A_C0 || a == A_C1 || a == A_C2 || a == A_P0 || a == A_P1 || a == A_P2;
        if (!summed) most = std::max(most, act_elems(net, a));
        if (summed && first && ok) ok = alloc_buffer(net, act_elems(net, a) * 4, (void **)&net->gr[a]);
    }
    for (int q = 0; q < 2 && first && ok; ++q) ok = alloc_buffer(net, most * 2, (void **)&net->gbf[q]);
    if (ok && !net->scratch && rbgs_conv_get_engine() == RBGS_CONV_MMA_SYNC)
        ok = alloc_buffer(net, most * 4, (void **)&net->scratch);
    if (!ok) {
        free_buffers(net);
        set_error("U-Net gradient buffers: out of device memory");
        return RBGS_ENOMEM;
    }
    return RBGS_OK;
}

#define UNET_TRY(x)                              \
    do {                                         \
        rbgs_status st_ = (x);                   \
        if (st_ != RBGS_OK) return st_;          \
    } while (0)

// grid of an elementwise kernel: `per_row` vectors per image row
dim3 ew_grid(int per_row, long rows) {
    return dim3((unsigned)((per_row + kEw - 1) / kEw), (unsigned)(rows < 32768 ? rows : 32768));
}

rbgs_status forward(rbgs_unet *net, const float *x) {
    const int B = net->B, H = net->H, W = net->W;
    cudaStream_t s = net->stream;
    const long P = (long)B * H * W;
    if ((reinterpret_cast<uintptr_t>(x) & 15u) == 0)
        pack_input_kernel<true><<<nblocks(P), 256, 0, s>>>(x, (uint4 *)net->act[A_IN], P);
    else
        pack_input_kernel<false><<<nblocks(P), 256, 0, s>>>(x, (uint4 *)net->act[A_IN], P);
    RBGS_LAUNCH_CHECK();
    auto conv = [&](int li, int in, int out) {
        const Layer &L = net->layers[li];
        return conv_forward(net->act[in], net->wb + L.w_off, net->w + L.b_off, net->act[out], B, H >> L.level,
                            W >> L.level, L.cin, L.cout, L.ks, L.relu, 0, s);
    };
    auto pool = [&](int in, int out) {
        const int lv = kActLv[in], h = H >> lv, w = W >> lv, C = kActCh[in];
        const uint4 *i = (const uint4 *)net->act[in];
        uint4 *o = (uint4 *)net->act[out];
        const dim3 g = ew_grid((w / 2) * (C / 8), (long)B * h / 2);
        if (C == 32) avgpool_kernel<32><<<g, kEw, 0, s>>>(i, o, (long)B * h / 2, w);
        else if (C == 64) avgpool_kernel<64><<<g, kEw, 0, s>>>(i, o, (long)B * h / 2, w);
        else avgpool_kernel<128><<<g, kEw, 0, s>>>(i, o, (long)B * h / 2, w);
        RBGS_LAUNCH_CHECK();
        return RBGS_OK;
    };
    auto upcat = [&](int lo, int skip, int out) {
        const int lv = kActLv[out], h = H >> lv, w = W >> lv;
        const uint4 *l = (const uint4 *)net->act[lo], *k = (const uint4 *)net->act[skip];
        uint4 *o = (uint4 *)net->act[out];
        const dim3 g = ew_grid(w * (kActCh[out] / 8), (long)B * h);
        if (lv == 0) up_concat_kernel<64, 32><<<g, kEw, 0, s>>>(l, k, o, (long)B * h, w);
        else if (lv == 1) up_concat_kernel<128, 64><<<g, kEw, 0, s>>>(l, k, o, (long)B * h, w);
        else up_concat_kernel<256, 128><<<g, kEw, 0, s>>>(l, k, o, (long)B * h, w);
        RBGS_LAUNCH_CHECK();
        return RBGS_OK;
    };
    UNET_TRY(conv(0, A_IN, A_E0A));
    UNET_TRY(conv(1, A_E0A, A_S0));
    UNET_TRY(pool(A_S0, A_P0));
    UNET_TRY(conv(2, A_P0, A_E1A));
    UNET_TRY(conv(3, A_E1A, A_S1));
    UNET_TRY(pool(A_S1, A_P1));
    UNET_TRY(conv(4, A_P1, A_E2A));
    UNET_TRY(conv(5, A_E2A, A_S2));
    UNET_TRY(pool(A_S2, A_P2));
    UNET_TRY(conv(6, A_P2, A_B3A));
    UNET_TRY(conv(7, A_B3A, A_B3B));
    UNET_TRY(upcat(A_B3B, A_S2, A_C2));
    UNET_TRY(conv(8, A_C2, A_D2A));
    UNET_TRY(conv(9, A_D2A, A_D2B));
    UNET_TRY(upcat(A_D2B, A_S1, A_C1));
    UNET_TRY(conv(10, A_C1, A_D1A));
    UNET_TRY(conv(11, A_D1A, A_D1B));
    UNET_TRY(upcat(A_D1B, A_S0, A_C0));
    UNET_TRY(conv(12, A_C0, A_D0A));
    UNET_TRY(conv(13, A_D0A, A_D0B));
    const Layer &L = net->layers[14];
    return conv_forward(net->act[A_D0B], net->wb + L.w_off, net->w + L.b_off, net->out8, B, H, W, L.cin, L.cout,
                        L.ks, 0, 1, s);
}

// Backward from gbf[0], the bf16 gradient of the 8-channel output; fills net->grad.  Along a
// chain of convolutions the data gradient leaves its kernel as the next layer's bf16
// pre-activation gradient (the ReLU's mask from that layer's output); at the concatenations and
// poolings it leaves as FP32 and one kernel forms the sum and the mask.
rbgs_status backward(rbgs_unet *net) {
    const int B = net->B, H = net->H, W = net->W;
    cudaStream_t s = net->stream;
    RBGS_CUDA(cudaMemsetAsync(net->grad, 0, net->nparams * sizeof(float), s));
    TransposeTable tt;
    for (int li = 0; li < 15; ++li) {
        const Layer &L = net->layers[li];
        tt.off[li] = L.w_off, tt.cin[li] = L.cin, tt.cout[li] = L.cout, tt.taps[li] = L.ks * L.ks;
    }
    transpose_all_kernel<<<dim3(64, 15), 256, 0, s>>>(net->wb, net->wtt, tt);
    RBGS_LAUNCH_CHECK();
    int g = 0;  // gbf[g]: the gradient of the layer at hand
    // layer li with input activation `in`: to_g: its data gradient becomes gbf[g ^ 1] (and g
    // moves there), else the FP32 gr[in]
    enum { TO_G, TO_F32, NONE };
    auto conv_bwd = [&](int li, int in, int to) {
        const Layer &L = net->layers[li];
        const rbgs_status st = conv_backward_layer(
            net->act[in], net->gbf[g], to == TO_F32 ? net->gr[in] : to == TO_G ? net->scratch : nullptr,
            to == TO_G ? net->gbf[g ^ 1] : nullptr,
            net->grad + L.w_off, net->grad + L.b_off, net->wtt + L.w_off, B, H >> L.level, W >> L.level, L.cin, L.cout,
            L.ks, s);
        if (to == TO_G) g ^= 1;
        return st;
    };
    // gbf[g] = gradient of act[lo] (level lv + 1), upsampled into the concatenation cat (level lv)
    auto up_bwd = [&](int cat, int lo) {
        const int lv = kActLv[cat], h = H >> lv, w = W >> lv;
        const float4 *d = (const float4 *)net->gr[cat];
        const uint2 *y = (const uint2 *)net->act[lo];
        uint2 *o = (uint2 *)net->gbf[g];
        const dim3 gr = ew_grid((w / 2) * (kActCh[lo] / 4), (long)B * h / 2);
        if (lv == 0) up_grad_kernel<64, 32><<<gr, kEw, 0, s>>>(d, y, o, (long)B * h / 2, w);
        else if (lv == 1) up_grad_kernel<128, 64><<<gr, kEw, 0, s>>>(d, y, o, (long)B * h / 2, w);
        else up_grad_kernel<256, 128><<<gr, kEw, 0, s>>>(d, y, o, (long)B * h / 2, w);
        RBGS_LAUNCH_CHECK();
        return RBGS_OK;
    };
    // gbf[g] = gradient of act[skip], in the concatenation cat and pooled into `pooled`
    auto skip_bwd = [&](int cat, int pooled, int skip) {
        const int lv = kActLv[skip], h = H >> lv, w = W >> lv;
        const float4 *d = (const float4 *)net->gr[cat], *pd = (const float4 *)net->gr[pooled];
        const uint2 *y = (const uint2 *)net->act[skip];
        uint2 *o = (uint2 *)net->gbf[g];
        const dim3 gr = ew_grid(w * (kActCh[skip] / 4), (long)B * h);
        if (lv == 0) skip_grad_kernel<64, 32><<<gr, kEw, 0, s>>>(d, pd, y, o, (long)B * h, w);
        else if (lv == 1) skip_grad_kernel<128, 64><<<gr, kEw, 0, s>>>(d, pd, y, o, (long)B * h, w);
        else skip_grad_kernel<256, 128><<<gr, kEw, 0, s>>>(d, pd, y, o, (long)B * h, w);
        RBGS_LAUNCH_CHECK();
        return RBGS_OK;
    };
    UNET_TRY(conv_bwd(14, A_D0B, TO_G));
    UNET_TRY(conv_bwd(13, A_D0A, TO_G));
    UNET_TRY(conv_bwd(12, A_C0, TO_F32));
    UNET_TRY(up_bwd(A_C0, A_D1B));
    UNET_TRY(conv_bwd(11, A_D1A, TO_G));
    UNET_TRY(conv_bwd(10, A_C1, TO_F32));
    UNET_TRY(up_bwd(A_C1, A_D2B));
    UNET_TRY(conv_bwd(9, A_D2A, TO_G));
    UNET_TRY(conv_bwd(8, A_C2, TO_F32));
    UNET_TRY(up_bwd(A_C2, A_B3B));
    UNET_TRY(conv_bwd(7, A_B3A, TO_G));
    UNET_TRY(conv_bwd(6, A_P2, TO_F32));
    UNET_TRY(skip_bwd(A_C2, A_P2, A_S2));
    UNET_TRY(conv_bwd(5, A_E2A, TO_G));
    UNET_TRY(conv_bwd(4, A_P1, TO_F32));
    UNET_TRY(skip_bwd(A_C1, A_P1, A_S1));
    UNET_TRY(conv_bwd(3, A_E1A, TO_G));
    UNET_TRY(conv_bwd(2, A_P0, TO_F32));
    UNET_TRY(skip_bwd(A_C0, A_P0, A_S0));
    UNET_TRY(conv_bwd(1, A_E0A, TO_G));
    return conv_bwd(0, A_IN, NONE);
}

}  // namespace

extern "C" {

rbgs_status rbgs_unet_create(uint64_t seed, void *cuda_stream, rbgs_unet_t *out) {
    clear_error();
    if (!out) { set_error("out is NULL"); return RBGS_EINVAL; }
    *out = nullptr;
    rbgs_unet *net = new (std::nothrow) rbgs_unet();
    if (!net) { set_error("out of host memory"); return RBGS_ENOMEM; }
    net->stream = (cudaStream_t)cuda_stream;
    long off = 0;
    for (int li = 0; li < 15; ++li) {
        Layer L{kSpec[li][0], kSpec[li][1], kSpec[li][2], kSpec[li][3], kSpec[li][4], 0, 0};
        const long nw = (long)L.cout * L.ks * L.ks * L.cin;
        L.w_off = off;
        off += nw;
        L.b_off = off;
        off += L.cout;
        net->layers.push_back(L);
    }
    net->nparams = off;
    // He-uniform weights (fan-in = k*k*real input channels), zero biases
    std::vector<float> h(off, 0.f);
    uint64_t st = seed;
    for (const Layer &L : net->layers) {
        const int real_in = L.cin == kInCh ? kXCh : L.cin;
        const float a = std::sqrt(6.0f / (float)(L.ks * L.ks * real_in));
        const long nw = (long)L.cout * L.ks * L.ks * L.cin;
        for (long q = 0; q < nw; ++q) {
            const double u = (double)(splitmix(st) >> 11) * (1.0 / 9007199254740992.0);
            h[L.w_off + q] = (float)((2.0 * u - 1.0) * a);
        }
    }
    bool ok = cudaMalloc(&net->w, off * 4) == cudaSuccess && cudaMalloc(&net->grad, off * 4) == cudaSuccess &&
              cudaMalloc(&net->m, off * 4) == cudaSuccess && cudaMalloc(&net->v, off * 4) == cudaSuccess &&
              cudaMalloc(&net->wb, off * 2) == cudaSuccess && cudaMalloc(&net->wtt, off * 2) == cudaSuccess &&
              cudaMallocHost(&net->hloss, 4) == cudaSuccess;
    if (ok) {
        ok = cudaMemcpyAsync(net->w, h.data(), off * 4, cudaMemcpyHostToDevice, net->stream) == cudaSuccess &&
             cudaMemsetAsync(net->m, 0, off * 4, net->stream) == cudaSuccess &&
             cudaMemsetAsync(net->v, 0, off * 4, net->stream) == cudaSuccess;
        to_bf16_kernel<<<nblocks(off), 256, 0, net->stream>>>(net->w, (__nv_bfloat16 *)net->wb, off);
        ok = ok && cudaGetLastError() == cudaSuccess && cudaStreamSynchronize(net->stream) == cudaSuccess;
    }
    if (!ok) {
        cudaGetLastError();
        rbgs_unet_destroy(net);
        set_error("U-Net allocation failed");
        return RBGS_ENOMEM;
    }
    *out = net;
    return RBGS_OK;
}

long rbgs_unet_num_params(rbgs_unet_t net) { return net ? net->nparams : 0; }

rbgs_status rbgs_unet_get_params(rbgs_unet_t net, float *params) {
    clear_error();
    if (!net || !params) { set_error("NULL argument"); return RBGS_EINVAL; }
    RBGS_CUDA(cudaMemcpyAsync(params, net->w, net->nparams * 4, cudaMemcpyDefault, net->stream));
    RBGS_CUDA(cudaStreamSynchronize(net->stream));
    return RBGS_OK;
}

rbgs_status rbgs_unet_set_params(rbgs_unet_t net, const float *params) {
    clear_error();
    if (!net || !params) { set_error("NULL argument"); return RBGS_EINVAL; }
    RBGS_CUDA(cudaMemcpyAsync(net->w, params, net->nparams * 4, cudaMemcpyDefault, net->stream));
    to_bf16_kernel<<<nblocks(net->nparams), 256, 0, net->stream>>>(net->w, (__nv_bfloat16 *)net->wb, net->nparams);
    RBGS_LAUNCH_CHECK();
    RBGS_CUDA(cudaMemsetAsync(net->m, 0, net->nparams * 4, net->stream));
    RBGS_CUDA(cudaMemsetAsync(net->v, 0, net->nparams * 4, net->stream));
    net->step = 0;
    RBGS_CUDA(cudaStreamSynchronize(net->stream));
    return RBGS_OK;
}

rbgs_status rbgs_unet_forward(rbgs_unet_t net, const float *x, float *y, int B, int H, int W) {
    clear_error();
    if (!net || !x || !y || B < 1 || H < 8 || W < 8 || H % 8 || W % 8) {
        set_error("rbgs_unet_forward: bad arguments (H, W multiples of 8)");
        return RBGS_EINVAL;
    }
    UNET_TRY(ensure_buffers(net, B, H, W));
    UNET_TRY(forward(net, x));
    const long P = (long)B * H * W;
    extract_pred_kernel<<<nblocks(P), 256, 0, net->stream>>>(net->out8, y, P);
    RBGS_LAUNCH_CHECK();
    return RBGS_OK;
}

rbgs_status rbgs_unet_train_step(rbgs_unet_t net, const float *x, const float *target, const float *mask_loss,
                                 int B, int H, int W, float lr, float *loss, float *grads) {
    clear_error();
    if (!net || !x || !target || !mask_loss || B < 1 || H < 8 || W < 8 || H % 8 || W % 8) {
        set_error("rbgs_unet_train_step: bad arguments");
        return RBGS_EINVAL;
    }
    UNET_TRY(ensure_buffers(net, B, H, W));
    UNET_TRY(ensure_gradients(net));
    UNET_TRY(forward(net, x));
    const long P = (long)B * H * W;
    RBGS_CUDA(cudaMemsetAsync(net->dloss, 0, 8, net->stream));  // [0] loss, [1] sum(mask)
    mask_sum_kernel<<<nblocks(P), 256, 0, net->stream>>>(mask_loss, net->dloss + 1, P);
    RBGS_LAUNCH_CHECK();
    loss_kernel<<<nblocks(P), 256, 0, net->stream>>>(net->out8, target, mask_loss, net->dloss + 1,
                                                    (uint4 *)net->gbf[0], net->dloss, P);
    RBGS_LAUNCH_CHECK();
    UNET_TRY(backward(net));
    if (grads) {
        RBGS_CUDA(cudaMemcpyAsync(grads, net->grad, net->nparams * 4, cudaMemcpyDefault, net->stream));
    } else {
        net->step += 1;
        const float b1 = 0.9f, b2 = 0.999f;
        const float c1 = 1.f / (1.f - std::pow(b1, (float)net->step));
        const float c2 = 1.f / (1.f - std::pow(b2, (float)net->step));
        adam_kernel<<<nblocks(net->nparams), 256, 0, net->stream>>>(net->w, net->grad, net->m, net->v,
                                                                    (__nv_bfloat16 *)net->wb, net->nparams, lr, b1,
                                                                    b2, c1, c2, 1e-8f);
        RBGS_LAUNCH_CHECK();
    }
    RBGS_CUDA(cudaMemcpyAsync(net->hloss, net->dloss, 4, cudaMemcpyDeviceToHost, net->stream));
    RBGS_CUDA(cudaStreamSynchronize(net->stream));
    if (loss) *loss = *net->hloss;
    return umma_conv_check(net->stream);
}

void rbgs_unet_destroy(rbgs_unet_t net) {
    if (!net) return;
    cudaStreamSynchronize(net->stream);
    for (void *p : net->bufs) cudaFree(p);
    cudaFree(net->w);
    cudaFree(net->grad);
    cudaFree(net->m);
    cudaFree(net->v);
    cudaFree(net->wb);
    cudaFree(net->wtt);
    if (net->hloss) cudaFreeHost(net->hloss);
    delete net;
}

}  // extern "C"
