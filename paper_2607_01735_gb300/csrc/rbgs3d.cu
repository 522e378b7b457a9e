// The 3D variant of the red-black scheme (the paper's outlook, Section 5): the 7-point
// update u = (h2 f + N + S + W + E + D + U) / 6 over one colour at a time, i + j + k even
// (red) then odd (black).  C ABI in include/rbgs3d.h.
//
// Layout: the 2D colour split applied along k.  For every grid line (i, j), 0 <= i, j <=
// N+1, colour c holds a row of W values; element m is the point k = 2m + ((i + j + c) & 1).
// A point and its four neighbours in i and j share m (those lines have the other parity);
// its k-neighbours sit in the other colour's row of the same line, at m-1/m or m/m+1.
// W = ceil((N+2)/2) rounded up to 32 values (256-byte rows).
//
// Half-sweep: the pairs of values of a plane (line j, pair of elements) are flattened over the
// threads, and a thread walks its place (j, m) down a chunk of planes i.  The other colour's
// values at planes i-1, i, i+1 stay in registers, so each is loaded once per chunk; lines j-1
// and j+1 of plane i are other threads' places and come through L1.  (One flattened loop over
// all (i, j, m) with five line loads and two index divisions per pair, and a division by 6 of
// three FP64 operations, ran at 31 GLUP/s at 511^3, 2.12 ms a half-sweep.)  Arithmetic: six
// adds in the order above, each one correctly rounded fused multiply-add by a run-time 1.0, and
// one correctly rounded division by 6 on the integer pipes (div6.cuh): the same bits as the
// plain sequential loop.  The FP64 pipe bounds it, six instructions
// per update, 83% busy (ncu): 85.9 GLUP/s at 511^3, 0.78 ms a half-sweep, 79 at 255^3 (27 before).
#include <algorithm>
#include <cmath>
#include <new>
#include <type_traits>

#include "../../include/rbgs3d.h"
#include "common.cuh"
#include "div6.cuh"
#include "fp64.cuh"
#include "sweep_impl.cuh"

struct rbgs3d_ctx {
    int n, W;
    double h2;
    cudaStream_t stream;
    double *u[2], *hf[2];
    double *staging;   // natural-layout (N+2)^3 buffer for host inputs and outputs
    double *partials;  // [2 * kBlocks3]: per block sums, both colours
    double *dsum;      // [2]
    double *hsum;      // pinned mirror of dsum
    double den2;
};

namespace rbgs {
namespace {

constexpr int kThreads3 = 256;
constexpr int kBlocks3 = 4096;  // grid-stride blocks of the reductions (<= partial slots)
constexpr int kMaxN3 = 2048;

__host__ __device__ inline int width3(int n) {
    const int w = (n + 3) / 2;
    return (w + 31) / 32 * 32;
}

// natural (N+2)^3 u -> colour rows; f (N^3) -> h2 f colour rows, zero off the interior.
__global__ void pack3_kernel(const double *__restrict__ u_nat, const double *__restrict__ f_nat, double h2,
                             double *__restrict__ u0, double *__restrict__ u1, double *__restrict__ hf0,
                             double *__restrict__ hf1, int n, int W) {
    const int L = n + 2;
    const size_t total = (size_t)L * L * W;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (size_t)gridDim.x * blockDim.x) {
        const int m = (int)(q % W);
        const size_t line = q / W;
        const int i = (int)(line / L), j = (int)(line % L);
        const int k = 2 * m;
        // colour of (i, j, k) is (i + j) & 1; (i, j, k + 1) the other one
        const double a = k <= n + 1 ? u_nat[line * L + k] : 0.0;
        const double b = k + 1 <= n + 1 ? u_nat[line * L + k + 1] : 0.0;
        const bool in_line = i >= 1 && i <= n && j >= 1 && j <= n;
        const size_t fl = ((size_t)(i - 1) * n + (j - 1)) * n;
        const double fa = (in_line && k >= 1 && k <= n) ? __dmul_rn(h2, f_nat[fl + k - 1]) : 0.0;
        const double fb = (in_line && k + 1 <= n) ? __dmul_rn(h2, f_nat[fl + k]) : 0.0;
        const bool even = ((i + j) & 1) == 0;
        (even ? u0 : u1)[q] = a;
        (even ? u1 : u0)[q] = b;
        (even ? hf0 : hf1)[q] = fa;
        (even ? hf1 : hf0)[q] = fb;
    }
}

__global__ void unpack3_kernel(const double *__restrict__ u0, const double *__restrict__ u1,
                               double *__restrict__ u_nat, int n, int W) {
    const int L = n + 2;
    const size_t total = (size_t)L * L * W;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (size_t)gridDim.x * blockDim.x) {
        const int m = (int)(q % W);
        const size_t line = q / W;
        const int i = (int)(line / L), j = (int)(line % L);
        const int k = 2 * m;
        const bool even = ((i + j) & 1) == 0;
        if (k <= n + 1) u_nat[line * L + k] = (even ? u0 : u1)[q];
        if (k + 1 <= n + 1) u_nat[line * L + k + 1] = (even ? u1 : u0)[q];
    }
}

// A thread's place in every plane: line j and the pair of elements m0, m0 + 1.
struct Place3 {
    int j, m0;
    bool act;
};

// Pairs per line and the multiplier ceil(2^32 / npairs) of the division by it: item / npairs =
// umulhi(item, mul) exactly, as item (mul npairs - 2^32) < 2^22 2^10 (n <= 2048).  An integer
// division costs FP64-pipe instructions, which a short chunk would notice.
struct Pairs3 {
    int npairs;
    unsigned mul;
};

__device__ __forceinline__ Place3 place3(int block, int n, const Pairs3 &d) {
    const int item = block * kThreads3 + (int)threadIdx.x;
    const int npairs = d.npairs;
    const int line = npairs == 1 ? item : (int)__umulhi((unsigned)item, d.mul);
    return Place3{1 + line, 2 * (item - line * npairs), line < n};
}

// One half-sweep of colour C over planes [i0, i0 + chunk) by block (x: places, y: chunk).
template <int C>
__global__ void __launch_bounds__(kThreads3)
half_sweep3_kernel(double *__restrict__ self, const double *__restrict__ other, const double *__restrict__ hf,
                   int n, int W, Pairs3 npairs, int chunk, double one) {
    constexpr int NV = 2;  // 4 and 8 values measured 1.5% and 10% slower
    const Place3 pl = place3(blockIdx.x, n, npairs);
    if (!pl.act) return;
    const int m0 = pl.m0;
    const int i0 = 1 + blockIdx.y * chunk, i1 = min(n, i0 + chunk - 1);
    const size_t plane = (size_t)(n + 2) * W;
    size_t at = ((size_t)i0 * (n + 2) + pl.j) * W + m0;
    double vn[NV], vm[NV], vs[NV], vw[NV], ve[NV], f[NV];
    load_row<NV>(vn, other + at - plane, true);
    load_row<NV>(vm, other + at, true);
    for (int i = i0; i <= i1; ++i, at += plane) {
        load_row<NV>(vs, other + at + plane, true);
        load_row<NV>(vw, other + at - W, true);
        load_row<NV>(ve, other + at + W, true);
        load_row<NV>(f, hf + at, true);
        // value v at k = 2(m0+v) + p: k-1 and k+1 at elements m0+v-1+p and m0+v+p
        const int p = (i + pl.j + C) & 1;
        const bool in = p ? m0 + NV < W : m0 > 0;
        const double x = in ? __ldg(other + at + (p ? NV : -1)) : 0.0;
        double r[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            r[v] = add_fma(add_fma(add_fma(add_fma(f[v], vn[v], one), vs[v], one), vw[v], one), ve[v], one);
            r[v] = add_fma(r[v], p ? vm[v] : (v ? vm[v ? v - 1 : 0] : x), one);
            r[v] = add_fma(r[v], p ? (v + 1 < NV ? vm[v + 1 < NV ? v + 1 : 0] : x) : vm[v], one);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) r[v] = div6(r[v]);
        const int k0 = 2 * m0 + p;  // natural k of value 0; value v at k0 + 2v
        if (k0 >= 1 && k0 + 2 * (NV - 1) <= n) {
            store_row<NV>(self + at, r);
        } else {
#pragma unroll
            for (int v = 0; v < NV; ++v)
                if (k0 + 2 * v >= 1 && k0 + 2 * v <= n) self[at + v] = r[v];
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) vn[v] = vm[v], vm[v] = vs[v];
    }
}

// Both colours' arrays of a reduction.
struct Fields3 {
    const double *u[2], *hf[2];
};

// The colour that a block of a reduction walks, its number among the colour's blocks and how many
// these are.  C 0, 1: all blocks; kBoth: the first half of the blocks red, the others black.
constexpr int kBoth = 2;
struct Share3 {
    int colour, block, blocks;
};
template <int C>
__device__ __forceinline__ Share3 share3() {
    if (C != kBoth) return Share3{C, (int)blockIdx.x, (int)gridDim.x};
    const int half = gridDim.x >> 1, c = (int)blockIdx.x >= half ? 1 : 0;
    return Share3{c, (int)blockIdx.x - c * half, half};
}

// Per-block sums of rt^2 over the interior points of a colour, the same walk as a half-sweep
// (places and chunks of planes as a grid-stride loop over `tasks` = x_blocks * chunks).
template <int C>
__global__ void __launch_bounds__(kThreads3)
residual3_kernel(const Fields3 fld, int n, int W, Pairs3 npairs, int chunk, int x_blocks, int tasks, double one,
                 double *__restrict__ partials) {
    __shared__ double smem[kThreads3 / 32];
    const Share3 sh = share3<C>();
    const int colour = sh.colour;
    const double *__restrict__ self = colour ? fld.u[1] : fld.u[0], *__restrict__ other = colour ? fld.u[0] : fld.u[1];
    const double *__restrict__ hf = colour ? fld.hf[1] : fld.hf[0];
    const size_t plane = (size_t)(n + 2) * W;
    double acc = 0.0;
    for (int task = sh.block; task < tasks; task += sh.blocks) {
        const Place3 pl = place3(task % x_blocks, n, npairs);
        if (!pl.act) continue;
        const int i0 = 1 + task / x_blocks * chunk, i1 = min(n, i0 + chunk - 1);
        size_t at = ((size_t)i0 * (n + 2) + pl.j) * W + pl.m0;
        double2 vn = ldg2(other + at - plane), vm = ldg2(other + at);
        for (int i = i0; i <= i1; ++i, at += plane) {
            const double2 vs = ldg2(other + at + plane);
            const double2 vw = ldg2(other + at - W), ve = ldg2(other + at + W);
            const double2 f2 = ldg2(hf + at), me = ldg2(self + at);
            const int p = (i + pl.j + colour) & 1;
            const bool in = p ? pl.m0 + 2 < W : pl.m0 > 0;
            const double x = in ? __ldg(other + at + (p ? 2 : -1)) : 0.0;
            double s0 = add_fma(add_fma(add_fma(add_fma(f2.x, vn.x, one), vs.x, one), vw.x, one), ve.x, one);
            double s1 = add_fma(add_fma(add_fma(add_fma(f2.y, vn.y, one), vs.y, one), vw.y, one), ve.y, one);
            s0 = add_fma(add_fma(s0, p ? vm.x : x, one), p ? vm.y : vm.x, one);
            s1 = add_fma(add_fma(s1, p ? vm.y : vm.x, one), p ? x : vm.y, one);
            const double r0 = add_fma(s0, -__dmul_rn(6.0, me.x), one), r1 = add_fma(s1, -__dmul_rn(6.0, me.y), one);
            const int k0 = 2 * pl.m0 + p;
            if (k0 >= 1 && k0 <= n) acc = __fma_rn(r0, r0, acc);
            if (k0 + 2 <= n) acc = __fma_rn(r1, r1, acc);
            vn = vm;
            vm = vs;
        }
    }
    const double t = block_sum<kThreads3>(acc, smem);
    if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

// Per-block sums of (h^2 b)^2 over the interior points of a colour: h2 f plus, in N, S, W, E, D,
// U order, the neighbours on the shell.  The same walk and the same order of additions as
// residual3_kernel, so rho is exactly 1 for u = 0 inside and on the shell.  Only points next
// to the shell read u; everywhere else b is h2 f and the walk streams it.
template <int C>
__global__ void __launch_bounds__(kThreads3)
norm3_kernel(const Fields3 fld, int n, int W, Pairs3 npairs, int chunk, int x_blocks, int tasks,
             double *__restrict__ partials) {
    __shared__ double smem[kThreads3 / 32];
    const Share3 sh = share3<C>();
    const int colour = sh.colour;
    const double *__restrict__ other = colour ? fld.u[0] : fld.u[1], *__restrict__ hf = colour ? fld.hf[1] : fld.hf[0];
    const int L = n + 2;
    const size_t plane = (size_t)L * W;
    // a shell neighbour of a point has the other colour
    auto shell = [&](int i, int j, int k) { return other[((size_t)i * L + j) * W + (k >> 1)]; };
    double acc = 0.0;
    for (int task = sh.block; task < tasks; task += sh.blocks) {
        const Place3 pl = place3(task % x_blocks, n, npairs);
        if (!pl.act) continue;
        const int j = pl.j, i0 = 1 + task / x_blocks * chunk, i1 = min(n, i0 + chunk - 1);
        const double *row = hf + ((size_t)i0 * L + j) * W + pl.m0;
        const bool inner = j > 1 && j < n && pl.m0 > 0 && 2 * pl.m0 + 3 < n;  // for either parity
        int i = i0;
        if (inner && i0 > 1) {  // four planes' loads in flight, no index work
            const int last = min(i1, n - 1);
            for (; i + 3 <= last; i += 4, row += 4 * plane) {
                const double2 a = ldg2(row), b = ldg2(row + plane), c = ldg2(row + 2 * plane), d = ldg2(row + 3 * plane);
                acc = __fma_rn(a.x, a.x, acc), acc = __fma_rn(a.y, a.y, acc);
                acc = __fma_rn(b.x, b.x, acc), acc = __fma_rn(b.y, b.y, acc);
                acc = __fma_rn(c.x, c.x, acc), acc = __fma_rn(c.y, c.y, acc);
                acc = __fma_rn(d.x, d.x, acc), acc = __fma_rn(d.y, d.y, acc);
            }
        }
        for (; i <= i1; ++i, row += plane) {
            const double2 f2 = ldg2(row);
            const int k0 = 2 * pl.m0 + ((i + j + colour) & 1);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int k = k0 + 2 * q;
                if (k < 1 || k > n) continue;
                double b = q ? f2.y : f2.x;
                if (i == 1) b = __dadd_rn(b, shell(0, j, k));
                if (i == n) b = __dadd_rn(b, shell(n + 1, j, k));
                if (j == 1) b = __dadd_rn(b, shell(i, 0, k));
                if (j == n) b = __dadd_rn(b, shell(i, n + 1, k));
                if (k == 1) b = __dadd_rn(b, shell(i, j, 0));
                if (k == n) b = __dadd_rn(b, shell(i, j, n + 1));
                acc = __fma_rn(b, b, acc);
            }
        }
    }
    const double t = block_sum<kThreads3>(acc, smem);
    if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

// The blocks' partial sums added in a fixed order (one block).
__global__ void __launch_bounds__(kThreads3)
final3_kernel(const double *__restrict__ partials, int count, double *__restrict__ out) {
    __shared__ double smem[kThreads3 / 32];
    double v = 0.0;
    for (int q = threadIdx.x; q < count; q += kThreads3) v = __dadd_rn(v, partials[q]);
    const double t = block_sum<kThreads3>(v, smem);
    if (threadIdx.x == 0) *out = t;
}

int grid_for(size_t items) {
    static const int cap = [] {
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            sms = 152;
        }
        return 8 * sms;
    }();
    const size_t want = (items + kThreads3 - 1) / kThreads3;
    return (int)(want < (size_t)cap ? (want < 1 ? 1 : want) : cap);
}

bool dev_ptr(const void *p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

void free3(rbgs3d_ctx *c) {
    if (!c) return;
    for (int q = 0; q < 2; ++q) {
        cudaFree(c->u[q]);
        cudaFree(c->hf[q]);
    }
    cudaFree(c->staging);
    cudaFree(c->partials);
    cudaFree(c->dsum);
    if (c->hsum) cudaFreeHost(c->hsum);
    delete c;
}

// Launch shape of a walk over an n^3 grid: blocks of places, and planes per chunk.  Chunks of 8
// planes load the other colour's planes 1.25 times (from L2; 8 / 16 / 64 planes: 1553 / 1567 /
// 1585 us a sweep at 511^3); smaller grids take shorter chunks, so that there are about four
// blocks for each one that is resident.
struct Walk3 {
    Pairs3 npairs;
    int x_blocks, chunk, chunks;
};

Walk3 walk3(int n) {
    Walk3 w;
    const int np = active_width(n) / 2;
    w.npairs = Pairs3{np, (unsigned)(((1ull << 32) + np - 1) / np)};
    w.x_blocks = (n * np + kThreads3 - 1) / kThreads3;
    const long want = 4L * grid_for((size_t)1 << 40);  // 4 x 8 blocks for each SM
    long chunk = (long)n * w.x_blocks / want;
    w.chunk = (int)(chunk < 1 ? 1 : chunk > 8 ? 8 : chunk);
    w.chunks = (n + w.chunk - 1) / w.chunk;
    return w;
}

// Runs a reduction over both colours and adds its partials, red ones first: one launch for both
// where the blocks of both run at once (a residual of 7^3 / 33^3 / 63^3 / 64^3 takes 24.6 / 25.9 /
// 28.7 / 27.9 us, with a launch per colour 27.9 / 27.6 / 37.9 / 32.0), else one per colour, whose
// parity is then a constant (95^3 52, 300^3 524 us).
template <class Launch>
rbgs_status reduce3(rbgs3d_ctx *c, double *out, Launch launch) {
    const Walk3 w = walk3(c->n);
    const int tasks = w.x_blocks * w.chunks, blocks = std::min(tasks, kBlocks3);
    const Fields3 fld{{c->u[0], c->u[1]}, {c->hf[0], c->hf[1]}};
    if (2 * blocks <= grid_for((size_t)1 << 40)) {
        launch(std::integral_constant<int, kBoth>(), 2 * blocks, fld, w, tasks, c->partials);
    } else {
        launch(std::integral_constant<int, 0>(), blocks, fld, w, tasks, c->partials);
        RBGS_LAUNCH_CHECK();
        launch(std::integral_constant<int, 1>(), blocks, fld, w, tasks, c->partials + blocks);
    }
    RBGS_LAUNCH_CHECK();
    final3_kernel<<<1, kThreads3, 0, c->stream>>>(c->partials, 2 * blocks, out);
    RBGS_LAUNCH_CHECK();
    return RBGS_OK;
}

// sum rt^2 into dsum[0] (stream-ordered)
rbgs_status enqueue_residual3(rbgs3d_ctx *c) {
    return reduce3(c, c->dsum, [c](auto C, int blocks, const Fields3 &fld, const Walk3 &w, int tasks, double *partials) {
        residual3_kernel<decltype(C)::value><<<blocks, kThreads3, 0, c->stream>>>(fld, c->n, c->W, w.npairs, w.chunk,
                                                                                  w.x_blocks, tasks, 1.0, partials);
    });
}

// sum (h^2 b)^2 into dsum[1] (stream-ordered)
rbgs_status enqueue_norm3(rbgs3d_ctx *c) {
    return reduce3(c, c->dsum + 1, [c](auto C, int blocks, const Fields3 &fld, const Walk3 &w, int tasks,
                                       double *partials) {
        norm3_kernel<decltype(C)::value><<<blocks, kThreads3, 0, c->stream>>>(fld, c->n, c->W, w.npairs, w.chunk,
                                                                              w.x_blocks, tasks, partials);
    });
}

}  // namespace
}  // namespace rbgs

using namespace rbgs;

extern "C" {

rbgs_status rbgs3d_create(int n, double h2, const double *f, const double *u_init, void *cuda_stream,
                          rbgs3d_t *out) {
    clear_error();
    if (!out) { set_error("out is NULL"); return RBGS_EINVAL; }
    *out = nullptr;
    if (n < 1 || n > kMaxN3) { set_error("n = %d outside 1..%d", n, kMaxN3); return RBGS_EINVAL; }
    if (!(h2 > 0.0) || !std::isfinite(h2)) { set_error("h2 must be finite and > 0"); return RBGS_EINVAL; }
    if (!f || !u_init) { set_error("f and u_init must not be NULL"); return RBGS_EINVAL; }
    rbgs3d_ctx *c = new (std::nothrow) rbgs3d_ctx();
    if (!c) { set_error("out of host memory"); return RBGS_ENOMEM; }
    c->n = n;
    c->W = width3(n);
    c->h2 = h2;
    c->stream = (cudaStream_t)cuda_stream;
    const size_t L = (size_t)n + 2;
    const size_t colour = L * L * c->W * sizeof(double);
    bool ok = true;
    for (int q = 0; q < 2 && ok; ++q)
        ok = cudaMalloc(&c->u[q], colour) == cudaSuccess && cudaMalloc(&c->hf[q], colour) == cudaSuccess;
    ok = ok && cudaMalloc(&c->partials, 2 * kBlocks3 * sizeof(double)) == cudaSuccess;
    ok = ok && cudaMalloc(&c->dsum, 2 * sizeof(double)) == cudaSuccess;
    ok = ok && cudaMallocHost(&c->hsum, 2 * sizeof(double)) == cudaSuccess;
    const bool host_in = !dev_ptr(f) || !dev_ptr(u_init);
    ok = ok && (!host_in || cudaMalloc(&c->staging, L * L * L * sizeof(double)) == cudaSuccess);
    if (!ok) {
        cudaGetLastError();
        free3(c);
        set_error("allocation of the 3D solver's %zu-byte buffers failed", 4 * colour);
        return RBGS_ENOMEM;
    }
    // inputs in host memory go through device copies (u_init through the staging buffer,
    // f through a temporary one); device inputs are read in place
    const double *fv = f, *uv = u_init;
    const size_t nf = (size_t)n * n * n, nu = L * L * L;
    double *fstage = nullptr;
    if (host_in) {
        if (!dev_ptr(f)) {
            if (cudaMalloc(&fstage, nf * sizeof(double)) != cudaSuccess) {
                cudaGetLastError();
                free3(c);
                set_error("allocation of the 3D solver's f staging failed");
                return RBGS_ENOMEM;
            }
            if (cudaMemcpyAsync(fstage, f, nf * sizeof(double), cudaMemcpyDefault, c->stream) != cudaSuccess) {
                cudaGetLastError();
                cudaFree(fstage);
                free3(c);
                set_error("copy of f failed");
                return RBGS_ECUDA;
            }
            fv = fstage;
        }
        if (!dev_ptr(u_init)) {
            if (cudaMemcpyAsync(c->staging, u_init, nu * sizeof(double), cudaMemcpyDefault, c->stream) != cudaSuccess) {
                cudaGetLastError();
                cudaFree(fstage);
                free3(c);
                set_error("copy of u_init failed");
                return RBGS_ECUDA;
            }
            uv = c->staging;
        }
    }
    pack3_kernel<<<grid_for(L * L * c->W), kThreads3, 0, c->stream>>>(uv, fv, h2, c->u[0], c->u[1], c->hf[0],
                                                                      c->hf[1], n, c->W);
    rbgs_status st = cudaGetLastError() == cudaSuccess ? RBGS_OK : RBGS_ECUDA;
    if (st == RBGS_OK) st = enqueue_norm3(c);
    if (st == RBGS_OK && (cudaMemcpyAsync(c->hsum + 1, c->dsum + 1, sizeof(double), cudaMemcpyDeviceToHost, c->stream) !=
                              cudaSuccess ||
                          cudaStreamSynchronize(c->stream) != cudaSuccess)) {
        cudaGetLastError();
        st = RBGS_ECUDA;
    }
    cudaFree(fstage);
    if (st != RBGS_OK) {
        set_error("3D set-up failed");
        free3(c);
        return st;
    }
    c->den2 = c->hsum[1];
    *out = c;
    return RBGS_OK;
}

rbgs_status rbgs3d_sweep(rbgs3d_t c, long nsweeps) {
    clear_error();
    if (!c) { set_error("ctx is NULL"); return RBGS_EINVAL; }
    if (nsweeps < 0) { set_error("nsweeps < 0"); return RBGS_EINVAL; }
    const Walk3 w = walk3(c->n);
    const dim3 grid(w.x_blocks, w.chunks);
    for (long it = 0; it < nsweeps; ++it) {
        half_sweep3_kernel<0><<<grid, kThreads3, 0, c->stream>>>(c->u[0], c->u[1], c->hf[0], c->n, c->W, w.npairs,
                                                                      w.chunk, 1.0);
        RBGS_LAUNCH_CHECK();
        half_sweep3_kernel<1><<<grid, kThreads3, 0, c->stream>>>(c->u[1], c->u[0], c->hf[1], c->n, c->W, w.npairs,
                                                                      w.chunk, 1.0);
        RBGS_LAUNCH_CHECK();
    }
    return RBGS_OK;
}

rbgs_status rbgs3d_residual(rbgs3d_t c, double *rel) {
    clear_error();
    if (!c || !rel) { set_error("ctx and rel must not be NULL"); return RBGS_EINVAL; }
    rbgs_status st = enqueue_residual3(c);
    if (st != RBGS_OK) return st;
    RBGS_CUDA(cudaMemcpyAsync(c->hsum, c->dsum, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    RBGS_CUDA(cudaStreamSynchronize(c->stream));
    const double r2 = c->hsum[0];
    *rel = c->den2 > 0.0 ? std::sqrt(r2) / std::sqrt(c->den2) : std::sqrt(r2);
    if (!std::isfinite(*rel)) {
        set_error("residual is not finite");
        return RBGS_ENONFINITE;
    }
    return RBGS_OK;
}

rbgs_status rbgs3d_get_solution(rbgs3d_t c, double *u_out) {
    clear_error();
    if (!c || !u_out) { set_error("ctx and u_out must not be NULL"); return RBGS_EINVAL; }
    const size_t L = (size_t)c->n + 2, nu = L * L * L;
    const int grid = grid_for(L * L * c->W);
    if (dev_ptr(u_out)) {
        unpack3_kernel<<<grid, kThreads3, 0, c->stream>>>(c->u[0], c->u[1], u_out, c->n, c->W);
        RBGS_LAUNCH_CHECK();
        return RBGS_OK;
    }
    if (!c->staging && cudaMalloc(&c->staging, nu * sizeof(double)) != cudaSuccess) {
        cudaGetLastError();
        set_error("staging allocation failed");
        return RBGS_ENOMEM;
    }
    unpack3_kernel<<<grid, kThreads3, 0, c->stream>>>(c->u[0], c->u[1], c->staging, c->n, c->W);
    RBGS_LAUNCH_CHECK();
    RBGS_CUDA(cudaMemcpyAsync(u_out, c->staging, nu * sizeof(double), cudaMemcpyDefault, c->stream));
    RBGS_CUDA(cudaStreamSynchronize(c->stream));
    return RBGS_OK;
}

void rbgs3d_destroy(rbgs3d_t c) {
    if (!c) return;
    cudaStreamSynchronize(c->stream);
    free3(c);
}

}  // extern "C"
