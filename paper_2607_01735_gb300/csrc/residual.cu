// Residual-norm reduction (the convergence test of the solver).
//
// For every interior point, rt = ((((h2f + N) + S) + W) + E) - 4 u equals h^2 (b - A u)
// for the linear system of Eq. (1) with the ring folded into b.  One kernel walks strips of rows
// of the colour-split grid as the half-sweeps do (the other colour's rows i-1, i, i+1 in
// registers), squares each rt and reduces: warp shuffle, then the block; the last block to
// finish adds the blocks' partials in a fixed order and writes the results to the device and to
// page-locked host memory, so a residual is one launch and a wait.  The result is the same on
// every run.  Measured with the wait: 127^2 16 us (one launch per colour, a final sum and two
// copies: 32-44), 511^2 20-24 us (30-45), 16384^2 2.91 ms for both colours (3.00), the FP64
// pipe 93% busy there.  One value's chain of dependent operations after the other, each behind
// its own test: with the two values' chains interleaved the pipe was 84% busy.
//
// The adds run as fused multiply-adds by a run-time 1.0 (one rounding of the exact sum,
// the same value as the add, on GB300's faster-issuing DFMA path), and rt as
// fma(-4, u, s), the same value as s + (-4u) because 4u is exact.  GB300's FP64 pipe, not
// HBM, bounds this walk.
//
// ||h^2 b|| depends only on f and the ring; it is reduced once per problem by
// rhs_norm_kernel (h2f plus the ring neighbours of each boundary-adjacent point), walking
// the colour rows without any index division.
//
// Right after a full sweep the black points' rt is exactly zero: each black value was set
// to s * 0.25 from the very sum s the residual forms (the red values have not moved since),
// and 4 (s * 0.25) = s exactly (where s * 0.25 is subnormal and rounded, |rt| < 2^-1072 and
// its square adds nothing to the sum).  The red-black ordering gives this for any right-hand
// side (Section 2, Eq. (1)).  So after a sweep only the red points are walked: half the
// work, and the same sum bit for bit (the black partials were exact zeros).
//
// The same walk also serves the mixed-precision refinement: with the sum it forms max |rt| (exact,
// order-independent) and stores (float)rt, from which the scaled defect (float)(rt * 2^-e) follows
// by an exact multiplication (mixed.cu) unless some rt is far below 1.  (A second walk that formed
// rt again with the scale known took 0.97 ms an outer step at 8192^2; the multiplication takes 0.08:
// 200 sweeps in two outer steps 13.8 ms, now 12.1.)
#include "common.cuh"
#include "fp64.cuh"
#include "sweep_impl.cuh"

namespace rbgs {
namespace {

constexpr int kAhead = 8;  // partials loaded at once by the finishing block

// The last block of a launch adds all its partials in a fixed order (whichever block is last),
// so a reduction is one launch.  ticket: zero before the launch, zero again after it.
// Every block calls this with its own partials written (by thread 0).
template <int THREADS>
__device__ __forceinline__ bool last_block(unsigned *ticket, unsigned blocks) {
    __shared__ bool s_last;
    if (threadIdx.x == 0) {
        __threadfence();  // this block's partials before its ticket
        s_last = atomicAdd(ticket, 1u) == blocks - 1;
        if (s_last) {
            *ticket = 0;
            __threadfence();  // every partial is visible from here on
        }
    }
    __syncthreads();
    return s_last;
}

template <int THREADS>
__device__ __forceinline__ double sum_partials(const double *partials, int count, double *smem) {
    double v = 0.0;
    for (int q = threadIdx.x; q < count; q += kAhead * THREADS) {
        double t[kAhead];
#pragma unroll
        for (int r = 0; r < kAhead; ++r) t[r] = q + r * THREADS < count ? __ldcg(partials + q + r * THREADS) : 0.0;
#pragma unroll
        for (int r = 0; r < kAhead; ++r) v = __dadd_rn(v, t[r]);
    }
    __syncthreads();
    return block_sum<THREADS>(v, smem);
}

// (float)r for 2^-126 <= |r| < 2^127 or r = 0 (m: the bits of |r|), rounded to nearest even on the
// integer pipe: the walk's FP64 pipe is full, and the conversion would be a seventh instruction on
// it (the walk with it 1.09 ms at 8192^2, with this 0.97).
__device__ __forceinline__ float narrow(double r, long long m) {
    const unsigned long long t = (unsigned long long)m + 0x0FFFFFFFull + ((m >> 29) & 1);
    const unsigned f = m ? (unsigned)(t >> 29) - (896u << 23) : 0u;  // exponent bias 1023 to 127
    return __uint_as_float(f | ((unsigned)__double2hiint(r) & 0x80000000u));
}

struct ResidualArgs {
    const double *u[2], *hf[2];
    int n, W, kact;
    int rows, bx, items, colours;  // strips: rows each, bx of them across, `items` per colour
    int lanes;                     // blocks that share a colour's strips
    double *partials;       // sums, then (from kMaxPartials) maxima
    double *out;            // [0] sum rt^2, [2] max |rt|
    double *host;           // the same in page-locked host memory ([2] negative: see MAX), and [3] the device status
    const int *status;
    unsigned *ticket;
    float *r32[2];          // WRITE, MAX: FP32 colour arrays of pitch W32
    int W32;
    double scale, one;
};

// MAX: also reduce max |rt| and store (float)rt into the FP32 colour arrays at interior points;
// host[2] is -max where some 0 < |rt| < 2^-102, whose binary32 form, scaled down by up to 2^24, may
// have lost bits.  WRITE: only
// store (float)(rt * scale) there: the scaled defect that the refinement hands to its FP32 inner
// solver.
// Values per thread: PTS neighbouring ones of a colour row.  The grid is one wave of resident
// blocks, each walking every gridDim.x-th strip of the red and then of the black points (a grid
// of strips ran 1.4 waves at 16384^2).  Small grids give the black points blocks of their own.
// Either way the red points' sum does not depend on whether the black ones are walked: their
// partials keep their places and the black ones come after them.
template <bool MAX, bool WRITE, int PTS>
__global__ void __launch_bounds__(kSweepThreads) residual_kernel(const ResidualArgs a) {
    __shared__ double smem[kSweepThreads / 32];
    const int n = a.n, W = a.W;
    const double one = a.one;
    const int lane = threadIdx.x & 31;
    double acc = 0.0, mx = 0.0;
    bool tiny = false;
    const int own = (int)blockIdx.x >= a.lanes ? 1 : 0;  // blocks past `lanes`: the black points alone
    const int last_colour = (int)gridDim.x > a.lanes ? own : a.colours - 1;
    for (int colour = own; colour <= last_colour; ++colour) {
    const double *__restrict__ self = colour ? a.u[1] : a.u[0], *__restrict__ other = colour ? a.u[0] : a.u[1];
    const double *__restrict__ hf = colour ? a.hf[1] : a.hf[0];
    float *__restrict__ r32 = colour ? a.r32[1] : a.r32[0];
        for (int item = blockIdx.x - own * a.lanes; item < a.items; item += a.lanes) {
            const int strip = item / a.bx;
            const int k0 = PTS * ((item - strip * a.bx) * kSweepThreads + threadIdx.x);
            const bool act = k0 < a.kact;
            const int i0 = 1 + strip * a.rows, i1 = min(n, i0 + a.rows - 1);
            double up[PTS], mid[PTS], dn[PTS], f[PTS], me[PTS];
            load_row<PTS>(up, other + (size_t)(i0 - 1) * W + k0, act);
            load_row<PTS>(mid, other + (size_t)i0 * W + k0, act);
            for (int i = i0; i <= i1; ++i) {
                const size_t row = (size_t)i * W;
                load_row<PTS>(dn, other + row + W + k0, act);
                load_row<PTS>(f, hf + row + k0, act);
                load_row<PTS>(me, self + row + k0, act);
                const int p = (i + colour) & 1;
                // value q: west/east at k0+q-1, k0+q (p = 0) or k0+q, k0+q+1 (p = 1)
                double w[PTS], e[PTS];
                if (p == 0) {
                    double x = __shfl_up_sync(0xffffffffu, mid[PTS - 1], 1);
                    if (lane == 0) x = (act && k0 > 0) ? __ldg(other + row + k0 - 1) : 0.0;
#pragma unroll
                    for (int q = 0; q < PTS; ++q) w[q] = q ? mid[q ? q - 1 : 0] : x, e[q] = mid[q];
                } else {
                    double x = __shfl_down_sync(0xffffffffu, mid[0], 1);
                    if (lane == 31) x = (k0 + PTS < a.kact) ? __ldg(other + row + k0 + PTS) : 0.0;
#pragma unroll
                    for (int q = 0; q < PTS; ++q) w[q] = mid[q], e[q] = q + 1 < PTS ? mid[q + 1 < PTS ? q + 1 : 0] : x;
                }
                const int j0 = 2 * k0 + p;
                float keep[PTS];
#pragma unroll
                for (int q = 0; q < PTS; ++q) {
                    if (!(act && j0 + 2 * q >= 1 && j0 + 2 * q <= n)) continue;
                    const double s =
                        add_fma(add_fma(add_fma(add_fma(f[q], up[q], one), dn[q], one), w[q], one), e[q], one);
                    const double r = __fma_rn(-4.0, me[q], s);
                    if (WRITE) {
                        r32[(size_t)i * a.W32 + k0 + q] = __double2float_rn(__dmul_rn(r, a.scale));
                    } else {
                        acc = __fma_rn(r, r, acc);
                        // |r| compares as its bits do; a NaN sorts above everything and the sum shows it
                        if (MAX) {
                            const long long m = __double_as_longlong(r) & 0x7FFFFFFFFFFFFFFFll;
                            tiny |= (unsigned long long)(m - 1) < 0x398FFFFFFFFFFFFFull;  // 2^-102: 0x399 << 52
                            keep[q] = narrow(r, m);
                            mx = m > __double_as_longlong(mx) ? __longlong_as_double(m) : mx;
                        }
                    }
                }
                if (MAX) {
                    float *to = r32 + (size_t)i * a.W32 + k0;
                    if (PTS == 2 && act && j0 >= 1 && j0 + 2 <= n) {
                        *reinterpret_cast<float2 *>(to) = make_float2(keep[0], keep[PTS - 1]);
                    } else {
#pragma unroll
                        for (int q = 0; q < PTS; ++q)
                            if (act && j0 + 2 * q >= 1 && j0 + 2 * q <= n) to[q] = keep[q];
                    }
                }
#pragma unroll
                for (int q = 0; q < PTS; ++q) up[q] = mid[q], mid[q] = dn[q];
            }
        }
    }
    if (WRITE) return;
    const int blocks = gridDim.x, slot = blockIdx.x;
    const double t = block_sum<kSweepThreads>(acc, smem);
    if (threadIdx.x == 0) a.partials[slot] = t;
    if (MAX) {
        const bool any = __syncthreads_or(tiny);
        const double m = block_max<kSweepThreads>(mx, smem);
        if (threadIdx.x == 0) a.partials[kMaxPartials + slot] = any ? -m : m;
    }
    if (!last_block<kSweepThreads>(a.ticket, blocks)) return;
    const double sum = sum_partials<kSweepThreads>(a.partials, blocks, smem);
    if (threadIdx.x == 0) a.out[0] = a.host[0] = sum, a.host[3] = (double)*a.status;
    if (MAX) {
        bool any = false;
        double v = 0.0;
        for (int q = threadIdx.x; q < blocks; q += kSweepThreads) {
            const double m = __ldcg(a.partials + kMaxPartials + q);
            any |= m < 0.0;
            v = fmax(v, fabs(m));
        }
        any = __syncthreads_or(any);
        const double m = block_max<kSweepThreads>(v, smem);
        if (threadIdx.x == 0) a.out[2] = m, a.host[2] = any ? -m : m;
    }
}

__device__ __forceinline__ double at(const double *const *u, int W, int i, int j) {
    return u[(i + j) & 1][(size_t)i * W + (j >> 1)];
}

struct ColourPtrs { const double *p[2]; };

// Partial sums of (h^2 b)^2: h2f plus, in N, S, W, E order, the neighbours on the ring.
// Thread t of block (x, y) takes elements k0 = 2t and k0 + 1 of both colour rows (one 16-byte
// load per colour row) down the block's rows, loading four rows ahead of their use so that
// eight loads are in flight.  Away from the first and last interior row and column, b is h2f
// itself (no ring neighbour), so those rows take four fused multiply-adds and no index
// arithmetic: the walk is bound by HBM, not by instruction issue.
constexpr int kNormThreads = 256;
constexpr int kNormRowsAhead = 4;

__global__ void __launch_bounds__(kNormThreads)
rhs_norm_kernel(ColourPtrs u, ColourPtrs hf, int n, int W, int kact, int rows_per_block,
                double *__restrict__ partials, double *__restrict__ out, double *__restrict__ host,
                unsigned *ticket) {
    __shared__ double smem[kNormThreads / 32];
    const int k0 = 2 * (blockIdx.x * kNormThreads + threadIdx.x);
    const int i0 = 1 + blockIdx.y * rows_per_block, i1 = min(n, i0 + rows_per_block - 1);
    // this thread's columns 2 k0 + {0..3} all lie in 2..n-1
    const bool inner_cols = k0 > 0 && 2 * k0 + 3 < n;
    double acc = 0.0;
    if (k0 < kact) {  // k0 + 1 < W always (W is even and at least kact)
        for (int i = i0; i <= i1; i += kNormRowsAhead) {
            double2 v[kNormRowsAhead][2];
#pragma unroll
            for (int r = 0; r < kNormRowsAhead; ++r) {
                const size_t row = (size_t)min(i + r, i1) * W;  // rows past i1: reloaded, unused
                v[r][0] = ldg2(hf.p[0] + row + k0);
                v[r][1] = ldg2(hf.p[1] + row + k0);
            }
#pragma unroll
            for (int r = 0; r < kNormRowsAhead; ++r) {
                const int ii = i + r;
                if (ii > i1) break;
                if (inner_cols && ii > 1 && ii < n) {
                    acc = __fma_rn(v[r][0].x, v[r][0].x, acc);
                    acc = __fma_rn(v[r][0].y, v[r][0].y, acc);
                    acc = __fma_rn(v[r][1].x, v[r][1].x, acc);
                    acc = __fma_rn(v[r][1].y, v[r][1].y, acc);
                    continue;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int c = q >> 1, k = k0 + (q & 1);
                    const int j = 2 * k + ((ii + c) & 1);  // natural column of element k, colour c
                    if (j < 1 || j > n) continue;
                    double b = (q & 1) ? v[r][c].y : v[r][c].x;
                    if (ii == 1) b = __dadd_rn(b, at(u.p, W, 0, j));
                    if (ii == n) b = __dadd_rn(b, at(u.p, W, n + 1, j));
                    if (j == 1) b = __dadd_rn(b, at(u.p, W, ii, 0));
                    if (j == n) b = __dadd_rn(b, at(u.p, W, ii, n + 1));
                    acc = __fma_rn(b, b, acc);
                }
            }
        }
    }
    const double t = block_sum<kNormThreads>(acc, smem);
    if (threadIdx.x == 0) partials[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = t;
    if (!last_block<kNormThreads>(ticket, gridDim.x * gridDim.y)) return;
    const double sum = sum_partials<kNormThreads>(partials, gridDim.x * gridDim.y, smem);
    if (threadIdx.x == 0) *out = *host = sum;
}

// Rows per block: up to `most`, fewer where that would leave the GPU with fewer than about four
// blocks per SM (a thread walks its rows one after another: 16 rows of a 127^2 grid took 17 us,
// one row takes 4), and at most `blocks` blocks in all (a power-of-two number of rows then).
int block_rows(int n, int bx, int most, int blocks) {
    static const int sms = [] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) {
            cudaGetLastError();
            v = 152;
        }
        return v;
    }();
    const long r = (long)n * bx / (4L * sms);
    int rows = (int)(r < 1 ? 1 : r > most ? most : r);
    while ((size_t)bx * ((n + rows - 1) / rows) > (size_t)blocks) rows *= 2;
    return rows;
}

// red_only: the black points' rt is known to be zero (the iterate is the result of a full
// sweep); only the red partials are formed and summed.
template <bool MAX, bool WRITE>
rbgs_status residual_pass(const rbgs_ctx *c, double scale, cudaStream_t s, bool red_only) {
    const Geometry &g = c->g;
    ResidualArgs a;
    for (int q = 0; q < 2; ++q) {
        a.u[q] = c->f64.u[q], a.hf[q] = c->f64.hf[q];
        a.r32[q] = WRITE || MAX ? c->f32.hf[q] : nullptr;
    }
    a.n = g.n, a.W = g.W, a.kact = active_width(g.n), a.W32 = c->f32.W;
    a.colours = red_only ? 1 : 2;
    a.partials = c->partials, a.out = c->dsum, a.host = c->hsum;
    a.status = c->dstatus, a.ticket = c->pcounter + 1;
    a.scale = scale, a.one = 1.0;
    static const int wave = [] {  // resident blocks of the GPU, per template instance
        int dev = 0, sms = 0, per_sm = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, residual_kernel<MAX, WRITE, 2>, kSweepThreads, 0) !=
                cudaSuccess ||
            sms < 1 || per_sm < 1) {
            cudaGetLastError();
            return 1024;
        }
        return sms * per_sm < kMaxPartials ? sms * per_sm : kMaxPartials;
    }();
    // strips of up to 16 rows, and on large grids the tallest ones that give each block four:
    // short strips start over too often (84% of the FP64 pipe at 8192^2 with 16 rows, 92% so)
    a.bx = (a.kact + 2 * kSweepThreads - 1) / (2 * kSweepThreads);
    a.rows = block_rows(g.n, a.bx, 16, 1 << 30);
    const int strips = 4 * wave / a.bx;
    if (strips > 0 && (g.n + strips - 1) / strips > a.rows) a.rows = (g.n + strips - 1) / strips;
    a.items = a.bx * ((g.n + a.rows - 1) / a.rows);
    a.lanes = a.items < wave ? a.items : wave;
    const int grid = !red_only && 2 * a.lanes <= wave ? 2 * a.lanes : a.lanes;
    residual_kernel<MAX, WRITE, 2><<<grid, kSweepThreads, 0, s>>>(a);
    RBGS_LAUNCH_CHECK();
    return RBGS_OK;
}

}  // namespace

rbgs_status launch_residual_sum(const rbgs_ctx *c, cudaStream_t s) {
    return residual_pass<false, false>(c, 1.0, s, c->black_fresh);
}

// write_r32 = false: sum rt^2 -> dsum[0], max |rt| -> dsum[2], r32 = (float)rt at interior points.
// write_r32 = true:  r32 = (float)(rt * scale) at interior points.
rbgs_status launch_defect(const rbgs_ctx *c, bool write_r32, double scale, cudaStream_t s) {
    return write_r32 ? residual_pass<false, true>(c, scale, s, false) : residual_pass<true, false>(c, scale, s, false);
}

rbgs_status launch_rhs_norm(const rbgs_ctx *c, cudaStream_t s) {
    const Geometry &g = c->g;
    ColourPtrs u{{c->f64.u[0], c->f64.u[1]}}, hf{{c->f64.hf[0], c->f64.hf[1]}};
    const int kact = active_width(g.n);
    const int bx = (kact + 2 * kNormThreads - 1) / (2 * kNormThreads);
    const int rows = block_rows(g.n, bx, 16, kMaxPartials);
    const dim3 grid(bx, (g.n + rows - 1) / rows);
    rhs_norm_kernel<<<grid, kNormThreads, 0, s>>>(u, hf, g.n, g.W, kact, rows, c->partials, c->dsum + 1,
                                                     c->hsum + 1, c->pcounter + 2);
    RBGS_LAUNCH_CHECK();
    return RBGS_OK;
}

}  // namespace rbgs
