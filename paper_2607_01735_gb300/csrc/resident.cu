// Many sweeps of a small grid in one cooperative launch, each block's tile held in shared memory.
//
// On a small grid a half-sweep is less work than a launch or a grid barrier (about 2 us each).
// Here the grid is cut into tiles, one per block and SM.  A block keeps both colours of its tile
// and of a halo around it, and h2 f, in shared memory for the whole launch.  A period of K
// sweeps (2K half-sweeps of Eq. (1), red then black) runs inside the block: half-sweep s updates
// the tile plus a margin that shrinks from 2K - 1 rows (and as many columns) to none, so what
// the tile ends with is exact, and only the block barrier separates the colours.  After a period
// a block needs its halo's black values again (the red ones are recomputed), 2K rows and K values
// of a colour row deep, from its eight neighbours: no wait on any other block.
//
// Exchange: a slot of global memory per black point and parity of the period, which holds the
// value with the period's number (tile_exchange.cuh).  Two parities suffice: a block writes the
// slots of period q + 2 only after it has read its neighbours' period q + 1 values, which they
// wrote after reading its period q ones.  The numbers continue from launch to launch (the last
// block to finish advances them in device memory), so nothing is cleared, and a captured launch
// can be replayed.  Every wait is bounded: after kRPolls polls, or when another block has given
// up, the block records a status and leaves; the host reports it as RBGS_ETIMEOUT at its next
// synchronising call.
//
// Tile and period: chosen per grid size from a model of the three costs (plan below): the
// updates of the shrinking regions, a fixed cost per half-sweep (the chain of dependent
// operations and the block barrier), and the exchange.
//
// While solvers on other streams are at work, a launch takes a part of the SMs (shared_plan).
//
// Measured, a sweep, against what ran before (cached graphs of one launch per colour, or one
// cooperative launch with a grid barrier per colour): FP64 127^2 1.1 us (3.9), 255^2 1.7 (4.0),
// 511^2 3.4 (6.4), 1023^2 9.7 (14.1), 1190^2 12.9 (19.4); fused 255^2 1.3 us (4.4), 1023^2 4.3
// (7.2 as wavefront passes); FP32 255^2 0.8 us (3.1), 511^2 1.2 (3.3), 1000^2 2.8 (3.9).  What
// bounds it: from about 700^2 the FP64 pipe (70% of its rate at 1023^2 by ncu, the shrinking
// margins included), below the chain of a half-sweep and the exchange, about 1 us together.
//
// Three kinds of values, as in wavefront.cu: double (bit-exact FP64), float (inner sweeps of the
// refinement) and int64 (the fused update on its block's fixed-point grid; the iterate is
// converted as it is loaded, and the last sweep's sums are written as binary64).  Each equals
// one launch per colour bit for bit.
#include <type_traits>

#include "common.cuh"
#include "fixed64.cuh"
#include "fp64.cuh"
#include "per_device.cuh"
#include "sweep_impl.cuh"
#include "tile_exchange.cuh"

namespace rbgs {
namespace {

constexpr int kRThreads = 512;
constexpr uint32_t kRPolls = 1u << 22;
constexpr int kMaxPeriod = 8;       // sweeps per period at most
constexpr int kSmemMax = 220 * 1024;
constexpr unsigned long long kNoScale = 0x8000000000000000ull;  // fused: no valid scale

template <typename T>
struct ResTypes {
    using S = T;  // type of the iterate in global memory
};
template <>
struct ResTypes<int64_t> {
    using S = double;
};

template <typename T>
struct RArgs {
    using S = typename ResTypes<T>::S;
    S *u0, *u1;
    const T *hf0, *hf1;
    const unsigned long long *words;  // fused: [2] the block's scale
    unsigned long long *slots;        // [parity][row W + k]: 1 (float) or 2 words each
    unsigned *epoch;                  // [0] number of the last period, [1] blocks that have finished
    int *status;
    int n, W, kmax, kint;             // values of a colour row holding columns 0..n+1, 1..n
    int gx, gy, period;               // tiles; K
    int pitch, erows;                 // values per row and rows of the tile with its halo
    long long sweeps;
    double one;
};

// The region a half-sweep updates when its margin is e rows: rows i0.., values k0.. (w of them)
struct Region {
    int i0, k0, w, items;
    unsigned mul;  // ceil(2^32 / w): item / w = umulhi(item, mul) while item w < 2^32
};

__device__ __forceinline__ float r_update(float hf, float vn, float vs, float vw, float ve, double) {
    float s = __fadd_rn(hf, vn);
    s = __fadd_rn(s, vs);
    s = __fadd_rn(s, vw);
    s = __fadd_rn(s, ve);
    return __fmul_rn(s, 0.25f);
}
__device__ __forceinline__ double r_update(double hf, double vn, double vs, double vw, double ve, double one) {
    return update_f64<false>(0, hf, vn, vs, vw, ve, one);
}

template <typename T>
__global__ void __launch_bounds__(kRThreads, 1) resident_kernel(const RArgs<T> a) {
    using S = typename ResTypes<T>::S;
    using Bits = typename std::conditional<sizeof(T) == 8, uint64_t, uint32_t>::type;
    constexpr bool FUSED = std::is_same<T, int64_t>::value;
    constexpr int kWords = kSlotWords<Bits>;
    extern __shared__ __align__(16) unsigned char r_shared[];
    __shared__ Region regions[2 * kMaxPeriod];
    __shared__ int s_nrcv, s_abort;
    const int tid = threadIdx.x;
    const double one = a.one;
    const int n = a.n, W = a.W, kmax = a.kmax, K = a.period, pitch = a.pitch;
    const int ty = blockIdx.x / a.gx, tx = blockIdx.x % a.gx;
    // the tile's rows and values (balanced: sizes differ by one at most)
    const int ra = 1 + ty * n / a.gy, rb = 1 + (ty + 1) * n / a.gy;
    const int ka = tx * a.kint / a.gx, kb = (tx + 1) * a.kint / a.gx;
    const int ibase = ra - 2 * K, kbase = ka - K - 1;  // grid place of shared element 0
    const int plane = a.erows * pitch;                 // elements of one colour
    T *su = reinterpret_cast<T *>(r_shared);           // u: red, black; then h2 f: red, black
    T *sf = su + 2 * plane;
    int2 *rcv = reinterpret_cast<int2 *>(sf + 2 * plane);  // halo points: {shared element, grid element}

    if (block_given_up(a.status)) return;  // a wait of an earlier launch gave up
    unsigned long long ew = 0;
    if (FUSED) ew = a.words[2];
    const bool ok_scale = ew != kNoScale;
    const int e2 = ok_scale ? (int)(long long)ew : 0;
    const unsigned seq0 = *reinterpret_cast<volatile unsigned *>(a.epoch);
    if (tid == 0) s_nrcv = 0, s_abort = 0;
    if (tid < 2 * K) {
        const int e = tid, ek = (e + 1) >> 1;
        Region r;
        r.i0 = max(1, ra - e);
        r.k0 = max(0, ka - ek);
        r.w = min(a.kint, kb + ek) - r.k0;
        r.items = (min(n, rb - 1 + e) - r.i0 + 1) * r.w;
        r.mul = 0xFFFFFFFFu / (unsigned)r.w + 1u;
        regions[e] = r;
    }
    __syncthreads();
    for (int q = tid; q < plane; q += kRThreads) {
        const int i = ibase + q / pitch, k = kbase + q % pitch;
        T v0 = T(0), v1 = T(0), f0 = T(0), f1 = T(0);
        if (i >= 0 && i <= n + 1 && k >= 0 && k < kmax) {
            const size_t at = (size_t)i * W + k;
            if constexpr (FUSED) {
                if (ok_scale) v0 = to_fixed(a.u0[at], e2), v1 = to_fixed(a.u1[at], e2);
            } else {
                v0 = a.u0[at], v1 = a.u1[at];
            }
            f0 = a.hf0[at], f1 = a.hf1[at];
            // a black point of the halo, inside the ring and outside the tile: received each period
            const int j = 2 * k + ((i + 1) & 1);
            if (i >= 1 && i <= n && i < rb + 2 * K && j >= 1 && j <= n && k >= ka - K && k < kb + K &&
                !(i >= ra && i < rb && k >= ka && k < kb))
                rcv[atomicAdd(&s_nrcv, 1)] = make_int2(plane + q, (int)at);
        }
        su[q] = v0, su[plane + q] = v1;
        sf[q] = f0, sf[plane + q] = f1;
    }
    __syncthreads();
    const int nrcv = s_nrcv;
    const size_t parity_words = (size_t)(n + 2) * W * kWords;

    // one half-sweep of colour c with margin e; publish: the tile's outgoing black values with
    // number seq; final: fused only, the sums leave as binary64
    auto half_sweep = [&](int c, int e, bool publish, unsigned seq, bool final) {
        const Region r = regions[e];
        T *self = su + c * plane;
        const T *other = su + (c ^ 1) * plane;
        const T *f = sf + c * plane;
        unsigned long long *slots = a.slots + (seq & 1u) * parity_words;
        for (int base = 0; base < r.items; base += kRThreads) {
            if (base + (tid & ~31) >= r.items) break;  // warp-uniform: no item left for this warp
            const bool act = base + tid < r.items;
            const int item = act ? base + tid : base;
            const int row = r.w == 1 ? item : (int)__umulhi((unsigned)item, r.mul);
            const int i = r.i0 + row, k = r.k0 + (item - row * r.w);
            const int p = (i + c) & 1, j = 2 * k + p;
            const int q = (i - ibase) * pitch + (k - kbase);
            const bool in = act && j >= 1 && j <= n;
            T v;
            if constexpr (FUSED) {
                const int64_t s = f[q] + other[q - pitch] + other[q + pitch] + other[q - 1 + p] + other[q + p];
                v = fixed_quarter(s);
                if (final && in && i >= ra && i < rb && k >= ka && k < kb)
                    (c ? a.u1 : a.u0)[(size_t)i * W + k] =
                        ok_scale ? fixed_quarter_to_double(s, e2) : __longlong_as_double(0x7FF8000000000000ll);
            } else {
                v = r_update(f[q], other[q - pitch], other[q + pitch], other[q - 1 + p], other[q + p], one);
            }
            if (in) {
                self[q] = v;
                // the margin is 0 here, so (i, k) is in the tile: its outer 2K rows and K values
                if (publish && (i < ra + 2 * K || i >= rb - 2 * K || k < ka + K || k >= kb - K)) {
                    Bits b;
                    __builtin_memcpy(&b, &v, sizeof(T));
                    slot_put(slots + ((size_t)i * W + k) * kWords, b, seq);
                }
            }
        }
        __syncthreads();
    };

    unsigned seq = seq0;
    long long left = a.sweeps;
    // a launch of several tiles has at least two periods: a tile's result is written over the
    // iterate only after every neighbour has loaded (it has received their first period)
    int kk = (int)(left > K ? K : gridDim.x > 1 ? (left + 1) / 2 : left);
    while (left > 0) {
        left -= kk;
        ++seq;
        for (int s = 0; s < kk; ++s) {
            const bool last = left == 0 && s == kk - 1;
            half_sweep(0, 2 * (kk - s) - 1, false, seq, last);
            half_sweep(1, 2 * (kk - s) - 2, left > 0 && s == kk - 1 && gridDim.x > 1, seq, last);
        }
        if (left == 0) break;
        kk = (int)(left < K ? left : K);
        // the halo's black values of this period
        if (!receive_slots<T, Bits, kRThreads>(su, rcv, nrcv, a.slots + (seq & 1u) * parity_words, seq, a.status,
                                               &s_abort, kRPolls))
            return;
    }
    if constexpr (!FUSED) {
        for (int q = tid; q < plane; q += kRThreads) {
            const int i = ibase + q / pitch, k = kbase + q % pitch;
            if (i < ra || i >= rb || k < ka || k >= kb) continue;
            const size_t at = (size_t)i * W + k;
            const int j = 2 * k + (i & 1);  // red; black is the other column of the pair
            if (j >= 1 && j <= n) a.u0[at] = su[q];
            const int jb = 2 * k + ((i + 1) & 1);
            if (jb >= 1 && jb <= n) a.u1[at] = su[plane + q];
        }
    }
    // the last block to finish advances the period number for the next launch
    if (tid == 0 && atomicAdd(&a.epoch[1], 1u) == gridDim.x - 1) {
        a.epoch[1] = 0;
        a.epoch[0] = seq;
    }
}

int device_sms() {
    static PerDevice<int> sms;
    return sms.get([] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            v = 0;
        }
        return v;
    });
}

template <typename T>
size_t resident_smem(int rows, int vals, int K) {
    const size_t pts = (size_t)(rows + 4 * K) * (vals + 2 * K + 2);
    const size_t halo = (size_t)4 * K * (vals + 2 * K) + (size_t)2 * K * rows;
    return pts * 4 * sizeof(T) + halo * sizeof(int2);
}

constexpr double kCyclesPerUs = 2070.0;  // of the clock at which the model's figures were taken

// Cycles of the model, per type: a warp's update of 32 points on its quarter of an SM (FP64: four
// adds at half a lane per clock), a half-sweep's chain and barrier, an exchange.  A region of
// items takes as long as the quarter with the most warps, so a plan is better off just below a
// multiple of 128 items.  Fitted to sweeps at 63^2 and 1023^2 with the period forced to 1 to 4.
template <typename T>
struct Costs {
    static constexpr double warp = 300, chain = 500, exchange = 1600;
};
template <>
struct Costs<float> {
    static constexpr double warp = 76, chain = 250, exchange = 1900;
};
template <>
struct Costs<int64_t> {
    static constexpr double warp = 117, chain = 590, exchange = 1550;
};

// The current device takes a cooperative launch of this kernel with one block on every SM.  The
// shared-memory limit is raised for every context, not once per device: the plain launches that
// this kernel replaced needed none, and a cudaDeviceReset takes it back.
template <typename T>
bool can_run() {
    static PerDevice<bool> fits;
    if (cudaFuncSetAttribute(resident_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) !=
        cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return fits.get([] {
        int dev = 0, coop = 0, per_sm = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, resident_kernel<T>, kRThreads, kSmemMax) !=
                cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        return coop != 0 && per_sm >= 1;
    });
}

// The fastest plan of at most `blocks` tiles.
template <typename T>
ResidentPlan plan_for(int n, int blocks) {
    ResidentPlan best{};
    if (!can_run<T>()) return best;
    double best_cost = 0.0;
    const int kint = n / 2 + 1;
    for (int K = 1; K <= kMaxPeriod; ++K) {
        for (int gx = 1; gx <= blocks && gx <= kint; ++gx) {
            int gy = blocks / gx;
            if (n / gy < 2 * K) gy = n / (2 * K) > 1 ? n / (2 * K) : 1;
            const int vals = (kint + gx - 1) / gx, rows = (n + gy - 1) / gy;
            // A halo reaches no further than the next tile; and every tile has a black interior
            // point to send to each of its neighbours, so that no tile runs ahead of one that
            // has yet to read from it: 2K rows hold both parities, and two values of which the
            // inner one is no ring value in either.
            if (gx > 1 && kint / gx < (K > 2 ? K : 2)) continue;
            if (resident_smem<T>(rows, vals, K) > (size_t)kSmemMax) continue;
            double cost = gx * gy > 1 ? Costs<T>::exchange : 0.0;
            for (int e = 0; e < 2 * K; ++e) {
                const int m = gy > 1 ? 2 * e : 0, mk = gx > 1 ? 2 * ((e + 1) / 2) : 0;
                const int warps = ((rows + m) * (vals + mk) + 31) / 32;
                cost += Costs<T>::chain + Costs<T>::warp * ((warps + 3) / 4);
            }
            cost /= K;
            if (best.rows == 0 || cost < best_cost) {
                best_cost = cost;
                best = ResidentPlan{gx, gy, rows, vals, K, cost / kCyclesPerUs};
            }
        }
    }
    return best;
}

// The plan for a launch when `streams` streams share the device: of the plans for 1, 2, 3, 4, 6, 8,
// 12 and 16 equal parts of it, the one with the least time for all streams' sweeps by the model.
// A part's tiles are larger, so a sweep takes longer but recomputes less of its neighbours' rows:
// FP64 127^2 1.2 us on 152 SMs, 2.3 on 19.
template <typename T>
const ResidentPlan &shared_plan(ResidentState &r, int n, int streams) {
    static constexpr int parts[kResidentShares] = {1, 2, 3, 4, 6, 8, 12, 16};
    const int sms = device_sms();
    int best = 0;
    double least = r.plan[0].us * streams;
    for (int q = 1; q < kResidentShares && parts[q - 1] < streams; ++q) {
        if (!r.planned[q]) {
            r.plan[q] = plan_for<T>(n, sms / parts[q]);
            r.planned[q] = true;
        }
        const ResidentPlan &p = r.plan[q];
        if (p.rows == 0) break;  // nor do smaller parts hold the grid
        const int at_once = sms / (p.gx * p.gy);
        const double us = p.us * ((streams + at_once - 1) / at_once);
        if (us < least) least = us, best = q;
    }
    return r.plan[best];
}

template <typename T>
rbgs_status run_resident(RArgs<T> &a, rbgs_ctx *c, ResidentState &r, long nsweeps, int streams, cudaStream_t s) {
    const ResidentPlan &pl = shared_plan<T>(r, a.n, streams);
    const size_t smem = resident_smem<T>(pl.rows, pl.vals, pl.period);
    a.gx = pl.gx, a.gy = pl.gy, a.period = pl.period;
    a.pitch = pl.vals + 2 * pl.period + 2, a.erows = pl.rows + 4 * pl.period;
    a.sweeps = nsweeps;
    a.one = 1.0;
    void *args[] = {&a};
    const cudaError_t e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(resident_kernel<T>),
                                                      dim3(pl.gx * pl.gy), dim3(kRThreads), args, smem, s);
    if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
        cudaGetLastError();
        return kLaunchRefused;
    }
    RBGS_CUDA(e);
    stream_busy(c->device, s, pl.us * (double)nsweeps);
    return RBGS_OK;
}

template <typename T>
RArgs<T> base_args(const rbgs_ctx *c, int W, const ResidentState &r) {
    RArgs<T> a{};
    a.n = c->g.n, a.W = W, a.kmax = (c->g.n + 3) / 2, a.kint = c->g.n / 2 + 1;
    a.slots = r.slots, a.epoch = r.epoch, a.status = c->dstatus;
    return a;
}

}  // namespace

ResidentPlan resident_plan(int n, int kind) {
    const int sms = device_sms();
    return kind == 0 ? plan_for<double>(n, sms) : kind == 1 ? plan_for<float>(n, sms) : plan_for<int64_t>(n, sms);
}

size_t resident_slot_bytes(int n, int W, int kind) { return (size_t)2 * (n + 2) * W * (kind == 1 ? 8 : 16); }

rbgs_status launch_resident_sweeps_f64(rbgs_ctx *c, long nsweeps, int streams, cudaStream_t s) {
    RArgs<double> a = base_args<double>(c, c->g.W, c->res64);
    a.u0 = c->f64.u[0], a.u1 = c->f64.u[1], a.hf0 = c->f64.hf[0], a.hf1 = c->f64.hf[1];
    return run_resident(a, c, c->res64, nsweeps, streams, s);
}

rbgs_status launch_resident_sweeps_fused(rbgs_ctx *c, long nsweeps, int streams, cudaStream_t s) {
    RArgs<int64_t> a = base_args<int64_t>(c, c->g.W, c->res64);
    a.u0 = c->f64.u[0], a.u1 = c->f64.u[1], a.hf0 = c->hq[0], a.hf1 = c->hq[1];
    a.words = c->fwords;
    return run_resident(a, c, c->res64, nsweeps, streams, s);
}

rbgs_status launch_resident_sweeps_f32(rbgs_ctx *c, long nsweeps, int streams, cudaStream_t s) {
    RArgs<float> a = base_args<float>(c, c->f32.W, c->res32);
    a.u0 = c->f32.u[0], a.u1 = c->f32.u[1], a.hf0 = c->f32.hf[0], a.hf1 = c->f32.hf[1];
    return run_resident(a, c, c->res32, nsweeps, streams, s);
}

}  // namespace rbgs
