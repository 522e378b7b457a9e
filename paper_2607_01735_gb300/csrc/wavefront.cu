// Temporally blocked sweeps as a register wavefront: K sweeps (2K half-sweeps of Eq. (1),
// red then black as in Algorithm 1) per pass over memory, while a warp marches down the grid.
// One kernel for three kinds of values:
//   float   the inner sweeps of the mixed-precision refinement;
//   double  the bit-exact FP64 update;
//   int64   the fused FP64 update (rbgs_opts.fma = 1) on the fixed-point grid of its block of
//           sweeps (fused.cu).  Within a block the scale 2^e is fixed, so between half-sweeps
//           a value needs no binary64 form: the next half-sweep reads only T(u) =
//           trunc(u 2^e), and T of an updated point follows from its five-term sum in about
//           14 integer operations (fixed_quarter in fixed64.cuh).  The first pass of a block
//           converts the binary64 values as it loads them (kWfIn), the last one writes the
//           binary64 iterate straight from the sums (kWfLast).
// Each equals the corresponding one-launch-per-colour sweeps bit for bit.
//
// Wavefront.  Half-sweep h (h = 1..2K; odd h red, even h black) of row i needs only the rows
// i-1, i, i+1 that half-sweep h-1 left (the other colour).  At step t a warp applies
// half-sweep h to row t-h+1 for h = 1, 2, ..., 2K in that order, so what half-sweep h-1 has
// just produced is the row below, and its outputs of the two steps before are the row itself
// and the row above.  A level thus carries two rows of one colour; in[h-1] holds them in a
// ring of three register slots (the step loop is unrolled by six, so slots and row parities
// are compile-time constants).  Level 1 reads the black rows of the input; the red rows are
// never read, since level 1 overwrites them.  So a pass that is not the last of its sequence
// moves the black values in and out and h2 f in: 16 bytes per point in FP64 and 8 in FP32,
// over K sweeps.  h2 f of the live rows t-2K+1 .. t+D sits in a ring of 12 (K = 6: 18) rows in
// shared memory, filled by cp.async D rows ahead and read back by the lane that copied it
// (no barrier).  The ring's six-row groups are addressed through one base register each, which
// rotate every six steps, so the unrolled steps address it with constants.
//
// Decomposition.  A warp owns a strip of 32 P values of each colour row (P per lane) and a
// segment of rows.  West/east values cross lanes by shuffle; at the strip's edges they are
// wrong, and the damage moves inward by at most K values of a colour row over the 2K
// half-sweeps, so each strip stores only its middle 32 P - 2H values (H = K rounded up to a
// multiple of P) and neighbouring strips overlap by 2H.  A segment that outputs rows [a, b)
// starts 2K rows above a and runs 2K-1 rows past b.
//
// What bounds it (ncu, fused, K = 3, 8191^2): the integer ALU pipe, 74% busy, 30 warp
// instructions per 32 updates (one launch per colour: 107), DRAM at 3.7 TB/s.  Measured, a
// sweep: fused 16384^2 382 us = 702 GLUP/s (one launch per colour 1021 us, at 0.95 of the HBM
// bandwidth); fused 4095^2 31 us (96), 1500^2 9.9 us (16.2); FP32 K = 4 8192^2 36.8 us = 1825
// GLUP/s (46.7 with the ring of whole rows in registers that also moved the red values).
//
// The Dirichlet ring never changes, and every level meets it.  Its values sit in the ring
// places of the right-hand-side arrays, which no update reads: a level takes the value it has
// loaded from there instead of an update.
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "fixed64.cuh"
#include "fp64.cuh"
#include "per_device.cuh"
#include "sweep_impl.cuh"

namespace rbgs {
namespace {

constexpr int kWfWarps = 4;  // warps per block; each warp is an independent work item
constexpr int kWfThreads = 32 * kWfWarps;
constexpr int kWfAhead = 3;  // rows of h2 f loaded ahead of their first use
constexpr int kWfMinRows = 4;  // rows of a segment at least (2 to 12 measured at 1023^2 fused: 7.2 / 7.2 / 7.9 / 8.5 us for 2 / 4 / 8 / 12)
constexpr int kWfStep = 6;   // unrolled steps: slots repeat every 3, row parities every 2
constexpr int kWfIn = 1;     // int64 only: the input holds binary64 values
constexpr int kWfLast = 2;   // write both colours (int64: as binary64), not only black
constexpr unsigned long long kNoScale = 0x8000000000000000ull;  // fused: no valid scale

template <typename T>
struct WfArgs {
    const T *in;           // input black rows (kWfIn: the bits of binary64 values)
    const T *hf0, *hf1;    // right-hand-side term; on the Dirichlet ring, the ring's values
    T *o0, *o1;            // output iterate
    double *d0, *d1;       // fused, kWfLast: output iterate in binary64
    const unsigned long long *words;  // fused: [2] the block's scale
    int n, W, kmax;        // kmax: values of a colour row holding columns 0..n+1
    int strips, ow, halo;  // strip: values computed 32 P, stored ow, overlap halo per side
    int seg_h, edge_h;     // rows per segment (even): inner strips, the two edge strips
    int edge_items, items; // work items: (edge strip, segment) first, then (inner strip, segment)
    double one;            // 1.0, for the FP64 update's fma form
};

__device__ __forceinline__ float wf_update(float hf, float vn, float vs, float vw, float ve, double) {
    float s = __fadd_rn(hf, vn);
    s = __fadd_rn(s, vs);
    s = __fadd_rn(s, vw);
    s = __fadd_rn(s, ve);
    return __fmul_rn(s, 0.25f);
}

__device__ __forceinline__ double wf_update(double hf, double vn, double vs, double vw, double ve, double one) {
    return update_f64<false>(0, hf, vn, vs, vw, ve, one);
}

// P values at a 16-byte aligned address: from global memory, from shared memory, to global
template <typename T, int P>
__device__ __forceinline__ void wf_ldg(T (&v)[P], const T *p) {
    constexpr int V = 16 / (int)sizeof(T);
#pragma unroll
    for (int q = 0; q < P; q += V) {
        int4 t;  // volatile: issued here, a whole step before its use, not where it is used
        asm volatile("ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(t.x), "=r"(t.y), "=r"(t.z), "=r"(t.w)
                     : "l"(p + q));
        __builtin_memcpy(&v[q], &t, 16);
    }
}

template <typename T, int P>
__device__ __forceinline__ void wf_lds(T (&v)[P], uint32_t addr) {
    constexpr int V = 16 / (int)sizeof(T);
#pragma unroll
    for (int q = 0; q < P; q += V) {
        int4 t;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(t.x), "=r"(t.y), "=r"(t.z), "=r"(t.w)
                     : "r"(addr + q * (uint32_t)sizeof(T)));
        __builtin_memcpy(&v[q], &t, 16);
    }
}

template <typename T, int P>
__device__ __forceinline__ void wf_stg(T *p, const T (&v)[P]) {
    constexpr int V = 16 / (int)sizeof(T);
#pragma unroll
    for (int q = 0; q < P; q += V) {
        int4 t;
        __builtin_memcpy(&t, &v[q], 16);
        *reinterpret_cast<int4 *>(p + q) = t;
    }
}

// cp.async of the lane's P values; valid = false fills zeros without reading
template <typename T, int P>
__device__ __forceinline__ void wf_cp_async(uint32_t dst, const T *src, bool valid) {
    constexpr int V = 16 / (int)sizeof(T);
#pragma unroll
    for (int q = 0; q < P; q += V)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + q * (uint32_t)sizeof(T)),
                     "l"(src + q), "r"(valid ? 16 : 0)
                     : "memory");
}

template <int K>
constexpr int wf_ring_rows() {
    return (2 * K + kWfAhead + kWfStep - 1) / kWfStep * kWfStep;
}

template <typename T, int K, int P>
constexpr size_t wf_smem() {
    return (size_t)kWfWarps * wf_ring_rows<K>() * 2 * 32 * P * sizeof(T);
}

// Resident blocks per SM that the registers are allotted for: 3 (168 registers a thread) for every
// instance but float K = 6 (2: 255).  Spills: none but in float K = 4 (16 to 24 bytes of stack, 20
// to 36 bytes moved each way) and K = 6 (48 to 56 bytes).  Measured at 16384^2 (fused, K = 3): 382 us a
// sweep with 3, 394 with 4, 540 with 5 (spills); at 1500^2, 9.9 and 11.5 us with 3 and 4.
template <typename T, int K>
constexpr int wf_blocks() {
    return std::is_same<T, float>::value && K == 6 ? 2 : 3;
}

template <typename T, int K, int P, int MODE>
__global__ void __launch_bounds__(kWfThreads, wf_blocks<T, K>()) wavefront_kernel(const WfArgs<T> a) {
    constexpr bool FUSED = std::is_same<T, int64_t>::value;
    constexpr bool IN = (MODE & kWfIn) != 0, LAST = (MODE & kWfLast) != 0;
    constexpr int D = kWfAhead, U = kWfStep, R = wf_ring_rows<K>(), G = R / U, H = 2 * K;
    constexpr uint32_t kColour = 32 * P * sizeof(T), kRow = 2 * kColour;  // bytes in shared memory
    static_assert(P * sizeof(T) % 16 == 0, "a lane's values are whole 16-byte vectors");
    extern __shared__ __align__(16) unsigned char wf_shared[];
    const int wid = blockIdx.x * kWfWarps + (threadIdx.x >> 5);
    if (wid >= a.items) return;  // whole warps only
    unsigned long long ew = 0;
    if (FUSED) {
        ew = a.words[2];
        if (ew == kNoScale && !LAST) return;  // no valid scale: only the last pass writes (NaN)
    }
    const int e = ew == kNoScale ? 0 : (int)(long long)ew;
    const int lane = threadIdx.x & 31;
    const int n = a.n, W = a.W;
    const bool edge = wid < a.edge_items;
    const int sides = a.strips > 1 ? 2 : 1, inner = a.strips - sides;
    const int strip = edge ? (wid % sides ? a.strips - 1 : 0) : 1 + (wid - a.edge_items) % inner;
    const int seg = edge ? wid / sides : (wid - a.edge_items) / inner;
    const int seg_h = edge ? a.edge_h : a.seg_h;
    const int ks = strip * a.ow - a.halo;
    const int k0 = ks + lane * P;  // a multiple of P
    const bool kin = k0 >= 0 && k0 < a.kmax;
    unsigned msk0 = 0, msk1 = 0;  // interior columns for row parity offset 0 / 1
#pragma unroll
    for (int q = 0; q < P; ++q) {
        const int j = 2 * (k0 + q);
        if (kin && j >= 1 && j <= n) msk0 |= 1u << q;
        if (kin && j + 1 >= 1 && j + 1 <= n) msk1 |= 1u << q;
    }
    const int olo = max(ks + a.halo, 0), ohi = min(ks + a.halo + a.ow, a.kmax);
    const int row_a = seg * seg_h, row_b = min(row_a + seg_h, n + 2);
    const int t_s = row_a - H;  // even: step t has the parity of its place in the unrolled loop
    const int t_e = min(row_b + H - 2, n + H);

    // lanes outside the grid's columns hold 1 (any finite non-zero value: their results are
    // discarded, and 1.0 keeps the FP64 quarter on its exponent path)
    const T filler = T(1);
    T in[H][3][P];  // in[h-1]: rows of the colour that level h reads
    auto load_in = [&](T (&dst)[P], int r) {
        if (kin && r >= 0 && r <= n + 1) {
            wf_ldg<T, P>(dst, a.in + (size_t)r * W + k0);
        } else {
#pragma unroll
            for (int q = 0; q < P; ++q) dst[q] = filler;
        }
    };
    auto convert = [&](T (&v)[P]) {
        if constexpr (IN) {
#pragma unroll
            for (int q = 0; q < P; ++q) v[q] = to_fixed(bitsd((uint64_t)v[q]), e);
        }
    };
    // shared-memory ring of h2 f: row r lives in slot (r - t_s + H) mod R
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(wf_shared) + (threadIdx.x >> 5) * (R * kRow) +
                           lane * (uint32_t)(P * sizeof(T));
    auto load_f = [&](uint32_t dst, int r) {
        const bool ok = kin && r >= 0 && r <= n + 1;
        const size_t off = ok ? (size_t)r * W + k0 : 0;
        wf_cp_async<T, P>(dst, a.hf0 + off, ok);
        wf_cp_async<T, P>(dst + kColour, a.hf1 + off, ok);
    };
    // rows t_s - 1, t_s, t_s + 1 of the input
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
            for (int q = 0; q < P; ++q) in[h][s][q] = filler;
    load_in(in[0][1], t_s - 1);
    load_in(in[0][2], t_s);
    load_in(in[0][0], t_s + 1);
#pragma unroll
    for (int r = 1; r < H + D; ++r) load_f(sbase + r % R * kRow, t_s - H + r);
    asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll
    for (int g = 0; g < D; ++g) asm volatile("cp.async.commit_group;" ::: "memory");
    convert(in[0][1]);
    convert(in[0][2]);
    uint32_t base_of[G];  // base_of[g]: address of slot 0 for slots 6 g .. 6 g + 5 of this block
#pragma unroll
    for (int g = 0; g < G; ++g) base_of[g] = sbase;

    // Blocks of six steps whose rows and loads all lie inside the grid, on a strip with no
    // boundary column, run without row and column checks.
    const bool full_cols = __all_sync(0xffffffffu, msk0 == (1u << P) - 1 && msk1 == (1u << P) - 1);
    const bool store_vec = k0 >= olo && k0 + P <= ohi;
    auto run_block = [&](int base, auto fast_tag) {
        constexpr bool FAST = decltype(fast_tag)::value;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int t = base + u;
            if (!FAST && t > t_e) break;
            const int lx = (u + H + D) % R;  // ring place of row t + D
            const uint32_t ldst = base_of[lx / U] + lx * kRow;
            if (FAST) {
                const size_t off = (size_t)(t + D) * W + k0;
                wf_cp_async<T, P>(ldst, a.hf0 + off, true);
                wf_cp_async<T, P>(ldst + kColour, a.hf1 + off, true);
            } else {
                load_f(ldst, t + D);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            asm volatile("cp.async.wait_group %0;" ::"n"(D) : "memory");  // h2 f rows up to t are here
            convert(in[0][u % 3]);  // input row t + 1
            const int p = u & 1;  // (row + colour) & 1 of every level's update at this step
            const unsigned msk = p ? msk1 : msk0;
#pragma unroll
            for (int h = 1; h <= H; ++h) {
                const int i = t - h + 1;
                const int c = (h - 1) & 1;  // colour updated by half-sweep h
                const T *up = in[h - 1][(u + 1) % 3], *mid = in[h - 1][(u + 2) % 3], *dn = in[h - 1][u % 3];
                const int fx = (u + H - h + 1) % R;  // ring place of row i
                T f[P], out[P];
                double last[P];
                wf_lds<T, P>(f, base_of[fx / U] + fx * kRow + c * kColour);
                // west/east neighbours at k-1, k (p = 0) or k, k+1 (p = 1)
                const T x = p == 0 ? __shfl_up_sync(0xffffffffu, mid[P - 1], 1)
                                   : __shfl_down_sync(0xffffffffu, mid[0], 1);
                // values that half-sweep h may change; the ring's values wait in h2 f's place
                const unsigned live = FAST ? ~0u : (i >= 1 && i <= n) ? msk : 0u;
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    const T w = p == 0 ? (q ? mid[q ? q - 1 : 0] : x) : mid[q];
                    const T ee = p == 0 ? mid[q] : (q + 1 < P ? mid[q + 1 < P ? q + 1 : 0] : x);
                    if constexpr (FUSED) {
                        const int64_t s = f[q] + up[q] + dn[q] + w + ee;
                        out[q] = fixed_quarter(s);
                        if (LAST && h >= H - 1)
                            last[q] = ew == kNoScale ? __longlong_as_double(0x7FF8000000000000ll)
                                                     : fixed_quarter_to_double(s, e);
                    } else {
                        out[q] = wf_update(f[q], up[q], dn[q], w, ee, a.one);
                    }
                    if (!FAST && !((live >> q) & 1u)) out[q] = (std::is_same<T, double>::value && !kin) ? filler : f[q];
                }
                if (h == 1) {  // level 1 has read row t - 1 for the last time: row t + 2 takes its slot
                    if (FAST)
                        wf_ldg<T, P>(in[0][(u + 1) % 3], a.in + (size_t)(t + 2) * W + k0);
                    else
                        load_in(in[0][(u + 1) % 3], t + 2);
                }
                if (h < H) {
#pragma unroll
                    for (int q = 0; q < P; ++q) in[h < H ? h : 0][u % 3][q] = out[q];
                }
                // rows i of levels 2K (black) and, in the last pass, 2K-1 (red) are final
                if ((h == H || (LAST && h == H - 1)) && i >= row_a && i < row_b) {
                    const size_t off = (size_t)i * W + k0;
                    if constexpr (FUSED && LAST) {
                        double *d = (c ? a.d1 : a.d0) + off;
#pragma unroll
                        for (int q = 0; q < P; ++q)
                            if (((live & msk) >> q & 1u) && k0 + q >= olo && k0 + q < ohi) d[q] = last[q];
                    } else {
                        T *d = (c ? a.o1 : a.o0) + off;
                        if (FAST) {
                            if (store_vec) wf_stg<T, P>(d, out);
                        } else if (kin) {
#pragma unroll
                            for (int q = 0; q < P; ++q)
                                if (k0 + q >= olo && k0 + q < ohi) d[q] = out[q];
                        }
                    }
                }
            }
        }
    };
    int turn = 0;  // six-row groups by which the ring has turned
    for (int base = t_s; base <= t_e; base += U) {
        const bool fast = full_cols && base >= H && base + U - 1 + D <= n + 1 && base + U - 1 <= t_e;
        if (fast)
            run_block(base, std::true_type{});
        else
            run_block(base, std::false_type{});
        turn = turn + 1 == G ? 0 : turn + 1;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int at = g + turn >= G ? g + turn - G : g + turn;  // the group that place g now names
            base_of[g] = sbase + (uint32_t)((at - g) * U) * kRow;
        }
    }
}

int sm_count_wf() {
    static PerDevice<int> sms;
    return sms.get([] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) {
            cudaGetLastError();
            v = 152;
        }
        return v;
    });
}

template <typename T, int K, int P, int MODE>
rbgs_status run_pass(WfArgs<T> &a, int parts, cudaStream_t s) {
    constexpr size_t smem = wf_smem<T, K, P>();
    a.halo = (K + P - 1) / P * P;
    a.ow = 32 * P - 2 * a.halo;
    a.strips = (a.kmax + a.ow - 1) / a.ow;
    static PerDevice<int> resident;  // blocks per SM, per template instance; 0: set-up failed
    const int per_sm = resident.get([] {
        int v = 0;
        if (cudaFuncSetAttribute(wavefront_kernel<T, K, P, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, wavefront_kernel<T, K, P, MODE>, kWfThreads, smem) !=
                cudaSuccess) {
            cudaGetLastError();
            v = 0;
        }
        return v;
    });
    if (per_sm < 1) {
        set_error("wavefront pass: no resident block fits");
        return RBGS_ECUDA;
    }
    const long capacity = (long)per_sm * kWfWarps * sm_count_wf() / parts;
    const long rows = a.n + 2, sides = a.strips > 1 ? 2 : 1, inner = a.strips - sides;
    // One wave of items, all of about the same length.  A step of an edge strip takes longer (its
    // checks), and a wave is as long as its longest item, so edge strips are cut into shorter
    // segments, by a factor between the two costs: 16384^2 fused, factor 1 / 1.7 / 2.2 / 2.8 /
    // 4: 613 / 424 / 395 / 382 / 412 us a sweep; 8192^2 FP32, 1 / 1.5 / 2.5 / 4: 53.4 / 41.5 /
    // 36.8 / 40.2 us.
    // In FP64 the adds take most of a step, and the factor is 1.3 (40 sweeps of depth 2 / 4, ms, by 1 /
    // 1.3 / 1.6 / 2.75: 2047^2 1.98 / 1.98 / 2.12 / 2.27 and 2.35 / 2.43 / 2.43 / 2.57, 3000^2 3.52 / 3.53 /
    // 3.52 / 3.85 and 4.03 / 3.87 / 3.99 / 4.17, 8191^2 20.4 / 20.2 / 20.2 / 20.8 and 23.7 / 22.2 / 22.4 / 23.1).
    constexpr double edge_cost = std::is_same<T, float>::value ? 2.5 : std::is_same<T, double>::value ? 1.3 : 2.75;
    auto even = [&](double h) {
        long v = (long)std::ceil(h);
        v = v < kWfMinRows ? kWfMinRows : v > rows ? rows : v;
        return (v + 1) & ~1L;
    };
    double h = (double)rows * (inner + edge_cost * sides) / capacity;
    long items = 0, edge_items = 0;
    for (;; h += 2.0) {
        a.seg_h = (int)even(h);
        a.edge_h = (int)even(h / edge_cost);
        edge_items = sides * ((rows + a.edge_h - 1) / a.edge_h);
        items = edge_items + inner * ((rows + a.seg_h - 1) / a.seg_h);
        if (items <= capacity || a.edge_h >= rows) break;
    }
    if (items > 0x7fffffffL / 2) {
        set_error("wavefront pass: grid too large");
        return RBGS_EINVAL;
    }
    a.edge_items = (int)edge_items;
    a.items = (int)items;
    const unsigned blocks = (unsigned)((items + kWfWarps - 1) / kWfWarps);
    wavefront_kernel<T, K, P, MODE><<<blocks, kWfThreads, smem, s>>>(a);
    RBGS_LAUNCH_CHECK();
    return RBGS_OK;
}

// nsweeps = (whole passes) k sweeps of fld through its partner buffer; the buffers are
// swapped when the result ends up there.
template <typename T, int K, int P>
rbgs_status run_field(ColourField<T> &fld, long passes, int parts, cudaStream_t s) {
    WfArgs<T> a{};
    a.hf0 = fld.hf[0], a.hf1 = fld.hf[1];
    a.n = fld.n, a.W = fld.W, a.kmax = (fld.n + 3) / 2, a.one = 1.0;
    T *const *buf[2] = {fld.u, fld.alt};
    for (long q = 0; q < passes; ++q) {
        a.in = buf[q & 1][1];
        a.o0 = buf[(q & 1) ^ 1][0], a.o1 = buf[(q & 1) ^ 1][1];
        const rbgs_status st = q + 1 == passes ? run_pass<T, K, P, kWfLast>(a, parts, s)
                                                 : run_pass<T, K, P, 0>(a, parts, s);
        if (st != RBGS_OK) return st;
    }
    if (passes & 1) {
        for (int q = 0; q < 2; ++q) {
            T *t = fld.u[q];
            fld.u[q] = fld.alt[q];
            fld.alt[q] = t;
        }
        fld.maps_ready = false;  // tensor maps of the TMA kernel name the old buffers
    }
    return RBGS_OK;
}

template <int MODE>
rbgs_status run_fused(WfArgs<int64_t> &a, int k, int parts, cudaStream_t s) {
    return k == 2 ? run_pass<int64_t, 2, 2, MODE>(a, parts, s) : run_pass<int64_t, 3, 2, MODE>(a, parts, s);
}

}  // namespace

template <>
rbgs_status launch_wavefront_passes<double>(ColourField<double> &fld, int k, long passes, int parts,
                                            cudaStream_t s) {
    switch (k) {
    case 2: return run_field<double, 2, 2>(fld, passes, parts, s);
    case 4: return run_field<double, 4, 2>(fld, passes, parts, s);
    default: set_error("FP64 wavefront depth must be 2 or 4 (got %d)", k); return RBGS_EINVAL;
    }
}

template <>
rbgs_status launch_wavefront_passes<float>(ColourField<float> &fld, int k, long passes, int parts,
                                           cudaStream_t s) {
    switch (k) {
    case 2: return run_field<float, 2, 4>(fld, passes, parts, s);
    case 4: return run_field<float, 4, 4>(fld, passes, parts, s);
    case 6: return run_field<float, 6, 4>(fld, passes, parts, s);
    default: set_error("FP32 wavefront depth must be 2, 4 or 6 (got %d)", k); return RBGS_EINVAL;
    }
}

// nsweeps fused sweeps (>= kFusedWaveMin) at the scale the last launch_fused_prepare chose.
rbgs_status launch_fused_wave_sweeps(const rbgs_ctx *c, long nsweeps, int parts, cudaStream_t s) {
    WfArgs<int64_t> a{};
    a.hf0 = c->hq[0], a.hf1 = c->hq[1];
    a.d0 = c->f64.u[0], a.d1 = c->f64.u[1];
    a.words = c->fwords;
    a.n = c->g.n, a.W = c->g.W, a.kmax = (c->g.n + 3) / 2;
    // depth 3: at 16384^2 a sweep takes 460 / 382 / 395 us with 2 / 3 / 4, at 4095^2 37 / 31 /
    // 34 us (2 moves more memory, 4 needs more registers and overlap)
    constexpr int depth = 3;
    bool first = true;
    int at = 0;
    while (nsweeps > 0) {
        // no pass of one sweep: 4 = 2 + 2; the first pass reads the binary64 iterate and the
        // last one writes it, so there are at least two
        const int k = nsweeps == 4 || nsweeps == 2 ? 2 : depth;
        a.in = first ? reinterpret_cast<const int64_t *>(c->f64.u[1]) : c->tq[at];
        a.o1 = c->tq[at ^ 1];
        const rbgs_status st = first              ? run_fused<kWfIn>(a, k, parts, s)
                               : k == nsweeps ? run_fused<kWfLast>(a, k, parts, s)
                                              : run_fused<0>(a, k, parts, s);
        if (st != RBGS_OK) return st;
        first = false;
        at ^= 1;
        nsweeps -= k;
    }
    return RBGS_OK;
}

}  // namespace rbgs
