// tcgen05 convolution (forward and data gradient) of 3x3 layers whose weights fit in shared
// memory: each input pixel is staged once per tile, and a tap is an offset of the operand
// descriptor.  Included by conv_umma.cu inside its anonymous namespace.
//
// The gather kernel copies every input value nine times, once per tap, and the TMA kernel loads
// nine boxes; on the layers with 16 to 96 channels those copies, not the MMAs, took the time (77
// to 250 TFLOP/s).  Here the M tile is a patch of 8 x 16 pixels (8 across, 16 rows) of one image,
// and a stage is the patch's slab of 10 x 18 pixels, all channels, loaded once (1.41 input values
// per output pixel).  In shared memory the slab is the K-major layout without swizzle: per group
// of 8 channels a plane of 16-byte rows, one per pixel, row by row of the slab.  Eight pixels in a
// row are one 128-byte core matrix, the next eight rows of the operand are the image row below
// (SBO = 10 pixels = 160 bytes), the next 8 channels are the next plane (LBO), and the tap
// (ty, tx) starts (10 ty + tx) 16-byte rows further on.  The weights sit in shared memory for the
// whole kernel, [K step of 16][channel group][output channel] 16-byte rows.  The K order is that
// of the other kernels (taps, then channels, 16 at a time), so the accumulated bits are too.
//
// Persistent, warp-specialised CTA (one per SM), as conv_umma_kernel: warps 0-7 copy slabs
// (cp.async, zero fill outside the image) into a ring of four stages and arrive on a stage's
// `full` barrier when their copies have landed; warp 8 issues the 9 CK / 16 MMAs of a tile into
// the accumulator of the stage's number and commits them to its `tfull` barrier, which hands the
// accumulator to the epilogue and the stage back to the producers; sixteen warps drain the four
// accumulators, four warps each (on the narrowest layers one tile's drain takes longer than its
// MMAs).  Every wait is bounded as in the other kernels.
//
// What bounds it: the thread that issues the MMAs.  Cycles per tile at 16 x 264^2, forward, by
// clock64 around its steps (the readings add 10 to 20% to the time): 16->32 (9 MMAs) 918 to issue
// and commit, 480 at its two waits, 1692 in all; 32->32 (18) 1636, 490, 2601; 96->32 (54) 3644, 535,
// 5023.  So an MMA takes 102, 91 and 67 cycles for 16 of products (its A operand is 4 KB of shared
// memory without swizzle).  A wait takes about 230 cycles on every layer, so that is a poll with its
// fences and not a wait for others: the producers need 308, 611 and 2321 cycles for a tile's copies
// and wait 692, 703 and 1365, and a drain takes 909 to 2083, four tiles at a time.
// Measured on 16 images of 264 x 264 (us; before: gathers forward, TMA data gradient; in
// brackets: the issuing thread chosen by lane number, see elect_one):
//   forward 16->32 123, now 56 [88]; 32->32 168, now 82 [115]; 96->32 393, now 154 [217]
//   at 132 x 132: 32->64 53, now 31 [41]; 64->64 81, now 39 [54]
//   data gradient 32->32 254, now 105 [117]; 96->32 270, now 187 [180]; at 132 x 132:
//   64->64 158, now 51 [58]; 32->64 154, now 45 [54]
// The TMA kernel with the patches it has now, data gradient: 96->32 287 (1 and 4 images: 29.9 and
// 62.4, here 28.9 and 60.3), 32->32 151; at 132 x 132 64->64 84, 32->64 82.

constexpr int kSlabW = 10, kSlabH = 18;
constexpr uint32_t kPlane = (kSlabW * kSlabH + 1) * 16;  // an odd number of 16-byte rows: 8 groups of a pixel hit 8 banks
constexpr int kSlabAcc = 4;  // accumulators, each with its own four epilogue warps
constexpr int kSlabThreads = kProducers + 32 + kSlabAcc * 128;
constexpr int kSlabMaxCk = 128, kSlabMaxN = 128;
constexpr uint32_t kSlabSmem = 220 * 1024;

struct SArgs {
    const uint16_t *src, *wts;  // forward: X and Wt[o][t][c]; data gradient: G and Wt_t[t][c][o]
    const float *bias;
    void *out;
    const uint16_t *Y;  // data gradient with gin: as in UArgs
    uint16_t *gin;
    int H, W, CK, N;    // CK: channels of src; N: output channels
    int relu, y_fp32, accumulate;
    int tiles_x, tiles_y, num_tiles;
    uint32_t stage_bytes, tmem_cols;
};

// Position of a tile, advanced by a fixed number of tiles at a time without divisions: a role's
// warps have little parallelism of their own, so the instructions of a step are its time (with
// three index divisions and a bounds check per copy, the producers took 2.2 us per tile).
struct SlabTile {
    int b, ty, tx;      // image, patch row, patch column
    int db, dty, dtx;   // the step
    __device__ __forceinline__ SlabTile(const SArgs &a, int tile, int step) {
        tx = tile % a.tiles_x, ty = tile / a.tiles_x % a.tiles_y, b = tile / a.tiles_x / a.tiles_y;
        dtx = step % a.tiles_x, dty = step / a.tiles_x % a.tiles_y, db = step / a.tiles_x / a.tiles_y;
    }
    __device__ __forceinline__ void next(const SArgs &a) {
        tx += dtx;
        const int cx = tx >= a.tiles_x;
        tx -= cx ? a.tiles_x : 0;
        ty += dty + cx;
        const int cy = ty >= a.tiles_y;
        ty -= cy ? a.tiles_y : 0;
        b += db + cy;
    }
};

// PIECES: 16-byte copies per producer thread and slab, at least 180 CK / 8 / 256
template <int MODE, int PIECES>
__global__ void __launch_bounds__(kSlabThreads, 1) conv_slab_kernel(const SArgs a) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kSlabAcc], tfull_bar[kSlabAcc], tempty_bar[kSlabAcc];
    __shared__ uint32_t tmem_slot;
    __shared__ float s_bias[kSlabMaxN];
    __shared__ int abort_word;
    volatile int *abort_flag = &abort_word;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp: uniform
    const int CK = a.CK, N = a.N, G8 = CK >> 3;
    const uint32_t sbase = (smem_addr(smem_raw) + 127u) & ~127u;
    const uint32_t wbase = sbase + (uint32_t)kSlabAcc * a.stage_bytes;

    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(&tmem_slot)),
                     "r"(a.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int b = 0; b < kSlabAcc; ++b) {
            mbar_init(&full_bar[b], kProducers);
            mbar_init(&tfull_bar[b], 1);
            mbar_init(&tempty_bar[b], 4);
        }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (MODE == U_FWD && threadIdx.x < N) s_bias[threadIdx.x] = a.bias ? a.bias[threadIdx.x] : 0.f;
    // the weights: 16 bytes = 8 K values of one output channel; vector v is K group v / N, channel v % N
    for (int v = threadIdx.x; v < 9 * G8 * N; v += kSlabThreads) {
        const int kg = v / N, n = v - kg * N, t = kg / G8, c = (kg - t * G8) * 8;
        const uint16_t *p = MODE == U_FWD ? a.wts + ((long)n * 9 + t) * CK + c : a.wts + ((long)t * N + n) * CK + c;
        cp_async16(wbase + (uint32_t)v * 16u, p, true);
    }
    cp_async_commit();
    cp_async_wait<0>();
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp < kMmaWarp) {
        // this thread's 16-byte pieces of a slab: shared offset, element offset in the image from
        // the slab's origin, slab row and column
        uint32_t soff[PIECES], rc[PIECES];
        int goff[PIECES];
        const int npieces = kSlabW * kSlabH * G8;
#pragma unroll
        for (int q = 0; q < PIECES; ++q) {
            const int v = threadIdx.x + q * kProducers;
            const int pos = v / G8, g = v - pos * G8, r = pos / kSlabW, c = pos - r * kSlabW;
            soff[q] = (uint32_t)g * kPlane + (uint32_t)pos * 16u;
            goff[q] = (r * a.W + c) * CK + g * 8;
            rc[q] = (uint32_t)r << 16 | (uint32_t)c;
        }
        SlabTile T(a, blockIdx.x, gridDim.x);
        int local = 0;
        for (int tile = blockIdx.x; tile < a.num_tiles; tile += gridDim.x, ++local, T.next(a)) {
            const int s = local % kSlabAcc;
            // the stage is free when the MMAs that read it four tiles ago are done: the same event
            // that fills its accumulator, so one commit per tile serves both
            if (!wait_or_abort(&tfull_bar[s], (((uint32_t)local / kSlabAcc) & 1u) ^ 1u, abort_flag)) break;
            const uint32_t dst = sbase + (uint32_t)s * a.stage_bytes;
            const int y0 = T.ty * 16 - 1, x0 = T.tx * 8 - 1;  // the slab's origin
            const uint16_t *origin = a.src + (((long)T.b * a.H + y0) * a.W + x0) * CK;
            if (y0 >= 0 && x0 >= 0 && y0 + kSlabH <= a.H && x0 + kSlabW <= a.W) {
#pragma unroll
                for (int q = 0; q < PIECES; ++q)
                    if ((int)threadIdx.x + q * kProducers < npieces) cp_async16(dst + soff[q], origin + goff[q], true);
            } else {
#pragma unroll
                for (int q = 0; q < PIECES; ++q) {
                    if ((int)threadIdx.x + q * kProducers < npieces) {
                        const bool ok = (unsigned)(y0 + (int)(rc[q] >> 16)) < (unsigned)a.H &&
                                        (unsigned)(x0 + (int)(rc[q] & 0xFFFFu)) < (unsigned)a.W;
                        cp_async16(dst + soff[q], ok ? origin + goff[q] : a.src, ok);
                    }
                }
            }
            // counts this thread's arrival once its copies have landed
            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_addr(&full_bar[s])) : "memory");
        }
        cp_async_wait<0>();
    } else if (warp == kMmaWarp) {
        if (elect_one()) {
            const uint32_t idesc = instr_desc(UM, N, 0, 0);
            const int steps = CK >> 4;
            // descriptor start addresses count 16-byte units, in the low bits: offsets just add
            const uint64_t wdesc = smem_desc(wbase, (uint32_t)N * 16u, 128, 0);
            const uint32_t bstep = (uint32_t)N * 2u, astep = 2u * (kPlane >> 4);
            int local = 0;
            for (int tile = blockIdx.x; tile < a.num_tiles; tile += gridDim.x, ++local) {
                const int buf = local % kSlabAcc;
                const uint32_t ph = ((uint32_t)local / kSlabAcc) & 1u;
                if (!wait_or_abort_spin(&tempty_bar[buf], ph ^ 1u, abort_flag) ||
                    !wait_or_abort_spin(&full_bar[buf], ph, abort_flag))
                    break;
                fence_proxy_async_smem();  // cp.async wrote through the generic proxy
                tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(buf * N);
                const uint64_t adesc = smem_desc(sbase + (uint32_t)buf * a.stage_bytes, kPlane, kSlabW * 16u, 0);
                uint64_t bd = wdesc;
#pragma unroll
                for (int t = 0; t < 9; ++t) {
                    const int ty = MODE == U_FWD ? t / 3 : 2 - t / 3, tx = MODE == U_FWD ? t % 3 : 2 - t % 3;
                    uint64_t ad = adesc + (uint32_t)(ty * kSlabW + tx);
                    for (int k = 0; k < steps; ++k) {
                        umma_bf16(acc, ad, bd, idesc, (t > 0 || k > 0) ? 1u : 0u);
                        ad += astep;
                        bd += bstep;
                    }
                }
                umma_commit(&tfull_bar[buf]);
            }
        }
    } else {
        const int q = warp & 3;                   // TMEM lane quarter
        const int grp = (warp - kEpiWarp0) >> 2;  // this warp's accumulator: tiles local = grp, grp + 4, ..
        const int row = q * 32 + lane;            // operand row: image row row / 8, column row % 8
        const int buf = grp;
        uint32_t ph = 0;
        SlabTile T(a, blockIdx.x + grp * gridDim.x, kSlabAcc * gridDim.x);
        for (int tile = blockIdx.x + grp * gridDim.x; tile < a.num_tiles; tile += kSlabAcc * gridDim.x, T.next(a), ph ^= 1u) {
            const bool ok = wait_or_abort(&tfull_bar[buf], ph, abort_flag);
            if (!__all_sync(0xffffffffu, ok)) break;  // tcgen05.ld below needs every lane of the warp
            tc_fence_after();
            const int y = T.ty * 16 + (row >> 3), x = T.tx * 8 + (row & 7);
            const bool pix = y < a.H && x < a.W;
            const long m = ((long)T.b * a.H + y) * a.W + x;
#pragma unroll 1
            for (int c0 = 0; c0 < N; c0 += 16) {
                uint32_t r[16];
                __syncwarp();
                tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * N + c0), r);
                if (!pix) continue;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int n = c0 + h * 8;
                    const long o = m * N + n;
                    float v[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(r[h * 8 + e]);
                    if (MODE == U_FWD) {
                        if (a.bias) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) v[e] += s_bias[n + e];
                        }
                        if (a.relu) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) v[e] = fmaxf(v[e], 0.f);
                        }
                    }
                    if (MODE == U_FWD && !a.y_fp32) {
                        *reinterpret_cast<uint4 *>(reinterpret_cast<uint16_t *>(a.out) + o) =
                            make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]),
                                       pack_bf16(v[6], v[7]));
                    } else if (MODE == U_BWD_DATA && a.gin) {
                        *reinterpret_cast<uint4 *>(a.gin + o) =
                            masked_bf16(v, __ldg(reinterpret_cast<const uint4 *>(a.Y + o)));
                    } else {
                        float4 *dst = reinterpret_cast<float4 *>(reinterpret_cast<float *>(a.out) + o);
                        float4 p0 = make_float4(v[0], v[1], v[2], v[3]), p1 = make_float4(v[4], v[5], v[6], v[7]);
                        if (MODE == U_BWD_DATA && a.accumulate) {
                            const float4 q0 = dst[0], q1 = dst[1];
                            p0.x += q0.x, p0.y += q0.y, p0.z += q0.z, p0.w += q0.w;
                            p1.x += q1.x, p1.y += q1.y, p1.z += q1.z, p1.w += q1.w;
                        }
                        dst[0] = p0;
                        dst[1] = p1;
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty_bar[buf]);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols)
                     : "memory");
}

template <int MODE, int PIECES>
bool slab_run(const SArgs &a, cudaStream_t s) {
    static PerDevice<cudaError_t> limit;
    if (raise_smem(limit, conv_slab_kernel<MODE, PIECES>, kSlabSmem) != cudaSuccess) return false;
    const int grid = a.num_tiles < sm_count() ? a.num_tiles : sm_count();
    conv_slab_kernel<MODE, PIECES><<<grid, kSlabThreads, kSlabSmem, s>>>(a);
    return true;
}

// Launches the slab kernel when it takes the shape: 3x3, CK and N multiples of 16 (one K step of
// an MMA and one epilogue read), at most 128 (12 pieces per producer; four accumulators in 512
// TMEM columns), the weights and the four stages in shared memory, and element offsets within a
// slab in 32 bits.  It was the faster kernel on every such layer measured (above), so there is no
// further line.  Returns false (nothing launched) otherwise.
template <int MODE>
bool slab_conv_launch(const uint16_t *src, const uint16_t *wts, const float *bias, void *out, const uint16_t *Y,
                      uint16_t *gin, int B, int H, int W, int CK, int N, int ks, int relu, int y_fp32, int accumulate,
                      cudaStream_t s, rbgs_status *st) {
    if (ks != 3 || CK % 16 != 0 || N % 16 != 0 || CK > kSlabMaxCk || N > kSlabMaxN) return false;
    if ((long)kSlabH * W * CK > 0x7fffffffL) return false;
    SArgs a{};
    a.stage_bytes = ((uint32_t)(CK / 8) * kPlane + 127u) & ~127u;
    const uint32_t wbytes = 9u * (uint32_t)CK * (uint32_t)N * 2u;
    if (wbytes + kSlabAcc * a.stage_bytes + 128 > kSlabSmem) return false;
    a.src = src, a.wts = wts, a.bias = bias, a.out = out, a.Y = Y, a.gin = gin;
    a.H = H, a.W = W, a.CK = CK, a.N = N;
    a.relu = relu, a.y_fp32 = y_fp32, a.accumulate = accumulate;
    a.tiles_x = (W + 7) / 8, a.tiles_y = (H + 15) / 16;
    const long tiles = (long)B * a.tiles_x * a.tiles_y;
    if (tiles > 0x7fffffffL - 4096) return false;  // a tile index plus a step of the grid stays in range
    a.num_tiles = (int)tiles;
    uint32_t cols = 32;
    while ((int)cols < kSlabAcc * N) cols <<= 1;
    a.tmem_cols = cols;
    const int need = (kSlabW * kSlabH * (CK / 8) + kProducers - 1) / kProducers;
    const bool ok = need <= 2   ? slab_run<MODE, 2>(a, s)
                    : need <= 3 ? slab_run<MODE, 3>(a, s)
                    : need <= 6 ? slab_run<MODE, 6>(a, s)
                    : need <= 9 ? slab_run<MODE, 9>(a, s)
                                : slab_run<MODE, 12>(a, s);
    if (!ok) {
        set_error("cudaFuncSetAttribute failed for the slab convolution");
        *st = RBGS_ECUDA;
        return true;
    }
    const cudaError_t e = cudaGetLastError();
    *st = RBGS_OK;
    if (e != cudaSuccess) {
        set_error("slab convolution launch failed: %s", cudaGetErrorString(e));
        *st = RBGS_ECUDA;
    }
    return true;
}
