// Exchange of values between the tiles of the resident kernel (resident.cu) through slots in
// global memory, with bounded waits.
//
// A value travels with its period's number in the same 64-bit word (a 64-bit value as two words,
// a 32-bit value as one), so a reader that finds the number has the value: no fences, no flags,
// one trip through L2.
//
// Every wait is bounded: after `max_polls` polls, or when the status word says that another block
// has given up, the reader sets bit 1 of the status and the whole block leaves.
#pragma once

#include <cstdint>

namespace rbgs {

// 64-bit words per slot
template <typename Bits>
constexpr int kSlotWords = sizeof(Bits) / 4;

__device__ __forceinline__ void slot_put(unsigned long long *slot, uint64_t bits, unsigned seq) {
    const unsigned long long s = (unsigned long long)seq << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(slot), "l"(s | (uint32_t)bits),
                 "l"(s | (uint32_t)(bits >> 32))
                 : "memory");
}
__device__ __forceinline__ void slot_put(unsigned long long *slot, uint32_t bits, unsigned seq) {
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(slot), "l"(((unsigned long long)seq << 32) | bits)
                 : "memory");
}
// true when the slot holds period seq's value, then in `bits`
__device__ __forceinline__ bool slot_get(const unsigned long long *slot, uint64_t &bits, unsigned seq) {
    unsigned long long a, b;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(slot) : "memory");
    bits = (uint64_t)(uint32_t)a | ((uint64_t)(uint32_t)b << 32);
    return (unsigned)(a >> 32) == seq && (unsigned)(b >> 32) == seq;
}
__device__ __forceinline__ bool slot_get(const unsigned long long *slot, uint32_t &bits, unsigned seq) {
    unsigned long long a;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(a) : "l"(slot) : "memory");
    bits = (uint32_t)a;
    return (unsigned)(a >> 32) == seq;
}

// Whether an earlier wait has given up, read once for the whole block: threads that read the
// status each for themselves could part ways when it is set at that moment, some leaving before a
// barrier that the others wait at.  Every thread of the block calls this.
__device__ __forceinline__ bool block_given_up(const int *status) {
    return __syncthreads_or(threadIdx.x == 0 ? *reinterpret_cast<const volatile int *>(status) : 0) != 0;
}

// Receives period seq's value of every entry of list (.x: place in to, .y: slot), THREADS threads
// with four slots each at a time.  False, for the whole block, when a wait gave up.  Ends with a
// block barrier; s_abort (shared) is 0 before the call.
template <typename T, typename Bits, int THREADS>
__device__ __forceinline__ bool receive_slots(T *to, const int2 *list, int count, const unsigned long long *slots,
                                              unsigned seq, int *status, int *s_abort, uint32_t max_polls) {
    for (int base = 0; base < count; base += 4 * THREADS) {
        unsigned pend = 0;
        int2 ent[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int at = base + (int)threadIdx.x + q * THREADS;
            if (at < count) ent[q] = list[at], pend |= 1u << q;
        }
        uint32_t polls = 0;
        while (pend) {
            Bits b[4];
            bool hit[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                hit[q] = ((pend >> q) & 1u) && slot_get(slots + (size_t)ent[q].y * kSlotWords<Bits>, b[q], seq);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (hit[q]) {
                    __builtin_memcpy(&to[ent[q].x], &b[q], sizeof(T));
                    pend &= ~(1u << q);
                }
            }
            if (pend && (++polls >= max_polls ||
                         ((polls & 1023u) == 0 && *reinterpret_cast<volatile int *>(status) != 0))) {
                atomicOr(status, 2);
                *s_abort = 1;
                break;
            }
        }
    }
    __syncthreads();
    return *s_abort == 0;
}

}  // namespace rbgs
