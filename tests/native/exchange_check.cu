// Test harness for the tile exchange's bounded waits (csrc/tile_exchange.cuh): one block receives
// `count` slots of which the last `missing` are never written.  Test infrastructure only.
#include "../../paper_2607_01735_gb300/csrc/tile_exchange.cuh"

namespace {

constexpr int kThreads = 64;

// out[0]: threads that were told that a wait gave up; out[1]: received values that differ
template <typename T, typename Bits>
__global__ void receive_kernel(unsigned long long *slots, int2 *list, T *to, int count, int missing, unsigned seq,
                               unsigned polls, int *status, int *out) {
    __shared__ int s_abort;
    if (threadIdx.x == 0) s_abort = 0;
    for (int q = threadIdx.x; q < count; q += kThreads) {
        list[q] = make_int2(count - 1 - q, q);
        // an earlier period's value in every slot; this period's in all but the missing ones
        rbgs::slot_put(slots + (size_t)q * rbgs::kSlotWords<Bits>, (Bits)(1000 + q), seq - 2);
        if (q < count - missing) rbgs::slot_put(slots + (size_t)q * rbgs::kSlotWords<Bits>, (Bits)(5 * q), seq);
    }
    __syncthreads();
    const bool ok = rbgs::receive_slots<T, Bits, kThreads>(to, list, count, slots, seq, status, &s_abort, polls);
    if (!ok) atomicAdd(&out[0], 1);
    if (ok)
        for (int q = threadIdx.x; q < count; q += kThreads)
            if (to[count - 1 - q] != (T)(Bits)(5 * q)) atomicAdd(&out[1], 1);
}

// Every thread of the block agrees on the status.  out[0]: threads told to leave
__global__ void entry_kernel(const int *status, int *out) {
    if (rbgs::block_given_up(status)) atomicAdd(&out[0], 1);
}

template <typename T, typename Bits>
int receive(int count, int missing, unsigned seq, unsigned polls, int *host) {
    unsigned char *d = nullptr;
    const size_t words = (size_t)count * rbgs::kSlotWords<Bits> * 8, lists = (size_t)count * sizeof(int2);
    const size_t bytes = 16 + words + lists + (size_t)count * sizeof(T);
    if (cudaMalloc(&d, bytes) != cudaSuccess) return 1;
    cudaMemset(d, 0, bytes);
    int *head = reinterpret_cast<int *>(d);  // [0] status, [1], [2] out
    receive_kernel<T, Bits><<<1, kThreads>>>(reinterpret_cast<unsigned long long *>(d + 16),
                                             reinterpret_cast<int2 *>(d + 16 + words),
                                             reinterpret_cast<T *>(d + 16 + words + lists), count, missing, seq, polls,
                                             head, head + 1);
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(host, head, 3 * sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? 0 : 2;
}

}  // namespace

// host[0]: the status word, host[1]: threads that left, host[2]: wrong values.
extern "C" int run_receive_check(int bits, int count, int missing, unsigned seq, unsigned polls, int *host) {
    return bits == 64 ? receive<long long, uint64_t>(count, missing, seq, polls, host)
                      : receive<unsigned, uint32_t>(count, missing, seq, polls, host);
}

extern "C" int run_entry_check(int status, int threads, int *host) {
    int *d = nullptr;
    if (cudaMalloc(&d, 2 * sizeof(int)) != cudaSuccess) return 1;
    const int h[2] = {status, 0};
    cudaMemcpy(d, h, sizeof h, cudaMemcpyHostToDevice);
    entry_kernel<<<1, threads>>>(d, d + 1);
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(host, d + 1, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? 0 : 2;
}
