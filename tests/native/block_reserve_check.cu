// rept::block_reserve over a block of 1,024 threads: the reserved ranges follow one another without a gap
// from the counter's old value, also where the block's requests together pass 2^32.  Exit code 0: they do.
#include <cstdint>
#include <cstdio>

#include "rept_common.cuh"

constexpr uint32_t kThreads = 1024;

template <class Sum>
__global__ void reserve(unsigned long long* counter, const uint32_t* want, unsigned long long* got) {
    __shared__ rept::BlockReserve<Sum> part;
    got[threadIdx.x] = rept::block_reserve(part, counter, want[threadIdx.x]);
}

template <class Sum>
int check(uint32_t most) {
    static uint32_t want[kThreads];
    static unsigned long long got[kThreads];
    const unsigned long long start = 12345ull;
    unsigned long long *d_counter, *d_got, end = 0, expect = start;
    uint32_t* d_want;
    for (uint32_t i = 0; i < kThreads; ++i) want[i] = i % 3u ? most - i : i % 2u;
    if (cudaMalloc(&d_counter, 8) || cudaMalloc(&d_got, sizeof got) || cudaMalloc(&d_want, sizeof want)) return 1;
    cudaMemcpy(d_counter, &start, 8, cudaMemcpyHostToDevice);
    cudaMemcpy(d_want, want, sizeof want, cudaMemcpyHostToDevice);
    reserve<Sum><<<1, kThreads>>>(d_counter, d_want, d_got);
    cudaMemcpy(got, d_got, sizeof got, cudaMemcpyDeviceToHost);
    if (cudaMemcpy(&end, d_counter, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    int bad = 0;
    for (uint32_t i = 0; i < kThreads; ++i) {
        bad += got[i] != expect;
        expect += want[i];
    }
    bad += end != expect;
    std::printf("requests up to %u: %d wrong\n", most, bad);
    return bad;
}

int main() {
    return check<uint32_t>(5000u) || check<unsigned long long>(5000u) || check<unsigned long long>(0x01000000u) ||
           check<unsigned long long>(0xFFFFFFFFu);
}
