// Every argument of the quotients of csrc/fdiv.cuh against the IEEE division:
// prints the number of arguments tried and of differing results, per quotient.
#include <cstdio>

#include "fdiv.cuh"

__global__ void check(int which, unsigned lo, unsigned hi, unsigned long long *bad) {
    unsigned long long n = 0;
    for (unsigned long long b = lo + blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; b < hi;
         b += (unsigned long long)gridDim.x * blockDim.x) {
        const float x = __uint_as_float((unsigned)b);
        float got, want;
        if (which == 0) {
            got = tsx::div_tanh(x);
            want = __fdiv_rn(x, __fadd_rn(x, 2.0f));
        } else if (which == 1) {
            got = tsx::div_atanh(x);
            want = __fdiv_rn(__fadd_rn(1.0f, x), __fsub_rn(1.0f, x));
        } else {
            got = tsx::div_log(x);
            want = __fdiv_rn(__fsub_rn(x, 1.0f), __fadd_rn(x, 1.0f));
        }
        n += __float_as_uint(got) != __float_as_uint(want);
    }
    if (n) atomicAdd(bad, n);
}

int main() {
    const unsigned lo[4] = {0u, 0x21800000u, 0x3E800000u, 0x3F3504F3u};  // 0, 2^-60, 1/4, sqrt(1/2)
    const unsigned hi[4] = {1u, 0x4C800000u, 0x3F800000u, 0x3FB504F4u};  // (0 alone), 2^26, 1, above sqrt(2)
    const int which[4] = {0, 0, 1, 2};
    unsigned long long *bad, h;
    if (cudaMalloc(&bad, 8) != cudaSuccess) return 1;
    for (int i = 0; i < 4; i++) {
        cudaMemset(bad, 0, 8);
        check<<<1216, 256>>>(which[i], lo[i], hi[i], bad);
        if (cudaMemcpy(&h, bad, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
        printf("%d %u %llu\n", which[i], hi[i] - lo[i], h);
    }
    return 0;
}
