// Reductions over the first nthr threads of a block (whole warps): the bottom
// solves, whose iterations are chains of such sums.
#pragma once

#include "mx_internal.cuh"

// The four sums of one call share their shuffles (each exchange halves what a
// lane still carries: 6 in place of 20) and lane group g = lane / 8 ends with sum
// g; every warp then adds the warps' sums itself, so all threads hold the same
// bits and take the same branches.  The two buffers alternate: a barrier lies
// between a call's reads and the writes of the next but one.
template <typename T>
struct TeamSum {
    T (*red)[4][32];  // two buffers in shared memory
    int nthr, turn = 0;

    __device__ __forceinline__ TeamSum(T (*r)[4][32], int n) : red(r), nthr(n) {}
    // (the form without .aligned: warps may arrive in parts, after a divergent branch)
    __device__ __forceinline__ void barrier() const { asm volatile("barrier.sync 1, %0;" ::"r"(nthr) : "memory"); }
    static __device__ __forceinline__ T group_sum(T k) {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
        return k;
    }
    __device__ __forceinline__ void sum(T (&a)[4]) {
        const int lane = threadIdx.x & 31, nw = nthr >> 5;
        const bool up16 = lane & 16, up8 = lane & 8;
        T k0 = up16 ? a[2] : a[0], k1 = up16 ? a[3] : a[1];
        k0 += __shfl_xor_sync(0xffffffffu, up16 ? a[0] : a[2], 16);
        k1 += __shfl_xor_sync(0xffffffffu, up16 ? a[1] : a[3], 16);
        T k = (up8 ? k1 : k0) + __shfl_xor_sync(0xffffffffu, up8 ? k0 : k1, 8);
        k = group_sum(k);
        if (nw > 1) {
            if ((lane & 7) == 0) red[turn][lane >> 3][threadIdx.x >> 5] = k;
            barrier();
            k = T(0);
            for (int q = lane & 7; q < nw; q += 8) k += red[turn][lane >> 3][q];
            k = group_sum(k);
            turn ^= 1;
        }
#pragma unroll
        for (int m = 0; m < 4; m++) a[m] = __shfl_sync(0xffffffffu, k, 8 * m);
    }
};

// The bottom solves' scalar divisions: they set step lengths, so the fast forms
// (a division subroutine's instructions would cost more than its arithmetic).
__device__ __forceinline__ float sdiv(float a, float b) { return __fdividef(a, b); }
