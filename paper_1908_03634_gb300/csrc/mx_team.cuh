// Reductions over the first nthr threads of a block (whole warps): the bottom
// solves, whose iterations are chains of such sums.
#pragma once

#include "mx_internal.cuh"

// A team's partial sums.  All that its threads exchange between barriers, the vectors
// of the solves too, goes through team_put and team_get, whose order against the barrier
// is fixed in the source: with plain accesses to the static array a build of an
// earlier solve read the first warp's sum and none of the others', for a reason
// that was not found.
template <typename T>
struct TeamShared {
    T red[2][4][32];
};

__device__ __forceinline__ void team_put(unsigned a, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void team_put(unsigned a, double v) {
    asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ float team_get(unsigned a, float) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ double team_get(unsigned a, double) {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}

// The four sums of one call share their shuffles (each exchange halves what a
// lane still carries: 6 in place of 20) and lane group g = lane / 8 ends with sum
// g; every warp then adds the warps' sums itself, so all threads hold the same
// bits and take the same branches.  The two buffers alternate: a barrier lies
// between a call's reads and the writes of the next but one.
template <typename T>
struct TeamSum {
    unsigned red;  // shared address of the two buffers of partial sums
    int nthr, turn = 0;

    __device__ __forceinline__ TeamSum(TeamShared<T> &S, int n)
        : red(unsigned(__cvta_generic_to_shared(&S.red[0][0][0]))), nthr(n) {}
    __device__ __forceinline__ unsigned slot(int g, int w) const {
        return red + ((turn * 4 + g) * 32 + w) * unsigned(sizeof(T));
    }
    // named barrier 1 of nthr threads, in the form that does not need a warp's threads
    // to arrive together
    __device__ __forceinline__ void barrier() {
        __syncwarp();
        asm volatile("barrier.sync 1, %0;" ::"r"(nthr) : "memory");
    }
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
            if ((lane & 7) == 0) team_put(slot(lane >> 3, threadIdx.x >> 5), k);
            barrier();
            k = T(0);
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int w = (lane & 7) + 8 * q;
                const T v = team_get(slot(lane >> 3, w), T(0));
                k += w < nw ? v : T(0);
            }
            k = group_sum(k);
            turn ^= 1;
        }
#pragma unroll
        for (int m = 0; m < 4; m++) a[m] = __shfl_sync(0xffffffffu, k, 8 * m);
    }
};

// Denominators of a bottom solve on vectors of norm 1 to 2 below this count as a
// breakdown; it keeps the divisions by them in the fast form's range.
#define BREAKDOWN 1e-30

// The bottom solves' scalar divisions: they set step lengths, so FP32 takes the fast
// form (a division subroutine's instructions would cost more than its arithmetic);
// FP64 solves divide in FP64.
__device__ __forceinline__ float sdiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double sdiv(double a, double b) { return a / b; }
