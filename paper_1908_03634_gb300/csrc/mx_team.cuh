// Reductions over the first nthr threads of a block (whole warps): the bottom
// solves, whose iterations are chains of such sums.
#pragma once

#include "mx_internal.cuh"

// What a team keeps in static shared memory: the partial sums and the mbarrier on
// which one lane of each warp arrives.  (A named barrier counts a warp once for each
// part in which it arrives, and after the sums' divergent branches that is up to the
// compiler.)  The sums are stored and loaded by inline assembly that clobbers memory:
// with plain accesses to the array one build of a bottom solve read the first warp's
// sum and none of the others', whatever the barrier between.  A wait ends after 2^20
// tries at the latest.
template <typename T>
struct TeamShared {
    unsigned long long bar;
    T red[2][4][32];
};

// One thread, before a block barrier and any use: a team of nthr threads.
template <typename T>
__device__ __forceinline__ void team_init(TeamShared<T> &S, int nthr) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(unsigned(__cvta_generic_to_shared(&S.bar))),
                 "r"(nthr >> 5)
                 : "memory");
}

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
    unsigned red, bar;  // shared addresses: two buffers of partial sums, the barrier
    int nthr, turn = 0, phase = 0;

    __device__ __forceinline__ TeamSum(TeamShared<T> &S, int n)
        : red(unsigned(__cvta_generic_to_shared(&S.red[0][0][0]))),
          bar(unsigned(__cvta_generic_to_shared(&S.bar))),
          nthr(n) {}
    __device__ __forceinline__ unsigned slot(int g, int w) const {
        return red + ((turn * 4 + g) * 32 + w) * unsigned(sizeof(T));
    }
    __device__ __forceinline__ void barrier() {
        __syncwarp();
        if ((threadIdx.x & 31) == 0)
            asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(bar) : "memory");
        int ok = 0;
#pragma unroll 1
        for (int spin = 0; !ok && spin < (1 << 20); spin++)
            asm volatile(
                "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                "selp.b32 %0, 1, 0, p;\n\t}"
                : "=r"(ok)
                : "r"(bar), "r"(phase)
                : "memory");
        __syncwarp();
        phase ^= 1;
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
