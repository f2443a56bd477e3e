// The coarse end of the V-cycle in one launch: the small levels, from the first
// one that fits down to the bottom solve and back up, with corrections and
// right-hand sides in shared memory and face coefficients in registers.  On
// these levels a grid-wide launch does a few microseconds of work, so one launch
// replaces the dozens of per-level launches (smoothing, restriction, BiCGStab
// bottom solve, prolongation) that would otherwise dominate.
//
// The kernel is a thread-block cluster.  A level of more than `dist_min` cells
// is cut along z: each CTA owns a run of plane pairs (so a coarse cell's eight
// children have one owner) and keeps a plane of the neighbours' values on either
// side; the owner of a boundary cell stores its update into the neighbour's copy
// through distributed shared memory, and a cluster barrier ends each colour
// pass.  Smaller levels run on CTA 0 with block barriers while the other CTAs
// wait at the next cluster barrier.  The work is latency: a colour pass is six
// shared loads and a division per cell between two barriers, so the cells'
// coefficients and neighbour indices are set up once per level visit and the
// passes touch shared memory only.
#include <algorithm>
#include <cstring>

#include "mx_coarse.cuh"
#include "mx_rbgs.cuh"
#include "mx_stencil.cuh"

constexpr int CT = 512;          // threads per CTA
constexpr int BOT_REGS = 3;      // bottom solves of up to BOT_REGS * CT cells keep their vectors in registers
constexpr int COARSE_NC = 16;    // CTAs of the cluster (8 where the device cannot place 16)

// cells per thread of the widest level a CTA may own
template <typename T>
struct CoarseCpt {
    static constexpr int value = sizeof(T) == sizeof(float) ? 8 : 4;
};
// levels above this many cells are spread over the cluster (below it one CTA's
// pass is shorter than a cluster barrier)
template <typename T>
constexpr int dist_min() {
    return sizeof(T) == sizeof(float) ? 4096 : 512;
}

// Exact division of x < 2^16 by d < 2^16 as a multiply-high with the
// precomputed m = ceil(2^32 / d) (the error x (m - 2^32/d) / 2^32 stays below
// 1/d, so the floor is exact).
struct FastDiv {
    unsigned d, m;
};
inline FastDiv fast_div(unsigned d) { return FastDiv{d, unsigned(((1ull << 32) + d - 1) / d)}; }
__device__ __forceinline__ int fdiv(int x, FastDiv f) { return f.d == 1 ? x : int(__umulhi(unsigned(x), f.m)); }

// One level of the coarse end.  Shared-memory offsets are in elements and equal
// in every CTA; the correction holds pp + 2 planes (a neighbour's plane first and
// last), the right-hand side pp planes.
template <typename T>
struct CoarseLevel {
    Level<T> L;
    FastDiv d0, d1, dh;  // n0, n1, n0 / 2
    int dist;            // spread over the cluster
    int pp;              // planes per CTA (even where dist)
    int eoff, foff;
};

template <typename T>
struct CoarseArgs {
    int nl;  // number of levels handled (the last is the bottom)
    CoarseLevel<T> lev[COARSE_MAX_LEVELS];
    int nu1, nu2, bot_iters, singular;
    int nc;    // CTAs
    int roff;  // scratch: the residuals of a level, then the bottom solve's vectors
    int total; // elements of shared memory
};

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_addr(const void *p, int rank) {
    unsigned a = unsigned(__cvta_generic_to_shared(p)), r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void remote_store(float *p, int rank, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_addr(p, rank)), "f"(v) : "memory");
}
__device__ __forceinline__ void remote_store(double *p, int rank, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cluster_addr(p, rank)), "d"(v) : "memory");
}
__device__ __forceinline__ float remote_load(const float *p, int rank) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr(p, rank)) : "memory");
    return v;
}
__device__ __forceinline__ double remote_load(const double *p, int rank) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(cluster_addr(p, rank)) : "memory");
    return v;
}
__device__ __forceinline__ void level_sync(int dist) {
    if (dist) cluster_sync();
    else __syncthreads();
}

// The part of a level a CTA owns, and where its boundary planes are copied to.
struct Slab {
    int k0, np;          // first plane, planes
    int dn, up;          // ranks holding copies of the first / last plane (-1: none)
    int dn_plane;        // plane of dn's buffer that copies this CTA's first plane
    int dist;
};

template <typename T>
__device__ __forceinline__ Slab slab_of(const CoarseLevel<T> &C, int rank) {
    Slab s;
    const int nz = C.L.g.n[2];
    const bool per = gper(C.L.g, 2);
    s.dist = C.dist;
    s.k0 = rank * C.pp;
    s.np = max(0, min(C.pp, nz - s.k0));
    const int last = (nz - 1) / C.pp;
    const bool first_here = rank == 0, last_here = rank == last;
    s.dn = first_here ? (per ? last : -1) : rank - 1;
    s.up = last_here ? (per ? 0 : -1) : rank + 1;
    s.dn_plane = (s.dn == last ? nz - last * C.pp : C.pp) + 1;
    return s;
}

// The cells of one thread: coefficients, own index and neighbour indices in the
// shared correction.  Slots [0, CPT/2) hold red cells, the rest black ones.
template <typename T, int CPT>
struct Cells {
    T b[CPT][6];
    T inv[CPT];            // FP64: 1 / sum of b
    unsigned xn[CPT];      // x neighbours (low half: i - 1)
    unsigned yn[CPT];      // y neighbours
    int at[CPT];           // own index; -1: no cell
};

// the 6 face coefficients of in-box cell (i,j,k) = c with 32-bit indexing (the
// same values as face_coefs)
template <typename T>
__device__ __forceinline__ void coefs32(const Level<T> &L, int i, int j, int k, int c, T b[6]) {
    const DGeom &g = L.g;
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxy = nx * ny;
    const bool px = gper(g, 0), py = gper(g, 1), pz = gper(g, 2);
    b[0] = L.bx[c];
    b[1] = (i + 1 < nx) ? L.bx[c + 1] : (px ? L.bx[c - (nx - 1)] : L.hx[j + ny * k]);
    b[2] = L.by[c];
    b[3] = (j + 1 < ny) ? L.by[c + nx] : (py ? L.by[c - (ny - 1) * nx] : L.hy[i + nx * k]);
    b[4] = L.bz[c];
    b[5] = (k + 1 < nz) ? L.bz[c + nxy] : (pz ? L.bz[c - (nz - 1) * nxy] : L.hz[i + nx * j]);
}

// Index 0 of the shared array holds 0: the neighbour beyond a non-periodic face.
template <typename T, int CPT>
__device__ __forceinline__ void load_cells(const CoarseLevel<T> &C, const Slab &s, Cells<T, CPT> &R) {
    const DGeom &g = C.L.g;
    const int nx = g.n[0], ny = g.n[1], nxy = nx * ny, half = (nxy * s.np) >> 1;
    const bool px = gper(g, 0), py = gper(g, 1);
#pragma unroll
    for (int q = 0; q < CPT; q++) {
        const int colour = q >= CPT / 2;
        const int m = threadIdx.x + CT * (q % (CPT / 2));
        R.at[q] = -1;
        if (m < half) {
            const int r = fdiv(m, C.dh);  // row j + n1 p
            const int p = fdiv(r, C.d1);
            const int j = r - p * ny, k = s.k0 + p;
            const int i = 2 * (m - r * int(C.dh.d)) + ((j + k + colour) & 1);
            coefs32(C.L, i, j, k, i + nx * (j + ny * k), R.b[q]);
            const int a = C.eoff + nxy + i + nx * r;
            R.at[q] = a;
            const int xl = i > 0 ? a - 1 : (px ? a + nx - 1 : 0), xh = i + 1 < nx ? a + 1 : (px ? a - (nx - 1) : 0);
            const int yl = j > 0 ? a - nx : (py ? a + (ny - 1) * nx : 0);
            const int yh = j + 1 < ny ? a + nx : (py ? a - (ny - 1) * nx : 0);
            R.xn[q] = unsigned(xl) | (unsigned(xh) << 16);
            R.yn[q] = unsigned(yl) | (unsigned(yh) << 16);
            if (sizeof(T) == sizeof(double)) {
                const T *b = R.b[q];
                R.inv[q] = T(1) / ((b[0] + b[1]) + (b[2] + b[3]) + (b[4] + b[5]));
            }
        }
    }
}

template <typename T, int CPT>
__device__ __forceinline__ void neighbours(const T *sm, const Cells<T, CPT> &R, int q, int nxy, T v[6]) {
    v[0] = sm[R.xn[q] & 0xffffu];
    v[1] = sm[R.xn[q] >> 16];
    v[2] = sm[R.yn[q] & 0xffffu];
    v[3] = sm[R.yn[q] >> 16];
    v[4] = sm[R.at[q] - nxy];
    v[5] = sm[R.at[q] + nxy];
}

// store cell `a`'s new value, and into the copies of it
template <typename T>
__device__ __forceinline__ void put(T *sm, int eoff, const Slab &s, int nxy, int a, T v) {
    sm[a] = v;
    const int ji = a - eoff - nxy;  // index within the slab
    if (ji < nxy && s.dn >= 0) {
        T *t = sm + eoff + s.dn_plane * nxy + ji;
        if (s.dist) remote_store(t, s.dn, v);
        else *t = v;
    }
    if (ji >= (s.np - 1) * nxy && s.up >= 0) {
        T *t = sm + eoff + ji - (s.np - 1) * nxy;
        if (s.dist) remote_store(t, s.up, v);
        else *t = v;
    }
}

// FP32: the same rounded operations as gs_update (bit for bit); FP64: the
// division as a product with the reciprocal taken once per level visit.
__device__ __forceinline__ float cell_update(const float b[6], const float v[6], float f, float h2, float) {
    return gs_update(b, v, f, h2);
}
__device__ __forceinline__ double cell_update(const double b[6], const double v[6], double f, double h2, double inv) {
    double num = b[0] * v[0];
    for (int q = 1; q < 6; q++) num = fma(b[q], v[q], num);
    return fma(-h2, f, num) * inv;
}

template <typename T, int CPT>
__device__ __forceinline__ void sweeps(T *sm, const CoarseLevel<T> &C, const Slab &s, const Cells<T, CPT> &R, int nu) {
    const int nxy = int(C.L.g.nxy), df = C.foff - C.eoff - nxy;
    const T h2 = T(C.L.g.h * C.L.g.h);
    for (int w = 0; w < nu; w++) {
#pragma unroll
        for (int colour = 0; colour < 2; colour++) {
            T e[CPT / 2];
#pragma unroll
            for (int h = 0; h < CPT / 2; h++) {
                const int q = colour * (CPT / 2) + h;
                if (R.at[q] >= 0) {
                    T v[6];
                    neighbours(sm, R, q, nxy, v);
                    e[h] = cell_update(R.b[q], v, sm[R.at[q] + df], h2, R.inv[q]);
                }
            }
#pragma unroll
            for (int h = 0; h < CPT / 2; h++) {
                const int q = colour * (CPT / 2) + h;
                if (R.at[q] >= 0) put(sm, C.eoff, s, nxy, R.at[q], e[h]);
            }
            level_sync(s.dist);
        }
    }
}

// residual of level C restricted to the right-hand side of F, the next one
template <typename T, int CPT>
__device__ __forceinline__ void restrict_down(T *sm, const CoarseArgs<T> &A, const CoarseLevel<T> &C,
                                              const CoarseLevel<T> &F, const Slab &s, const Cells<T, CPT> &R) {
    const int nx = C.L.g.n[0], nxy = int(C.L.g.nxy), df = C.foff - C.eoff - nxy;
    const T ih2 = T(1) / T(C.L.g.h * C.L.g.h);
    T *rs = sm + A.roff;
#pragma unroll
    for (int q = 0; q < CPT; q++)
        if (R.at[q] >= 0) {
            T v[6];
            neighbours(sm, R, q, nxy, v);
            rs[R.at[q] - C.eoff - nxy] = sm[R.at[q] + df] - flux_sum(R.b[q], v, sm[R.at[q]]) * ih2;
        }
    __syncthreads();
    const int mx = nx >> 1, mxy = nxy >> 2, nown = (nxy * s.np) >> 3;
    for (int t = threadIdx.x; t < nown; t += CT) {
        const int r = fdiv(t, F.d0);
        const int P = fdiv(r, F.d1);
        const int I = t - r * mx, J = r - P * int(F.d1.d), K = (s.k0 >> 1) + P;
        const T *c = rs + 2 * I + nx * (2 * J) + nxy * (2 * P);
        T sum = T(0);
        for (int dk = 0; dk < 2; dk++)
            for (int dj = 0; dj < 2; dj++)
                for (int di = 0; di < 2; di++) sum += c[di + nx * dj + nxy * dk];
        const int owner = F.dist ? K / F.pp : 0;
        T *dst = sm + F.foff + I + mx * J + mxy * (K - owner * F.pp);
        if (s.dist) remote_store(dst, owner, sum * T(0.125));
        else *dst = sum * T(0.125);
    }
    level_sync(s.dist);
}

// e += the parents' corrections
template <typename T, int CPT>
__device__ __forceinline__ void prolong_up(T *sm, const CoarseLevel<T> &C, const CoarseLevel<T> &F, const Slab &s,
                                           const Cells<T, CPT> &R) {
    const int nx = C.L.g.n[0], nxy = int(C.L.g.nxy), mx = nx >> 1, mxy = nxy >> 2;
#pragma unroll
    for (int q = 0; q < CPT; q++)
        if (R.at[q] >= 0) {
            const int r = fdiv(R.at[q] - C.eoff - nxy, C.d0);
            const int p = fdiv(r, C.d1);
            const int i = R.at[q] - C.eoff - nxy - r * nx, j = r - p * int(C.d1.d), K = (s.k0 + p) >> 1;
            const int owner = F.dist ? K / F.pp : 0;
            const T *src = sm + F.eoff + mxy + (i >> 1) + mx * (j >> 1) + mxy * (K - owner * F.pp);
            const T ec = s.dist ? remote_load(src, owner) : *src;
            put(sm, C.eoff, s, nxy, R.at[q], sm[R.at[q]] + ec);
        }
    level_sync(s.dist);
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// BiCGStab on a bottom level of at most 32 cells by one warp: one cell per
// lane, dot products by shuffles, the operator's neighbour values through a
// shared-memory vector; no block barriers.
template <typename T>
__device__ void warp_bicgstab(const Level<T> &L, T *x, const T *f, T *pv, int iters, int singular, T ih2) {
    const int n = int(L.g.N), lane = threadIdx.x;
    const bool act = lane < n;
    int i = 0, j = 0, k = 0;
    T b[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
    if (act) {
        i = lane % L.g.n[0];
        const int r = lane / L.g.n[0];
        j = r % L.g.n[1];
        k = r / L.g.n[1];
        face_coefs(L, i, j, k, lane, b);
    }
    auto apply = [&](T val) -> T {  // (L val)_lane, values exchanged through pv
        if (act) pv[lane] = val;
        __syncwarp();
        T y = T(0);
        if (act) {
            T v[6];
            nb_vals(L.g, (const T *)pv, i, j, k, lane, v);
            y = flux_sum(b, v, val) * ih2;
        }
        __syncwarp();
        return y;
    };
    T rhs = act ? f[lane] : T(0);
    if (singular) rhs -= warp_sum(rhs) / T(n);
    if (!act) rhs = T(0);
    T xv = T(0), r = rhs, r0 = rhs, p = T(0), v = T(0);
    const T bnorm2 = warp_sum(rhs * rhs);
    if (bnorm2 > T(0)) {
        const T tol2 = bnorm2 * T(1e-8);
        T rho = T(1), alpha = T(1), omega = T(1);
        for (int it = 0; it < iters; it++) {
            const T rho1 = warp_sum(r0 * r);
            if (rho1 == T(0) || omega == T(0)) break;
            const T beta = (rho1 / rho) * (alpha / omega);
            p = r + beta * (p - omega * v);
            v = apply(p);
            const T r0v = warp_sum(r0 * v);
            if (r0v == T(0)) break;
            alpha = rho1 / r0v;
            const T sv = r - alpha * v;
            if (warp_sum(sv * sv) <= tol2) {
                xv += alpha * p;
                break;
            }
            const T tv = apply(sv);
            const T tt = warp_sum(tv * tv), ts = warp_sum(tv * sv);
            omega = tt > T(0) ? ts / tt : T(0);
            xv += alpha * p + omega * sv;
            r = sv - omega * tv;
            rho = rho1;
            if (warp_sum(r * r) <= tol2) break;
        }
    }
    if (!act) xv = T(0);
    if (singular) xv -= warp_sum(xv) / T(n);
    if (act) x[lane] = xv;
}

// Sums of three values over the first nthr threads of the block (whole warps),
// in every one of them: warp shuffles, then each warp adds the warps' sums
// itself.  The two buffers alternate, so one barrier separates the writes of a
// reduction from those of the next but one.
template <typename T>
__device__ __forceinline__ void team_sum3(T &a, T &b, T &c, T (*red)[3][32], int &turn, int nthr) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = nthr >> 5;
    a = warp_sum(a);
    b = warp_sum(b);
    c = warp_sum(c);
    T(*buf)[32] = red[turn];
    turn ^= 1;
    if (lane == 0) {
        buf[0][w] = a;
        buf[1][w] = b;
        buf[2][w] = c;
    }
    asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
    a = lane < nw ? buf[0][lane] : T(0);
    b = lane < nw ? buf[1][lane] : T(0);
    c = lane < nw ? buf[2][lane] : T(0);
    for (int o = 8; o > 0; o >>= 1) {  // nw <= 16
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    a = __shfl_sync(0xffffffffu, a, 0);
    b = __shfl_sync(0xffffffffu, b, 0);
    c = __shfl_sync(0xffffffffu, c, 0);
}

// BiCGStab on L x = f (x starts at 0), projected onto mean-free vectors when
// the problem is singular; stops at relative residual 1e-4 or `iters`.  Each of
// nthr threads holds up to B cells (cell t + q nthr): their coefficients and all
// vectors stay in registers, the two vectors the operator is applied to pass
// through shared memory (element n holds 0 for faces without a neighbour), and
// the reductions that one step needs are taken together: five barriers per
// iteration.
template <typename T, int B>
__device__ void team_bicgstab(const Level<T> &L, T *x, const T *f, T *scr, int iters, int singular, T ih2, int nthr) {
    __shared__ T red[2][3][32];
    const int n = int(L.g.N), nx = L.g.n[0], ny = L.g.n[1], nz = L.g.n[2], nxy = nx * ny;
    const bool px = gper(L.g, 0), py = gper(L.g, 1), pz = gper(L.g, 2);
    T *pe = scr, *se = scr + n + 1;
    int turn = 0;
    T b[B][6], xv[B], r[B], r0[B], p[B], v[B], sv[B], tv[B];
    unsigned nb[B][3];
    T z0 = T(0), z1 = T(0), sum = T(0);
    if (threadIdx.x == 0) pe[n] = se[n] = T(0);
#pragma unroll
    for (int q = 0; q < B; q++) {
        const int c = threadIdx.x + q * nthr;
        xv[q] = r[q] = p[q] = v[q] = sv[q] = tv[q] = T(0);
        for (int d = 0; d < 6; d++) b[q][d] = T(0);
        nb[q][0] = nb[q][1] = nb[q][2] = unsigned(n) | (unsigned(n) << 16);
        if (c < n) {
            const int i = c % nx, rr = c / nx, j = rr % ny, k = rr / ny;
            coefs32(L, i, j, k, c, b[q]);
            const int xl = i > 0 ? c - 1 : (px ? c + nx - 1 : n), xh = i + 1 < nx ? c + 1 : (px ? c - (nx - 1) : n);
            const int yl = j > 0 ? c - nx : (py ? c + (ny - 1) * nx : n), yh = j + 1 < ny ? c + nx : (py ? c - (ny - 1) * nx : n);
            const int zl = k > 0 ? c - nxy : (pz ? c + (nz - 1) * nxy : n), zh = k + 1 < nz ? c + nxy : (pz ? c - (nz - 1) * nxy : n);
            nb[q][0] = unsigned(xl) | (unsigned(xh) << 16);
            nb[q][1] = unsigned(yl) | (unsigned(yh) << 16);
            nb[q][2] = unsigned(zl) | (unsigned(zh) << 16);
            r[q] = f[c];
            sum += r[q];
        }
    }
    auto apply = [&](const T *e, const T(&own)[B], T(&y)[B]) {
#pragma unroll
        for (int q = 0; q < B; q++) {
            T w[6];
            for (int d = 0; d < 3; d++) {
                w[2 * d] = e[nb[q][d] & 0xffffu];
                w[2 * d + 1] = e[nb[q][d] >> 16];
            }
            y[q] = flux_sum(b[q], w, own[q]) * ih2;
        }
    };
    auto share = [&](T *e, const T(&own)[B]) {
#pragma unroll
        for (int q = 0; q < B; q++)
            if (threadIdx.x + q * nthr < n) e[threadIdx.x + q * nthr] = own[q];
        asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
    };
    if (singular) {
        team_sum3(sum, z0, z1, red, turn, nthr);
        const T mean = sum / T(n);
#pragma unroll
        for (int q = 0; q < B; q++)
            if (threadIdx.x + q * nthr < n) r[q] -= mean;
    }
    T rho1 = T(0);
#pragma unroll
    for (int q = 0; q < B; q++) {
        r0[q] = r[q];
        rho1 += r[q] * r[q];
    }
    z0 = z1 = T(0);
    team_sum3(rho1, z0, z1, red, turn, nthr);
    const T bnorm2 = rho1;
    if (bnorm2 > T(0)) {
        const T tol2 = bnorm2 * T(1e-8);  // 1e-4 relative: ample for a multigrid bottom solve
        T rho = T(1), alpha = T(1), omega = T(1);
        for (int it = 0; it < iters; it++) {
            if (rho1 == T(0) || omega == T(0)) break;
            const T beta = (rho1 / rho) * (alpha / omega);
#pragma unroll
            for (int q = 0; q < B; q++) p[q] = r[q] + beta * (p[q] - omega * v[q]);
            share(pe, p);
            apply(pe, p, v);
            T r0v = T(0);
#pragma unroll
            for (int q = 0; q < B; q++) r0v += r0[q] * v[q];
            z0 = z1 = T(0);
            team_sum3(r0v, z0, z1, red, turn, nthr);
            if (r0v == T(0)) break;
            alpha = rho1 / r0v;
#pragma unroll
            for (int q = 0; q < B; q++) sv[q] = r[q] - alpha * v[q];
            share(se, sv);
            apply(se, sv, tv);
            T ss = T(0), tt = T(0), ts = T(0);
#pragma unroll
            for (int q = 0; q < B; q++) {
                ss += sv[q] * sv[q];
                tt += tv[q] * tv[q];
                ts += tv[q] * sv[q];
            }
            team_sum3(ss, tt, ts, red, turn, nthr);
            if (ss <= tol2) {
#pragma unroll
                for (int q = 0; q < B; q++) xv[q] += alpha * p[q];
                break;
            }
            omega = tt > T(0) ? ts / tt : T(0);
            T rr = T(0), rn = T(0);
#pragma unroll
            for (int q = 0; q < B; q++) {
                xv[q] += alpha * p[q] + omega * sv[q];
                r[q] = sv[q] - omega * tv[q];
                rr += r[q] * r[q];
                rn += r0[q] * r[q];
            }
            rho = rho1;
            z0 = T(0);
            team_sum3(rr, rn, z0, red, turn, nthr);
            if (rr <= tol2) break;
            rho1 = rn;
        }
    }
    if (singular) {
        sum = T(0);
#pragma unroll
        for (int q = 0; q < B; q++) sum += xv[q];
        z0 = z1 = T(0);
        team_sum3(sum, z0, z1, red, turn, nthr);
        const T mean = sum / T(n);
#pragma unroll
        for (int q = 0; q < B; q++) xv[q] -= mean;
    }
#pragma unroll
    for (int q = 0; q < B; q++)
        if (threadIdx.x + q * nthr < n) x[threadIdx.x + q * nthr] = xv[q];
}

// dot product accumulated in T (FP32 on the mixed path: the bottom solve only
// needs a 1e-4 reduction, and FP64 is slow on this part)
template <typename T>
__device__ T cta_dot(const T *a, const T *b, int n) {
    T s = T(0);
    for (int q = threadIdx.x; q < n; q += CT) s += b ? a[q] * b[q] : a[q];
    __shared__ T res;
    if constexpr (sizeof(T) == sizeof(float)) {
        float m = 0.f, z = 0.f;
        block_red3f(m, s, z);
    } else {
        double m = 0.0, z = 0.0;
        block_red3(m, s, z);
    }
    if (threadIdx.x == 0) res = s;
    __syncthreads();
    const T out = res;
    __syncthreads();
    return out;
}

template <typename T>
__device__ void cta_apply(const Level<T> &L, const T *x, T *y, T ih2) {
    const DGeom &g = L.g;
    for (int c = threadIdx.x; c < g.N; c += CT) {
        const int i = c % g.n[0], r = c / g.n[0], j = r % g.n[1], k = r / g.n[1];
        T b[6], v[6];
        coefs32(L, i, j, k, c, b);
        nb_vals(g, x, i, j, k, c, v);
        y[c] = flux_sum(b, v, x[c]) * ih2;
    }
    __syncthreads();
}

// The same solve with its vectors in shared memory, for bottoms too large for
// registers (levels that cannot be coarsened further).
template <typename T>
__device__ void cta_bicgstab(const Level<T> &L, T *x, const T *f, T *scr, int iters, int singular, T ih2) {
    const int n = int(L.g.N);
    T *r = scr, *r0 = scr + n, *p = scr + 2 * n, *v = scr + 3 * n, *sv = scr + 4 * n, *tv = scr + 5 * n;
    const T mean = singular ? cta_dot(f, (const T *)nullptr, n) / T(n) : T(0);
    for (int q = threadIdx.x; q < n; q += CT) {
        const T b = f[q] - mean;
        x[q] = T(0);
        r[q] = b;
        r0[q] = b;
        p[q] = T(0);
        v[q] = T(0);
    }
    __syncthreads();
    const T bnorm2 = cta_dot(r, r, n);
    if (!(bnorm2 > T(0))) return;
    const T tol2 = bnorm2 * T(1e-8);  // 1e-4 relative: ample for a multigrid bottom solve
    T rho = T(1), alpha = T(1), omega = T(1);
    for (int it = 0; it < iters; it++) {
        const T rho1 = cta_dot(r0, r, n);
        if (rho1 == T(0) || omega == T(0)) break;
        const T beta = (rho1 / rho) * (alpha / omega);
        for (int q = threadIdx.x; q < n; q += CT) p[q] = r[q] + beta * (p[q] - omega * v[q]);
        __syncthreads();
        cta_apply(L, p, v, ih2);
        const T r0v = cta_dot(r0, v, n);
        if (r0v == T(0)) break;
        alpha = rho1 / r0v;
        for (int q = threadIdx.x; q < n; q += CT) sv[q] = r[q] - alpha * v[q];
        __syncthreads();
        const T ss = cta_dot(sv, sv, n);
        if (ss <= tol2) {
            for (int q = threadIdx.x; q < n; q += CT) x[q] += alpha * p[q];
            __syncthreads();
            break;
        }
        cta_apply(L, sv, tv, ih2);
        const T tt = cta_dot(tv, tv, n);
        const T ts = cta_dot(tv, sv, n);
        omega = tt > T(0) ? ts / tt : T(0);
        for (int q = threadIdx.x; q < n; q += CT) {
            x[q] += alpha * p[q] + omega * sv[q];
            r[q] = sv[q] - omega * tv[q];
        }
        __syncthreads();
        rho = rho1;
        const T rr = cta_dot(r, r, n);
        if (rr <= tol2) break;
    }
    if (singular) {
        const T mx = cta_dot(x, (const T *)nullptr, n) / T(n);
        for (int q = threadIdx.x; q < n; q += CT) x[q] -= mx;
        __syncthreads();
    }
}

template <typename T>
__device__ void bottom_solve(const Level<T> &L, T *x, const T *f, T *scr, int iters, int singular) {
    const int n = int(L.g.N);
    const T ih2 = T(1) / T(L.g.h * L.g.h);
    if (n > BOT_REGS * CT) {
        cta_bicgstab(L, x, f, scr, iters, singular, ih2);
        return;
    }
    if (n <= 32) {
        if (threadIdx.x < 32) warp_bicgstab(L, x, f, scr, iters, singular, ih2);
    } else {
        // the fewest warps that hold the cells: their barriers cost less
        const int per = (n + CT - 1) / CT, nthr = ((n + per - 1) / per + 31) & ~31;
        if (int(threadIdx.x) < nthr) {
            if (per == 1) team_bicgstab<T, 1>(L, x, f, scr, iters, singular, ih2, nthr);
            else if (per == 2) team_bicgstab<T, 2>(L, x, f, scr, iters, singular, ih2, nthr);
            else team_bicgstab<T, 3>(L, x, f, scr, iters, singular, ih2, nthr);
        }
    }
    __syncthreads();
}

template <typename T>
__device__ __forceinline__ void coarse_body(const CoarseArgs<T> &A, int rank) {
    constexpr int CPT = CoarseCpt<T>::value;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *sm = reinterpret_cast<T *>(smem_raw);
    for (int q = threadIdx.x; q < A.roff; q += CT) sm[q] = T(0);
    __syncthreads();
    {  // right-hand side of the first level from global memory
        const CoarseLevel<T> &C = A.lev[0];
        const Slab s = slab_of(C, rank);
        const int nxy = int(C.L.g.nxy);
        const T *f = C.L.f + (long long)s.k0 * nxy;
        if (C.dist || rank == 0)
            for (int q = threadIdx.x; q < nxy * s.np; q += CT) sm[C.foff + q] = f[q];
    }
    level_sync(A.nc > 1);
    const int nb = A.nl - 1;
    Cells<T, CPT> R;
    for (int l = 0; l < nb; l++) {
        const CoarseLevel<T> &C = A.lev[l];
        if (!C.dist && rank != 0) break;
        const Slab s = slab_of(C, rank);
        load_cells(C, s, R);
        sweeps(sm, C, s, R, A.nu1);
        restrict_down(sm, A, C, A.lev[l + 1], s, R);
    }
    if (rank == 0) {
        const CoarseLevel<T> &C = A.lev[nb];
        bottom_solve(C.L, sm + C.eoff + C.L.g.nxy, sm + C.foff, sm + A.roff, A.bot_iters, A.singular);
    }
    bool dist_below = false;  // the level below was spread: the cluster is in step already
    for (int l = nb - 1; l >= 0; l--) {
        const CoarseLevel<T> &C = A.lev[l];
        if (!C.dist && rank != 0) continue;
        const Slab s = slab_of(C, rank);
        load_cells(C, s, R);
        if (C.dist && !dist_below) cluster_sync();
        dist_below = C.dist;
        prolong_up(sm, C, A.lev[l + 1], s, R);
        sweeps(sm, C, s, R, A.nu2);
    }
    const CoarseLevel<T> &C = A.lev[0];
    if (C.dist || rank == 0) {
        const Slab s = slab_of(C, rank);
        const int nxy = int(C.L.g.nxy);
        T *e = C.L.e + (long long)s.k0 * nxy;
        for (int q = threadIdx.x; q < nxy * s.np; q += CT) e[q] = sm[C.eoff + nxy + q];
    }
    if (A.nc > 1) cluster_sync();  // no CTA leaves while another may still read its shared memory
}

template <typename T>
__global__ void __launch_bounds__(CT, 1) coarse_vcycle_kernel(const __grid_constant__ CoarseArgs<T> A) {
    pdl_trigger();
    pdl_wait();
    coarse_body(A, int(blockIdx.x));
}

// batched: one CTA per box (boxes already converged return at once)
__global__ void __launch_bounds__(CT, 1) coarse_vcycle_batch_kernel(const CoarseArgs<float> *args,
                                                                    const SolveState *st) {
    if (st[blockIdx.x].done) return;
    coarse_body(args[blockIdx.x], 0);
}

// CTAs of a cluster on this device: 16 need as many free SMs in one GPC and the
// opt-in of coarse_init, which makes the first call; 8 are always allowed.
static int cluster_ctas() {
    static const int nc = [] {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(COARSE_NC);
        cfg.blockDim = dim3(CT);
        cfg.dynamicSmemBytes = COARSE_MAX_SMEM;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = COARSE_NC;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nf = 0, nd = 0;
        if (cudaOccupancyMaxActiveClusters(&nf, coarse_vcycle_kernel<float>, &cfg) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&nd, coarse_vcycle_kernel<double>, &cfg) != cudaSuccess || nf < 1 || nd < 1) {
            cudaGetLastError();
            return 8;
        }
        return COARSE_NC;
    }();
    return nc;
}

// The layout of levels [0, nl) over nc CTAs; false if they do not fit.
template <typename T>
static bool plan_coarse(CoarseArgs<T> &A, const Level<T> *levs, int nl, int nc) {
    if (nl < 1 || nl > COARSE_MAX_LEVELS) return false;
    std::memset(&A, 0, sizeof(A));
    A.nl = nl;
    const int cap = CT * CoarseCpt<T>::value;
    long long off = 4, scratch = 0;  // element 0 stays 0
    int used = 1;
    bool above_dist = true;
    for (int l = 0; l < nl; l++) {
        const DGeom &g = levs[l].g;
        CoarseLevel<T> &C = A.lev[l];
        if (g.N > 65535) return false;
        C.L = levs[l];
        C.d0 = fast_div(g.n[0]);
        C.d1 = fast_div(g.n[1]);
        C.dh = fast_div(g.n[0] > 1 ? g.n[0] / 2 : 1);
        C.dist = nc > 1 && l + 1 < nl && above_dist && g.N > dist_min<T>();
        above_dist = C.dist;
        C.pp = C.dist ? 2 * ((g.n[2] + 2 * nc - 1) / (2 * nc)) : g.n[2];
        if (C.dist) used = std::max(used, (g.n[2] + C.pp - 1) / C.pp);
        const long long own = g.nxy * C.pp;
        if (l + 1 < nl) {
            if (own > cap) return false;
            scratch = std::max(scratch, own);
        } else {
            if (g.N > COARSE_MAX_CELLS) return false;
            scratch = std::max(scratch, g.N > BOT_REGS * CT ? 6 * g.N : 2 * (g.N + 1));
        }
        C.eoff = int(off);
        off += own + 2 * g.nxy;
        C.foff = int(off);
        off += own;
        if (off > 65535) return false;  // neighbour indices are 16 bits
    }
    for (A.nc = 1; A.nc < used;) A.nc *= 2;
    A.roff = int(off);
    if ((off + scratch) * (long long)sizeof(T) > COARSE_MAX_SMEM) return false;
    A.total = int(off + scratch);
    return true;
}

template <typename T>
bool coarse_fits(const Level<T> *levs, int nl, int clustered) {
    CoarseArgs<T> A;
    return plan_coarse(A, levs, nl, clustered ? cluster_ctas() : 1);
}

template <typename T>
void k_coarse_vcycle(cudaStream_t s, const Level<T> *levs, int nl, int nu1, int nu2, int bot_iters, int singular) {
    CoarseArgs<T> A;
    plan_coarse(A, levs, nl, cluster_ctas());
    A.nu1 = nu1;
    A.nu2 = nu2;
    A.bot_iters = bot_iters;
    A.singular = singular;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(A.nc);
    cfg.blockDim = dim3(CT);
    cfg.dynamicSmemBytes = A.total * sizeof(T);
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = A.nc;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = A.nc > 1 ? 2 : 1;
    cudaLaunchKernelEx(&cfg, coarse_vcycle_kernel<T>, A);
}

template <typename T>
static cudaError_t allow(void (*kern)(CoarseArgs<T>)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, COARSE_MAX_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

// Allow the coarse kernels more than the default 48 KB of dynamic shared memory
// and clusters of 16 CTAs (called once per device, outside any stream capture).
cudaError_t coarse_init() {
    cudaError_t e = allow<float>(coarse_vcycle_kernel<float>);
    if (e == cudaSuccess) e = allow<double>(coarse_vcycle_kernel<double>);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(coarse_vcycle_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 COARSE_MAX_SMEM);
    if (e != cudaSuccess) return e;
    cluster_ctas();
    return cudaSuccess;
}

size_t coarse_args_bytes() { return sizeof(CoarseArgs<float>); }

size_t coarse_fill_args(void *dst, const Level<float> *levs, int nl, int nu1, int nu2, int bot_iters, int singular) {
    CoarseArgs<float> A;
    plan_coarse(A, levs, nl, 1);
    A.nu1 = nu1;
    A.nu2 = nu2;
    A.bot_iters = bot_iters;
    A.singular = singular;
    std::memcpy(dst, &A, sizeof(A));
    return A.total * sizeof(float);
}

void k_coarse_vcycle_batch(cudaStream_t s, const void *dev_args, const SolveState *st, int nbox, size_t smem) {
    if (nbox > 0)
        coarse_vcycle_batch_kernel<<<nbox, CT, smem, s>>>((const CoarseArgs<float> *)dev_args, st);
}

template bool coarse_fits<float>(const Level<float> *, int, int);
template bool coarse_fits<double>(const Level<double> *, int, int);
template void k_coarse_vcycle<float>(cudaStream_t, const Level<float> *, int, int, int, int, int);
template void k_coarse_vcycle<double>(cudaStream_t, const Level<double> *, int, int, int, int, int);
