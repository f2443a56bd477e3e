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
// wait at the next cluster barrier.
//
// The work is latency, and above all instruction fetch: a warp runs a level's
// code once, so code that is not in the instruction cache costs more than the
// arithmetic.  A thread therefore owns cells of one colour, and the loop over
// the passes is one short body: six shared loads through precomputed offsets,
// the update with the coefficients and reciprocal diagonal in registers, a store
// and a barrier.
#include <algorithm>
#include <cstring>

#include "mx_coarse.cuh"
#include "mx_rbgs.cuh"
#include "mx_stencil.cuh"
#include "mx_team.cuh"

constexpr int CT = 1024;         // threads per CTA
constexpr int BOT_ONE = 256;      // ... of up to BOT_ONE cells hold one cell per thread
constexpr int BOT_REGS = 2;      // bottom solves of up to BOT_REGS * CT cells keep their vectors in registers
constexpr int COARSE_NC = 16;    // CTAs of the cluster (8 where the device cannot place 16)

// cells per thread of the widest level a CTA may own, in a cluster and alone
constexpr int CELLS_CLUSTER = 2, CELLS_ALONE = 4;
// Levels above this many cells are spread over the cluster.  16^3 on one CTA took
// 3000 clocks per colour pass (four cells per thread, spilled registers), 1300
// spread over 8 CTAs, 600 of them the cluster barrier; 8^3 takes 500 on one CTA.
// FP64 is bound by its pipe (a warp instruction takes about 64 clocks of a
// quarter of the SM), so it spreads the next level down too.
template <typename T>
constexpr int dist_min() {
    return sizeof(T) == sizeof(float) ? 1024 : 512;
}

// Largest level taken.  An FP64 warp instruction takes 64 clocks of its quarter of
// the SM, so the 16 SMs of a cluster need 2.9 us for a colour pass of 32^3, more
// than its launch over the whole GPU; FP32 is limited by the cells a CTA may own.
template <typename T>
constexpr int level_max() {
    return sizeof(T) == sizeof(float) ? 65535 : 8192;
}

// Exact division of x < 2^16 by d < 2^16 as a multiply-high with the
// precomputed m = ceil(2^32 / d) (the error x (m - 2^32/d) / 2^32 stays below
// 1/d, so the floor is exact).
struct FastDiv {
    unsigned d, m;
};
inline FastDiv fast_div(unsigned d) { return FastDiv{d, unsigned(((1ull << 32) + d - 1) / d)}; }
__device__ __forceinline__ int fdiv(int x, FastDiv f) { return f.d == 1 ? x : int(__umulhi(unsigned(x), f.m)); }

// One level of the coarse end.  Shared-memory offsets are in bytes and equal in
// every CTA; the correction holds pp + 2 planes (a neighbour's plane first and
// last), the right-hand side pp planes.  The bottom level, which only its own solve
// visits, has no neighbours' planes: eoff lies a plane before its first cell.
template <typename T>
struct CoarseLevel {
    Level<T> L;
    FastDiv d0, d1, dh, dp;  // n0, n1, n0 / 2, pp
    int dist;            // spread over the cluster
    int pp;              // planes per CTA (even where dist)
    int eoff, foff;
    T h2, ih2;           // h^2 and 1 / h^2, rounded as the other kernels round them
};

template <typename T>
struct CoarseArgs {
    int nl;  // number of levels handled (the last is the bottom)
    CoarseLevel<T> lev[COARSE_MAX_LEVELS];
    int nu1, nu2, bot_iters, singular;
    int nc;    // CTAs
    int roff;  // scratch: the residuals of a level, then the bottom solve's vectors
    int total; // bytes of shared memory
};

extern __shared__ __align__(16) unsigned char coarse_smem[];
template <typename T>
__device__ __forceinline__ T &sm_at(int byte) {
    return *reinterpret_cast<T *>(coarse_smem + byte);
}

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// address of this CTA's shared byte in CTA `rank` of the cluster
__device__ __forceinline__ unsigned cluster_addr(int byte, int rank) {
    const unsigned a = unsigned(__cvta_generic_to_shared(coarse_smem)) + byte;
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void remote_store(unsigned a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void remote_store(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void remote_load(unsigned a, float &v) {
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void remote_load(unsigned a, double &v) {
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
}

// The threads that hold a level's cells: the cluster or the block.
__device__ __forceinline__ void level_sync(int dist) {
    if (dist) cluster_sync();
    else __syncthreads();
}

// the 6 face coefficients of in-box cell (i,j,k) = c with 32-bit indexing (the
// same values as face_coefs); addresses are selected, so the loads issue together
template <typename T>
__device__ __forceinline__ void coefs32(const Level<T> &L, int i, int j, int k, int c, T b[6]) {
    const DGeom &g = L.g;
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxy = nx * ny;
    const bool hx = i + 1 == nx && !gper(g, 0), hy = j + 1 == ny && !gper(g, 1), hz = k + 1 == nz && !gper(g, 2);
    const T *px = hx ? L.hx : L.bx, *py = hy ? L.hy : L.by, *pz = hz ? L.hz : L.bz;
    const int ox = hx ? j + ny * k : (i + 1 == nx ? c - (nx - 1) : c + 1);
    const int oy = hy ? i + nx * k : (j + 1 == ny ? c - (ny - 1) * nx : c + nx);
    const int oz = hz ? i + nx * j : (k + 1 == nz ? c - (nz - 1) * nxy : c + nxy);
    b[0] = L.bx[c];
    b[1] = px[ox];
    b[2] = L.by[c];
    b[3] = py[oy];
    b[4] = L.bz[c];
    b[5] = pz[oz];
}

// The cells of one thread, all of one colour: coefficients and shared offsets.
template <typename T, int SL>
struct Cells {
    T b[SL][6];
    T inv[SL];        // 1 / sum of b
    int at[SL];       // the cell's correction; 0: no cell
    unsigned xn[SL];  // its x neighbours (low half: i - 1), y neighbours
    unsigned yn[SL];
    unsigned push[SL];  // cluster address of the copy of it (0: none)
};

template <typename T, int SL>
__device__ __forceinline__ void neighbours(const Cells<T, SL> &R, int q, int plane, T v[6]) {
    v[0] = sm_at<T>(R.xn[q] & 0xffffu);
    v[1] = sm_at<T>(R.xn[q] >> 16);
    v[2] = sm_at<T>(R.yn[q] & 0xffffu);
    v[3] = sm_at<T>(R.yn[q] >> 16);
    v[4] = sm_at<T>(R.at[q] - plane);
    v[5] = sm_at<T>(R.at[q] + plane);
}

// One level on the way down (smoothing from e = 0, restriction to the level
// below) or up (prolongation, smoothing), with SL cells per thread.
template <typename T, int SL>
__device__ __forceinline__ void visit(const CoarseArgs<T> &A, int l, int rank, bool up) {
    constexpr int B = sizeof(T);
    const CoarseLevel<T> &C = A.lev[l], &F = A.lev[l + 1];
    const DGeom &g = C.L.g;
    const int nx = g.n[0], ny = g.n[1], nxy = nx * ny, dist = C.dist;
    const int k0 = rank * C.pp, np = max(0, min(C.pp, g.n[2] - k0)), half = (nxy * np) >> 1;
    const int team = dist ? CT / 2 : ((half + SL - 1) / SL + 31) & ~31;  // threads per colour
    const bool works = int(threadIdx.x) < 2 * team;
    const int colour = int(threadIdx.x) >= team;
    const int e0 = C.eoff + nxy * B, plane = nxy * B, df = C.foff - e0;
    Cells<T, SL> R;
    {
        // ranks that hold copies of the first and the last plane (-1: none)
        const bool px = gper(g, 0), py = gper(g, 1), pz = gper(g, 2);
        const int last = (g.n[2] - 1) / C.pp;
        const int dn = rank > 0 ? rank - 1 : (pz ? last : -1), upr = rank < last ? rank + 1 : (pz ? 0 : -1);
        const int dnp = dn == last ? g.n[2] - last * C.pp : C.pp;  // dn's planes
#pragma unroll
        for (int q = 0; q < SL; q++) {
            const int m = int(threadIdx.x) - colour * team + team * q;
            R.at[q] = 0;
            R.push[q] = 0;
            if (works && m < half) {
                const int r = fdiv(m, C.dh);  // row j + n1 p
                const int p = fdiv(r, C.d1);
                const int j = r - p * ny, k = k0 + p;
                const int i = 2 * (m - r * int(C.dh.d)) + ((j + k + colour) & 1);
                coefs32(C.L, i, j, k, i + nx * (j + ny * k), R.b[q]);
                const int a = e0 + (i + nx * r) * B;
                R.at[q] = a;
                // offset 0 holds 0: the neighbour beyond a non-periodic face
                const int xl = i > 0 ? a - B : (px ? a + (nx - 1) * B : 0);
                const int xh = i + 1 < nx ? a + B : (px ? a - (nx - 1) * B : 0);
                const int yl = j > 0 ? a - nx * B : (py ? a + (ny - 1) * nx * B : 0);
                const int yh = j + 1 < ny ? a + nx * B : (py ? a - (ny - 1) * nx * B : 0);
                R.xn[q] = unsigned(xl) | (unsigned(xh) << 16);
                R.yn[q] = unsigned(yl) | (unsigned(yh) << 16);
                const int in_plane = (i + nx * j) * B;
                if (p == 0 && dn >= 0) R.push[q] = cluster_addr(C.eoff + (dnp + 1) * plane + in_plane, dn);
                if (p == np - 1 && upr >= 0) R.push[q] = cluster_addr(C.eoff + in_plane, upr);
                if constexpr (B == 4) R.inv[q] = gs_inverse(R.b[q]);
                else R.inv[q] = C.L.di[i + nx * (j + ny * k)];
            }
        }
    }
    if (up) {  // e += the parents' corrections
        const int mx = nx >> 1, mxy = nxy >> 2;
#pragma unroll
        for (int q = 0; q < SL; q++)
            if (R.at[q]) {
                const int c = (R.at[q] - e0) / B;
                const int r = fdiv(c, C.d0);
                const int p = fdiv(r, C.d1);
                const int i = c - r * nx, j = r - p * ny, K = (k0 + p) >> 1;
                const int owner = F.dist ? fdiv(K, F.dp) : 0;
                const int src = F.eoff + (mxy + (i >> 1) + mx * (j >> 1) + mxy * (K - owner * F.pp)) * B;
                T ec;
                if (dist) remote_load(cluster_addr(src, owner), ec);
                else ec = sm_at<T>(src);
                const T v = sm_at<T>(R.at[q]) + ec;
                sm_at<T>(R.at[q]) = v;
                if (R.push[q]) remote_store(R.push[q], v);
            }
        level_sync(dist);
    }
    const T h2 = C.h2;
    const int passes = 2 * (up ? A.nu2 : A.nu1);
#pragma unroll 1
    for (int w = 0; w < passes; w++) {
        if ((w & 1) == colour) {
#pragma unroll
            for (int q = 0; q < SL; q++)
                if (R.at[q]) {
                    T v[6];
                    neighbours(R, q, plane, v);
                    const T e = gs_update(R.b[q], v, sm_at<T>(R.at[q] + df), h2, R.inv[q]);
                    sm_at<T>(R.at[q]) = e;
                    if (R.push[q]) remote_store(R.push[q], e);
                }
        }
        level_sync(dist);
    }
    if (!up) {  // the level below: right-hand side = means of the 8 residuals
        const T ih2 = C.ih2;
#pragma unroll
        for (int q = 0; q < SL; q++)
            if (R.at[q]) {
                T r = T(0);
                // FP64, after a black pass: the black residuals are rounding (as in
                // resid_restrict_red_kernel)
                if (B == sizeof(float) || colour == 0 || passes == 0) {
                    T v[6];
                    neighbours(R, q, plane, v);
                    r = sm_at<T>(R.at[q] + df) - flux_sum(R.b[q], v, sm_at<T>(R.at[q])) * ih2;
                }
                sm_at<T>(A.roff + R.at[q] - e0) = r;
            }
        __syncthreads();
        const int mx = nx >> 1, mxy = nxy >> 2, nown = (nxy * np) >> 3;
        for (int t = threadIdx.x; t < nown; t += CT) {
            const int r = fdiv(t, F.d0);
            const int P = fdiv(r, F.d1);
            const int I = t - r * mx, J = r - P * int(F.d1.d), K = (k0 >> 1) + P;
            const int c = A.roff + (2 * I + nx * (2 * J) + nxy * (2 * P)) * B;
            T sum = T(0);
#pragma unroll
            for (int d = 0; d < 8; d++)
                sum += sm_at<T>(c + ((d & 1) + nx * ((d >> 1) & 1) + nxy * (d >> 2)) * B);
            const int owner = F.dist ? fdiv(K, F.dp) : 0;
            const int dst = F.foff + (I + mx * J + mxy * (K - owner * F.pp)) * B;
            if (dist) remote_store(cluster_addr(dst, owner), sum * T(0.125));
            else sm_at<T>(dst) = sum * T(0.125);
        }
    }
}

// BiCGStab on L x = f (x starts at 0), projected onto mean-free vectors when
// the problem is singular; stops at relative residual 1e-4 or `iters`.  The
// operator is preconditioned from the right with its diagonal (v = L D^-1 p, so
// the residuals are those of L x = f): the stratified coefficients vary a hundredfold
// over the bottom level.  What is solved is h^2 L x' = f' with f' = f 2^m of norm 1 to
// 2 and x = x' h^2 / 2^m, so no sum or quotient depends on the unit of length or on
// how far the outer iteration has come; in FP32 the sums of (L p)^2 would vanish with
// cells of 1e8 units, and the quotients leave the fast division's range.  Each of
// nthr threads (whole warps) holds up to B cells (cell t + q nthr): coefficients
// and vectors stay in registers, and the vector the operator is applied to passes
// through shared memory (element n holds 0 for faces without a neighbour).
//
// The cost is instruction fetch and the latency of the sums, so the iteration is
// one rolled body run twice (v = L p, t = L s) with one reduction each:
//   r0.v gives alpha; s.s, t.t, t.s and r0.t give omega, the next residual's norm
//   s.s - 2 omega t.s + omega^2 t.t, and the next r0.r = -omega r0.t, since
//   r0.s = r0.r - alpha r0.v = 0.
// The operations are rounded explicitly, so the single and the batched kernel
// agree bit for bit.
template <typename T, int B>
__device__ __forceinline__ void team_bicgstab(TeamShared<T> &S, const Level<T> &L, T *x, const T *f, T *scr, int iters, int singular,
                                              T h2, int nthr) {
    const int n = int(L.g.N), nx = L.g.n[0], ny = L.g.n[1], nz = L.g.n[2], nxy = nx * ny;
    T b[B][6], den[B], dinv[B], xv[B], r[B], r0[B] = {}, p[B], v[B];
    unsigned nb[B][3];
    const unsigned vec = unsigned(__cvta_generic_to_shared(scr));
    if (threadIdx.x < 2) team_put(vec + (threadIdx.x * (n + 1) + n) * unsigned(sizeof(T)), T(0));
    T a[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
    for (int q = 0; q < B; q++) {
        const int c = threadIdx.x + q * nthr;
        xv[q] = r[q] = p[q] = v[q] = T(0);
        for (int d = 0; d < 6; d++) b[q][d] = T(0);
        nb[q][0] = nb[q][1] = nb[q][2] = unsigned(n) | (unsigned(n) << 16);
        if (c < n) {
            const int i = c % nx, rr = c / nx, j = rr % ny, k = rr / ny;
            const bool px = gper(L.g, 0), py = gper(L.g, 1), pz = gper(L.g, 2);
            coefs32(L, i, j, k, c, b[q]);
            const int xl = i > 0 ? c - 1 : (px ? c + nx - 1 : n), xh = i + 1 < nx ? c + 1 : (px ? c - (nx - 1) : n);
            const int yl = j > 0 ? c - nx : (py ? c + (ny - 1) * nx : n);
            const int yh = j + 1 < ny ? c + nx : (py ? c - (ny - 1) * nx : n);
            const int zl = k > 0 ? c - nxy : (pz ? c + (nz - 1) * nxy : n);
            const int zh = k + 1 < nz ? c + nxy : (pz ? c - (nz - 1) * nxy : n);
            nb[q][0] = unsigned(xl) | (unsigned(xh) << 16);
            nb[q][1] = unsigned(yl) | (unsigned(yh) << 16);
            nb[q][2] = unsigned(zl) | (unsigned(zh) << 16);
            r[q] = f[c];
            a[0] += r[q];
        }
        den[q] = radd(radd(radd(b[q][0], b[q][1]), radd(b[q][2], b[q][3])), radd(b[q][4], b[q][5]));
        dinv[q] = den[q] != T(0) ? rinv(den[q]) : T(0);
    }
    TeamSum<T> team(S, nthr);
    const T inv_n = T(1) / T(n);
    T mean = T(0), rho1 = T(0), rho = T(1), alpha = T(1), omega = T(1), tol2 = T(0);
    // step -1: the mean of f and ||f - mean||^2; then the iterations
    team.sum(a);
    if (singular) mean = a[0] * inv_n;
    a[0] = a[1] = a[2] = a[3] = T(0);
#pragma unroll
    for (int q = 0; q < B; q++) {
        if (int(threadIdx.x) + q * nthr < n) r[q] -= mean;
        a[0] = rfma(r[q], r[q], a[0]);
    }
    team.sum(a);
    rho1 = a[0];
    T unit = T(1);
    if (rho1 > T(0)) {
        unit = unit_scale(rho1);
        rho1 = rho1 * unit * unit;
#pragma unroll
        for (int q = 0; q < B; q++) r0[q] = r[q] = r[q] * unit;
        tol2 = rho1 * T(1e-8);  // 1e-4 relative: ample for a multigrid bottom solve
#pragma unroll 1
        for (int it = 0; it < iters; it++) {
            const T last = rho * omega;
            if (rho1 == T(0) || fabs(last) < T(BREAKDOWN)) break;
            const T beta = sdiv(rho1 * alpha, last);
            T w[B], y[B];
#pragma unroll
            for (int q = 0; q < B; q++) w[q] = p[q] = rfma(beta, rfma(-omega, v[q], p[q]), r[q]);
            bool stop = false;
#pragma unroll 1
            for (int h = 0; h < 2; h++) {  // y = L w: v = L p, then t = L s
                const unsigned e = vec + h * (n + 1) * unsigned(sizeof(T));
                const auto at = [&](unsigned c) { return team_get(e + c * unsigned(sizeof(T)), T(0)); };
#pragma unroll
                for (int q = 0; q < B; q++)
                    if (int(threadIdx.x) + q * nthr < n)
                        team_put(e + (threadIdx.x + q * nthr) * unsigned(sizeof(T)), rmul(w[q], dinv[q]));
                team.barrier();
                a[0] = a[1] = a[2] = a[3] = T(0);
#pragma unroll
                for (int q = 0; q < B; q++) {
                    const T s0 = rfma(b[q][0], at(nb[q][0] & 0xffffu), rmul(b[q][1], at(nb[q][0] >> 16)));
                    const T s1 = rfma(b[q][2], at(nb[q][1] & 0xffffu), rmul(b[q][3], at(nb[q][1] >> 16)));
                    const T s2 = rfma(b[q][4], at(nb[q][2] & 0xffffu), rmul(b[q][5], at(nb[q][2] >> 16)));
                    y[q] = rfma(-den[q], rmul(w[q], dinv[q]), radd(radd(s0, s1), s2));
                    a[0] = rfma(r0[q], y[q], a[0]);
                    a[1] = rfma(w[q], w[q], a[1]);
                    a[2] = rfma(y[q], y[q], a[2]);
                    a[3] = rfma(y[q], w[q], a[3]);
                }
                team.sum(a);
                if (h == 0) {
                    stop = fabs(a[0]) < T(BREAKDOWN);
                    if (stop) break;
                    alpha = sdiv(rho1, a[0]);
#pragma unroll
                    for (int q = 0; q < B; q++) {
                        v[q] = y[q];
                        w[q] = rfma(-alpha, y[q], r[q]);
                    }
                }
            }
            if (stop) break;
            const bool small = a[1] <= tol2;  // s is small enough: no second half step
            omega = !small && a[2] > T(0) ? sdiv(a[3], a[2]) : T(0);
#pragma unroll
            for (int q = 0; q < B; q++) {
                xv[q] = rfma(rfma(omega, w[q], rmul(alpha, p[q])), dinv[q], xv[q]);
                r[q] = rfma(-omega, y[q], w[q]);
            }
            if (small || rfma(-omega, rfma(-omega, a[2], rmul(T(2), a[3])), a[1]) <= tol2) break;
            rho = rho1;
            rho1 = -omega * a[0];
        }
    }
    a[0] = a[1] = a[2] = a[3] = T(0);
    if (singular) {
#pragma unroll
        for (int q = 0; q < B; q++) a[0] += xv[q];
        team.sum(a);
        mean = a[0] * inv_n;
    }
    const T back = h2 / unit;
#pragma unroll
    for (int q = 0; q < B; q++)
        if (int(threadIdx.x) + q * nthr < n)
            x[threadIdx.x + q * nthr] = rmul(xv[q] - (singular ? mean : T(0)), back);
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

// y = h^2 L x
template <typename T>
__device__ void cta_apply(const Level<T> &L, const T *x, T *y) {
    const DGeom &g = L.g;
    for (int c = threadIdx.x; c < g.N; c += CT) {
        const int i = c % g.n[0], r = c / g.n[0], j = r % g.n[1], k = r / g.n[1];
        T b[6], v[6];
        coefs32(L, i, j, k, c, b);
        nb_vals(g, x, i, j, k, c, v);
        y[c] = flux_sum(b, v, x[c]);
    }
    __syncthreads();
}

// The same solve with its vectors in shared memory, for bottoms too large for
// registers (levels that cannot be coarsened further).
template <typename T>
__device__ void cta_bicgstab(const Level<T> &L, T *x, const T *f, T *scr, int iters, int singular, T h2) {
    const int n = int(L.g.N);
    T *r = scr, *r0 = scr + n, *p = scr + 2 * n, *v = scr + 3 * n, *sv = scr + 4 * n, *tv = scr + 5 * n;
    const T mean = singular ? cta_dot(f, (const T *)nullptr, n) / T(n) : T(0);
    for (int q = threadIdx.x; q < n; q += CT) {
        const T b = f[q] - mean;
        x[q] = T(0);
        r[q] = b;
        p[q] = T(0);
        v[q] = T(0);
    }
    __syncthreads();
    T bnorm2 = cta_dot(r, r, n);
    if (!(bnorm2 > T(0))) return;
    const T unit = unit_scale(bnorm2), back = h2 / unit;
    bnorm2 = bnorm2 * unit * unit;
    for (int q = threadIdx.x; q < n; q += CT) r0[q] = r[q] = r[q] * unit;
    __syncthreads();
    const T tol2 = bnorm2 * T(1e-8);  // 1e-4 relative: ample for a multigrid bottom solve
    T rho = T(1), alpha = T(1), omega = T(1);
    for (int it = 0; it < iters; it++) {
        const T rho1 = cta_dot(r0, r, n);
        if (rho1 == T(0) || omega == T(0)) break;
        const T beta = (rho1 / rho) * (alpha / omega);
        for (int q = threadIdx.x; q < n; q += CT) p[q] = r[q] + beta * (p[q] - omega * v[q]);
        __syncthreads();
        cta_apply(L, p, v);
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
        cta_apply(L, sv, tv);
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
    const T mx = singular ? cta_dot(x, (const T *)nullptr, n) / T(n) : T(0);
    for (int q = threadIdx.x; q < n; q += CT) x[q] = (x[q] - mx) * back;
    __syncthreads();
}

// cells per thread, and threads, of a bottom solve in registers: the fewest warps that
// hold the cells (their barriers cost less); 0 threads: too large
__device__ __forceinline__ int bottom_per(int n) { return n <= BOT_ONE ? 1 : BOT_REGS; }
__device__ __forceinline__ int bottom_threads(int n) {
    const int per = bottom_per(n);
    return n > BOT_REGS * CT ? 0 : ((n + per - 1) / per + 31) & ~31;
}

template <typename T>
__device__ void bottom_solve(TeamShared<T> &S, const Level<T> &L, T h2, T *x, const T *f, T *scr, int iters, int singular) {
    const int n = int(L.g.N);
    const int per = bottom_per(n), nthr = bottom_threads(n);
    if (!nthr) {
        cta_bicgstab(L, x, f, scr, iters, singular, h2);
        return;
    }
    if (int(threadIdx.x) < nthr) {
        if (per == 1) team_bicgstab<T, 1>(S, L, x, f, scr, iters, singular, h2, nthr);
        else team_bicgstab<T, BOT_REGS>(S, L, x, f, scr, iters, singular, h2, nthr);
    }
    __syncthreads();
}

template <typename T, int SLMAX>
__device__ __forceinline__ void coarse_body(const CoarseArgs<T> &A, int rank) {
    constexpr int B = sizeof(T);
    __shared__ TeamShared<T> bottom;
    for (int q = threadIdx.x * B; q < A.roff; q += CT * B) sm_at<T>(q) = T(0);
    __syncthreads();
    const int first = rank * A.lev[0].pp, nxy0 = int(A.lev[0].L.g.nxy);  // this CTA's planes of the first level
    const int own0 = (A.lev[0].dist || rank == 0) ? nxy0 * max(0, min(A.lev[0].pp, A.lev[0].L.g.n[2] - first)) : 0;
    for (int q = threadIdx.x; q < own0; q += CT) sm_at<T>(A.lev[0].foff + q * B) = A.lev[0].L.f[first * nxy0 + q];
    if (A.nc > 1) cluster_sync();
    else __syncthreads();
    const int nb = A.nl - 1;
#pragma unroll 1
    for (int step = 0; step <= 2 * nb; step++) {  // down, bottom, up
        if (step == nb) {
            const CoarseLevel<T> &C = A.lev[nb];
            if (rank == 0)
                bottom_solve(bottom, C.L, C.h2, &sm_at<T>(C.eoff + int(C.L.g.nxy) * B), &sm_at<T>(C.foff), &sm_at<T>(A.roff),
                             A.bot_iters, A.singular);
            continue;
        }
        const bool up = step > nb;
        const int l = up ? 2 * nb - step : step, dist = A.lev[l].dist;
        if (!dist && rank != 0) continue;
        // a spread level above ones of CTA 0 alone: every CTA waits for CTA 0
        if (up && dist && !A.lev[l + 1].dist) cluster_sync();
        const int own = int(A.lev[l].L.g.nxy) * A.lev[l].pp;
        if (own <= CT) visit<T, 1>(A, l, rank, up);
        else visit<T, SLMAX>(A, l, rank, up);
        if (dist) cluster_sync();
        else __syncthreads();
    }
    for (int q = threadIdx.x; q < own0; q += CT)
        A.lev[0].L.e[first * nxy0 + q] = sm_at<T>(A.lev[0].eoff + (nxy0 + q) * B);
    if (A.nc > 1) cluster_sync();  // no CTA leaves while another may still read its shared memory
}

template <typename T>
__global__ void __launch_bounds__(CT, 1) coarse_vcycle_kernel(const __grid_constant__ CoarseArgs<T> A) {
    pdl_trigger();
    pdl_wait();
    coarse_body<T, CELLS_CLUSTER>(A, int(blockIdx.x));
}

// batched: one CTA per box (boxes already converged return at once)
__global__ void __launch_bounds__(CT, 1) coarse_vcycle_batch_kernel(const CoarseArgs<float> *args,
                                                                    const SolveState *st) {
    if (st[blockIdx.x].done) return;
    __shared__ CoarseArgs<float> A;
    static_assert(sizeof(A) % sizeof(int) == 0, "copied by words");
    for (int q = threadIdx.x; q < int(sizeof(A) / sizeof(int)); q += CT)
        reinterpret_cast<int *>(&A)[q] = reinterpret_cast<const int *>(args + blockIdx.x)[q];
    __syncthreads();
    coarse_body<float, CELLS_ALONE>(A, 0);
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
    const int cap = CT * (nc > 1 ? CELLS_CLUSTER : CELLS_ALONE), B = sizeof(T);
    // bytes; the element at 0 stays 0 (the bottom alone has no use for it)
    long long off = nl > 1 ? 16 : 0, scratch = 0;
    int used = 1;
    bool above_dist = true;
    for (int l = 0; l < nl; l++) {
        const DGeom &g = levs[l].g;
        CoarseLevel<T> &C = A.lev[l];
        if (g.N > level_max<T>()) return false;
        C.L = levs[l];
        C.dist = nc > 1 && l + 1 < nl && above_dist && g.N > dist_min<T>();
        above_dist = C.dist;
        C.pp = C.dist ? 2 * ((g.n[2] + 2 * nc - 1) / (2 * nc)) : g.n[2];
        if (C.dist) used = std::max(used, (g.n[2] + C.pp - 1) / C.pp);
        C.d0 = fast_div(g.n[0]);
        C.d1 = fast_div(g.n[1]);
        C.dh = fast_div(g.n[0] > 1 ? g.n[0] / 2 : 1);
        C.dp = fast_div(C.pp);
        C.h2 = T(g.h * g.h);
        C.ih2 = T(1.0 / (g.h * g.h));
        const long long own = g.nxy * C.pp;
        if (l + 1 < nl) {
            if (own > cap) return false;
            scratch = std::max(scratch, own);
        } else {
            if (g.N > COARSE_MAX_CELLS) return false;
            scratch = std::max(scratch, g.N > BOT_REGS * CT ? 6 * g.N : 2 * (g.N + 1));
        }
        if (l + 1 < nl) {
            C.eoff = int(off);
            off += (own + 2 * g.nxy) * B;
            if (off > 65535) return false;  // neighbour offsets are 16 bits
        } else {
            C.eoff = int(off - g.nxy * B);
            off += own * B;
        }
    }
    for (int l = 0; l < nl; l++) {
        A.lev[l].foff = int(off);
        off += levs[l].g.nxy * A.lev[l].pp * B;
    }
    for (A.nc = 1; A.nc < used;) A.nc *= 2;
    A.roff = int(off);
    off += scratch * B;
    A.total = int(off);
    return off <= COARSE_MAX_SMEM;
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
    cfg.dynamicSmemBytes = A.total;
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
    return A.total;
}

void k_coarse_vcycle_batch(cudaStream_t s, const void *dev_args, const SolveState *st, int nbox, size_t smem) {
    if (nbox > 0)
        coarse_vcycle_batch_kernel<<<nbox, CT, smem, s>>>((const CoarseArgs<float> *)dev_args, st);
}

template bool coarse_fits<float>(const Level<float> *, int, int);
template bool coarse_fits<double>(const Level<double> *, int, int);
template void k_coarse_vcycle<float>(cudaStream_t, const Level<float> *, int, int, int, int, int);
template void k_coarse_vcycle<double>(cudaStream_t, const Level<double> *, int, int, int, int, int);
