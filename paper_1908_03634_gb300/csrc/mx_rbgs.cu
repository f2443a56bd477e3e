// One full red-black Gauss-Seidel sweep (red cells, then black cells) of the
// FP32 correction equation L e = f in a single pass over memory.
//
// A block marches a tile of x-y columns up a chunk of z planes, one warp per row
// and one pair of cells (2m, 2m+1) per lane.  At plane k a lane updates its red
// cell from the old values, then the black cell of plane k-1 -- the same column --
// from the new red ones, and writes the finished pair of plane k-1 to a second
// buffer, so halos shared by neighbouring blocks never race.  The first and last
// lane and row of a tile only update red cells (recomputed by the neighbouring
// tile), and a chunk recomputes the red cells of the plane below and above it.
// Per cell the arithmetic is exactly that of the two-pass colour kernels
// (gs_update), so both produce bit-identical sweeps.
//
// Planes of e, f and the coefficients arrive by cp.async in 16-byte chunks into a
// ring of four shared-memory stages, three planes ahead of their first use; a
// thread's chunks, their sources (wrapped on periodic axes, the high-boundary
// planes beyond the last cell, zeros where there is no cell) and its shared
// offsets are fixed before the march, so a plane costs a thread three copies and
// ten shared loads at fixed offsets.  What the next plane reuses stays in
// registers.  One barrier per plane.
//
// Variants: ZERO = the input correction is identically 0 (first sweep of a
// V-cycle level: no read of e); PROLONG = the input is e + P e_coarse
// (piecewise-constant prolongation applied on load, the first sweep after the
// coarse-grid correction).
#include <algorithm>

#include "mx_async.cuh"
#include "mx_rbgs.cuh"
#include "mx_stencil.cuh"

constexpr int SW_ROWS = 16;           // warps of a block: 14 rows and a ring row on either side
constexpr int SW_TY = SW_ROWS - 2;
constexpr int SW_WMAX = 60;           // columns of a tile (lanes 1 .. 30), a multiple of 4
constexpr int SW_RS = SW_WMAX + 12;   // staged row: 4 columns more on either side, padded
constexpr int SW_STAGES = 4;
// rows of a stage: e on rows -2 .. 15 of the tile, by on -1 .. 15, the others on -1 .. 14
constexpr int SW_E = 0, SW_BY = 18, SW_F = 35, SW_BX = 51, SW_BZ = 67, SW_NROW = 83;
constexpr int SW_STAGE = SW_NROW * SW_RS;  // floats
constexpr int SW_THREADS = 32 * SW_ROWS;
constexpr int SW_COPIES = (SW_NROW * (SW_WMAX + 8) / 4 + SW_THREADS - 1) / SW_THREADS;
constexpr size_t SW_SMEM = sizeof(float) * (SW_STAGES * SW_STAGE + 2 * SW_THREADS);

struct SweepArgs {
    Level<float> L;
    const float *ein;
    float *eout;
    const float *ecoarse;
    int ncx, ncy;
    float h2;
    int w, zk;  // tile width, planes per chunk
};

template <int C>
__device__ __forceinline__ float comp(float2 v) {
    return C ? v.y : v.x;
}
// the x neighbours (left, right) of a value in column C of its pair: in the other
// column (own) or in the next lane's
template <int C>
__device__ __forceinline__ float left_of(float own, float other) {
    return C ? own : __shfl_up_sync(0xffffffffu, other, 1);
}
template <int C>
__device__ __forceinline__ float right_of(float own, float other) {
    return C ? __shfl_down_sync(0xffffffffu, other, 1) : own;
}

// position along an axis: the cell's index, wrapped on a periodic axis; ok = false
// (and index 0) where there is no cell
struct Pos {
    int at;
    bool ok;
};
__device__ __forceinline__ Pos pos_of(int u, int n, bool per) {
    Pos p{u, u >= 0 && u < n};
    if (!p.ok && per) {
        p.at = u < 0 ? u + n : u - n;
        p.ok = p.at >= 0 && p.at < n;
    }
    if (!p.ok) p.at = 0;
    return p;
}

// Shared memory by 32-bit address: a thread's base register plus offsets that are
// constants of the unrolled march.
template <int OFF>
__device__ __forceinline__ float lds(unsigned a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(a), "n"(OFF * 4));
    return v;
}
template <int OFF>
__device__ __forceinline__ float2 lds2(unsigned a) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2+%3];" : "=f"(v.x), "=f"(v.y) : "r"(a), "n"(OFF * 4));
    return v;
}
template <int OFF>
__device__ __forceinline__ void sts(unsigned a, float v) {
    asm volatile("st.shared.f32 [%0+%1], %2;" ::"r"(a), "n"(OFF * 4), "f"(v));
}
template <int OFF>
__device__ __forceinline__ void copy16(unsigned a, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0+%1], [%2], 16;" ::"r"(a), "n"(OFF * 4), "l"(src));
}

template <int MODE>
struct March {
    const SweepArgs &A;
    int bx, by;                   // tile
    float h2;
    int nz, k0, k1;
    bool pz, in, out, xedge;
    unsigned mine;                // shared address of this lane's pair in the first stage's row wy
    unsigned ring;                // and of its red value in the first plane of red values
    float *to;                    // the pair's place in plane k0 of eout, then k0+1, ...
    unsigned plane;               // bytes of a plane
    int cc, cs, cn;               // parents' offsets (PROLONG): the pair's, its rows below and above; -1: none
    // this thread's copies: source in plane 0, its stride between planes, destination
    // in the first stage (0: no copy)
    const float *src[SW_COPIES];
    unsigned stride[SW_COPIES], dst[SW_COPIES];

    // queue plane p's copies into stage S
    template <int S>
    __device__ __forceinline__ void fetch(int p) const {
        if (p <= k1 + 1) {
            const Pos z = pos_of(p, nz, pz);
            if (z.ok) {
#pragma unroll
                for (int q = 0; q < SW_COPIES; q++)
                    if (dst[q])
                        copy16<S * SW_STAGE>(dst[q], reinterpret_cast<const char *>(src[q]) +
                                                         (unsigned long long)unsigned(z.at) * stride[q]);
                if (xedge && threadIdx.x == 0 && row_in()) {  // the faces right of the last column
                    const unsigned d = hx_dst();
                    asm volatile("cp.async.ca.shared.global [%0+%1], [%2], 4;" ::"r"(d), "n"(S * SW_STAGE * 4),
                                 "l"(A.L.hx + hx_row() + A.L.g.n[1] * z.at));
                }
            } else {  // beyond a wall: no old values; above the last plane the faces there
#pragma unroll
                for (int q = 0; q < SW_COPIES; q++)
                    if (dst[q]) {
                        const unsigned off = dst[q] - stage0();
                        if (off >= SW_BZ * SW_RS * 4 && p == nz) copy16<S * SW_STAGE>(dst[q], A.L.hz + (src[q] - A.L.bz));
                        if (off < SW_BY * SW_RS * 4)
                            asm volatile("st.shared.v4.f32 [%0+%1], {%2, %2, %2, %2};" ::"r"(dst[q]), "n"(S * SW_STAGE * 4), "f"(0.f));
                    }
            }
        }
        cp_async_commit();
    }
    static __device__ __forceinline__ unsigned stage0() {
        extern __shared__ __align__(16) float sweep_smem[];
        return unsigned(__cvta_generic_to_shared(sweep_smem));
    }
    // row of this warp and the staged place of bx at column nx
    __device__ __forceinline__ int hx_row() const {
        return pos_of(by * SW_TY - 1 + int(threadIdx.y), A.L.g.n[1], gper(A.L.g, 1)).at;
    }
    __device__ __forceinline__ bool row_in() const {
        return pos_of(by * SW_TY - 1 + int(threadIdx.y), A.L.g.n[1], gper(A.L.g, 1)).ok;
    }
    __device__ __forceinline__ unsigned hx_dst() const {
        return stage0() + ((SW_BX + threadIdx.y) * SW_RS + A.L.g.n[0] - bx * A.w + 4) * 4;
    }

    __device__ __forceinline__ float parent(int o, int p) const {
        const Pos z = pos_of(p, nz, pz);
        return o >= 0 && z.ok && p <= k1 + 1 ? __ldg(A.ecoarse + o + A.ncx * A.ncy * (z.at >> 1)) : 0.f;
    }
    template <int S>
    __device__ __forceinline__ float2 old_pair(float par) const {
        if (MODE == RB_ZERO) return make_float2(0.f, 0.f);
        float2 v = lds2<S * SW_STAGE + (SW_E + 1) * SW_RS>(mine);
        if (MODE == RB_PROLONG) {
            v.x += par;
            v.y += par;
        }
        return v;
    }

    // carried from plane to plane
    float2 e0, bz0;              // old e and bz of plane k
    float em;                    // old e of plane k-1 in the red column of plane k
    float2 pbx;                  // plane k-1: bx, and by, by of the row above, bz, f of its black cell
    float pby, pbn, pbz, pf;
    float r1, r2;                // new red values of planes k-1 and k-2
    float pc, ps, pn;            // PROLONG: parents of the pair on plane k+1, of the rows below and above on k

    // plane k in stage S, red column C
    template <int C, int S>
    __device__ __forceinline__ void step(int k) {
        cp_async_wait<1>();  // plane k+1 has arrived (this thread's part)
        // warps of odd and even rows run different copies of this
        asm volatile("barrier.sync 0;" ::: "memory");
        fetch<(S + 3) % SW_STAGES>(k + 3);
        constexpr int G = S * SW_STAGE, U = (S + 1) % SW_STAGES * SW_STAGE;
        const float2 bx = lds2<G + SW_BX * SW_RS>(mine), f = lds2<G + SW_F * SW_RS>(mine);
        const float2 by = lds2<G + SW_BY * SW_RS>(mine), bn = lds2<G + (SW_BY + 1) * SW_RS>(mine);
        const float2 bu = lds2<U + SW_BZ * SW_RS>(mine);
        const float2 eu = old_pair<(S + 1) % SW_STAGES>(pc);
        float b[6], v[6];
        b[0] = comp<C>(bx);
        if constexpr (C == 1) b[1] = lds<G + SW_BX * SW_RS + 2>(mine);
        else b[1] = bx.y;
        b[2] = comp<C>(by);
        b[3] = comp<C>(bn);
        b[4] = comp<C>(bz0);
        b[5] = comp<C>(bu);
        v[0] = left_of<C>(e0.x, e0.y);
        v[1] = right_of<C>(e0.y, e0.x);
        v[2] = v[3] = 0.f;
        if constexpr (MODE != RB_ZERO) {
            v[2] = lds<G + SW_E * SW_RS + C>(mine);
            v[3] = lds<G + (SW_E + 2) * SW_RS + C>(mine);
        }
        if (MODE == RB_PROLONG) {
            v[2] += ps;
            v[3] += pn;
        }
        v[4] = em;
        v[5] = comp<C>(eu);
        const float upd = gs_update(b, v, comp<C>(f), h2);
        const float red = in && (pz || (k >= 0 && k < nz)) ? upd : 0.f;
        // black cell of plane k-1, same column
        const float xl = left_of<C>(r1, r1), xr = right_of<C>(r1, r1);
        const float bh = right_of<C>(pbx.y, pbx.x);
        if (out && k > k0) {
            constexpr int P = (S & 1) ? 0 : SW_THREADS;  // plane k-1's red values
            b[0] = comp<C>(pbx);
            b[1] = bh;
            b[2] = pby;
            b[3] = pbn;
            b[4] = pbz;
            b[5] = comp<C>(bz0);
            v[0] = xl;
            v[1] = xr;
            v[2] = lds<P - 32>(ring);
            v[3] = lds<P + 32>(ring);
            v[4] = r2;
            v[5] = red;
            const float blk = gs_update(b, v, pf, h2);
            *reinterpret_cast<float2 *>(to) = C ? make_float2(r1, blk) : make_float2(blk, r1);
            to = reinterpret_cast<float *>(reinterpret_cast<char *>(to) + plane);
        }
        sts<(S & 1) ? SW_THREADS : 0>(ring, red);
        // the other column is black on this plane
        em = comp<1 - C>(e0);
        pbx = bx;
        pby = comp<1 - C>(by);
        pbn = comp<1 - C>(bn);
        pbz = comp<1 - C>(bz0);
        pf = comp<1 - C>(f);
        e0 = eu;
        bz0 = bu;
        r2 = r1;
        r1 = red;
        if (MODE == RB_PROLONG) {
            pc = parent(cc, k + 2);
            ps = parent(cs, k + 1);
            pn = parent(cn, k + 1);
        }
    }

    // planes k0-1 .. k1, plane k in stage (k - k0 + 1) mod 4
    template <int C>
    __device__ __forceinline__ void run() {
        const int first = k0 - 1;
        pbx = make_float2(0.f, 0.f);
        pby = pbn = pbz = pf = r1 = r2 = 0.f;
        if (MODE == RB_PROLONG) {
            pc = parent(cc, first + 1);
            ps = parent(cs, first);
            pn = parent(cn, first);
        }
        fetch<3>(first - 1);
        fetch<0>(first);
        fetch<1>(first + 1);
        cp_async_wait<1>();
        asm volatile("barrier.sync 0;" ::: "memory");
        em = comp<C>(old_pair<3>(MODE == RB_PROLONG ? parent(cc, first - 1) : 0.f));
        e0 = old_pair<0>(MODE == RB_PROLONG ? parent(cc, first) : 0.f);
        bz0 = lds2<SW_BZ * SW_RS>(mine);
        fetch<2>(first + 2);
#pragma unroll 1
        for (int k = first; k <= k1; k += 4) {
            step<C, 0>(k);
            if (k + 1 > k1) break;
            step<1 - C, 1>(k + 1);
            if (k + 2 > k1) break;
            step<C, 2>(k + 2);
            if (k + 3 > k1) break;
            step<1 - C, 3>(k + 3);
        }
        cp_async_wait<0>();
    }
};

template <int MODE>
__device__ __forceinline__ void sweep_body(const SweepArgs &A, int bx, int by, int bz) {
    const Level<float> &L = A.L;
    const DGeom &g = L.g;
    const int nx = g.n[0], ny = g.n[1], nxy = nx * ny;
    const bool px = gper(g, 0), py = gper(g, 1);
    const int lane = threadIdx.x, wy = threadIdx.y, tid = lane + 32 * wy;
    const int x0 = bx * A.w, j0 = by * SW_TY;
    March<MODE> m{A, bx, by, A.h2};
    m.plane = unsigned(nxy) * 4u;
    m.nz = g.n[2];
    m.pz = gper(g, 2);
    m.k0 = bz * A.zk;
    m.k1 = min(m.k0 + A.zk, m.nz);
    const int i = x0 - 2 + 2 * lane, j = j0 - 1 + wy;
    const Pos x = pos_of(i, nx, px), y = pos_of(j, ny, py);
    m.in = x.ok && y.ok;
    m.out = lane >= 1 && 2 * lane <= A.w && i < nx && wy >= 1 && wy <= SW_TY && j < ny;
    m.xedge = !px && x0 + A.w >= nx;
    m.mine = m.stage0() + (wy * SW_RS + 2 * lane + 2) * 4;
    m.ring = m.stage0() + (SW_STAGES * SW_STAGE + tid) * 4;
    m.to = A.eout + x.at + nx * y.at + (long long)nxy * m.k0;
    if (MODE == RB_PROLONG) {
        const Pos s = pos_of(j - 1, ny, py), n = pos_of(j + 1, ny, py);
        m.cc = x.ok && y.ok ? (x.at >> 1) + A.ncx * (y.at >> 1) : -1;
        m.cs = x.ok && s.ok ? (x.at >> 1) + A.ncx * (s.at >> 1) : -1;
        m.cn = x.ok && n.ok ? (x.at >> 1) + A.ncx * (n.at >> 1) : -1;
    }
    const int nch = (A.w + 8) / 4, row0 = MODE == RB_ZERO ? SW_BY : SW_E;
#pragma unroll
    for (int q = 0; q < SW_COPIES; q++) {
        const int c = tid + q * SW_THREADS, r = row0 + c / nch, ch = c % nch;
        m.src[q] = L.f;
        m.stride[q] = m.dst[q] = 0;
        if (r >= SW_NROW) continue;
        const int u = x0 - 4 + 4 * ch;
        const float *base;
        int v;  // row of the box
        if (r < SW_BY) {
            base = A.ein;
            v = j0 - 2 + r - SW_E;
        } else if (r < SW_F) {
            base = L.by;
            v = j0 - 1 + r - SW_BY;
        } else if (r < SW_BX) {
            base = L.f;
            v = j0 - 1 + r - SW_F;
        } else if (r < SW_BZ) {
            base = L.bx;
            v = j0 - 1 + r - SW_BX;
        } else {
            base = L.bz;
            v = j0 - 1 + r - SW_BZ;
        }
        const Pos cx = pos_of(u, nx, px), cy = pos_of(v, ny, py);
        const bool above = r >= SW_BY && r < SW_F && v == ny && !py && cx.ok;  // the faces above the last row
        const unsigned dst = m.stage0() + (r * SW_RS + 4 * ch) * 4;
        if (above || (cx.ok && cy.ok)) {
            m.dst[q] = dst;
            m.src[q] = above ? L.hy + cx.at : base + cx.at + nx * cy.at;
            m.stride[q] = above ? unsigned(nx) * 4u : m.plane;
        } else {  // no cells there: zeros in every stage
            for (int t = 0; t < SW_STAGES; t++)
                asm volatile("st.shared.v4.f32 [%0], {%1, %1, %1, %1};" ::"r"(dst + t * SW_STAGE * 4), "f"(0.f));
        }
    }
    __syncthreads();  // the zeros above, before the first copies into the same rows
    // the pair's red cell at plane k is in column (j + k) & 1 (a periodic axis has an
    // even extent, so wrapping keeps the colour)
    if ((j + m.k0 - 1) & 1) m.template run<1>();
    else m.template run<0>();
}

template <int MODE>
__global__ void __launch_bounds__(SW_THREADS, 2) rbgs_sweep_kernel(const __grid_constant__ SweepArgs A) {
    pdl_trigger();
    pdl_wait();
    sweep_body<MODE>(A, blockIdx.x, blockIdx.y, blockIdx.z);
}

// tiles of equal width, a multiple of 4
__host__ __device__ inline int sweep_width(const DGeom &g) {
    const int tx = (g.n[0] + SW_WMAX - 1) / SW_WMAX;
    return ((g.n[0] + tx - 1) / tx + 3) / 4 * 4;
}

// batched: work[blockIdx.x] = (box, tile x, tile y, chunk of zk planes); to_e2: from
// e into e2, else from e2 into e
template <int MODE>
__global__ void __launch_bounds__(SW_THREADS, 2)
    rbgs_sweep_batch_kernel(const Level<float> *levs, const int4 *work, const SolveState *st, int level, int to_e2,
                            int zk) {
    const int4 q = work[blockIdx.x];
    if (st[q.x].done) return;
    __shared__ SweepArgs A;
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        A.L = levs[q.x * MX_MAXLEV + level];
        A.ein = to_e2 ? A.L.e : A.L.e2;
        A.eout = to_e2 ? A.L.e2 : A.L.e;
        A.h2 = float(A.L.g.h * A.L.g.h);
        A.w = sweep_width(A.L.g);
        A.zk = zk;
    }
    __syncthreads();
    sweep_body<MODE>(A, q.y, q.z, q.w);
}

dim3 rbgs_sweep_grid(const DGeom &g, int zk) {
    const int w = sweep_width(g);
    return dim3((g.n[0] + w - 1) / w, (g.n[1] + SW_TY - 1) / SW_TY, (g.n[2] + zk - 1) / zk);
}

void k_rbgs_sweep_batch(cudaStream_t s, const Level<float> *levs, const int4 *work, int nwork, const SolveState *st,
                        int level, int zero, int to_e2, int zk) {
    if (nwork <= 0) return;
    auto k = zero ? rbgs_sweep_batch_kernel<RB_ZERO> : rbgs_sweep_batch_kernel<RB_PLAIN>;
    k<<<nwork, dim3(32, SW_ROWS), SW_SMEM, s>>>(levs, work, st, level, to_e2, zk);
}

bool rbgs_fused_ok(const DGeom &g) {
    // rows in 16-byte chunks; a periodic axis wraps at most once and keeps the colour
    if (g.n[0] % 4 || g.n[0] < 32 || g.n[1] < 4 || g.n[2] < 4) return false;
    for (int d = 0; d < 3; d++)
        if (gper(g, d) && g.n[d] % 2) return false;
    return true;
}

cudaError_t rbgs_init() {
    const void *kernels[] = {(const void *)rbgs_sweep_kernel<RB_PLAIN>, (const void *)rbgs_sweep_kernel<RB_ZERO>,
                             (const void *)rbgs_sweep_kernel<RB_PROLONG>, (const void *)rbgs_sweep_batch_kernel<RB_PLAIN>,
                             (const void *)rbgs_sweep_batch_kernel<RB_ZERO>};
    for (const void *k : kernels) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(SW_SMEM));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The planes per chunk that make the fewest steps in a row: whole waves of two
// blocks per SM times the planes a block walks (its chunk, one on either side, and
// the time to the first plane).
int rbgs_sweep_zk(int nbox, const DGeom *g) {
    int nz = 0, zk = 1;
    for (int b = 0; b < nbox; b++) nz = std::max(nz, g[b].n[2]);
    long long best = -1;
    for (int c = 1; c <= nz && c <= 64; c++) {
        const int z = (nz + c - 1) / c;
        long long blocks = 0;
        for (int b = 0; b < nbox; b++) {
            const dim3 gr = rbgs_sweep_grid(g[b], z);
            blocks += (long long)gr.x * gr.y * gr.z;
        }
        const long long cost = (blocks + 2 * 152 - 1) / (2 * 152) * (z + 3);
        if (best < 0 || cost < best) {
            best = cost;
            zk = z;
        }
    }
    return zk;
}

void k_rbgs_fused(cudaStream_t s, const Level<float> &L, const float *ein, float *eout, int mode,
                  const Level<float> *coarse) {
    const DGeom &g = L.g;
    SweepArgs A{};
    A.L = L;
    A.ein = ein;
    A.eout = eout;
    A.ecoarse = coarse ? coarse->e : nullptr;
    A.ncx = coarse ? coarse->g.n[0] : 0;
    A.ncy = coarse ? coarse->g.n[1] : 0;
    A.h2 = float(g.h * g.h);
    A.w = sweep_width(g);
    A.zk = rbgs_sweep_zk(1, &g);
    const dim3 grid = rbgs_sweep_grid(g, A.zk);
    auto k = mode == RB_ZERO ? rbgs_sweep_kernel<RB_ZERO>
             : mode == RB_PROLONG ? rbgs_sweep_kernel<RB_PROLONG> : rbgs_sweep_kernel<RB_PLAIN>;
    launch_pdl(k, grid, dim3(32, SW_ROWS), SW_SMEM, s, A);
}
