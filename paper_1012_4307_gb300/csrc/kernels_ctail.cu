// Coarse levels of a cycle (Algorithm 1) in ONE launch of a thread-block cluster: 2D or 3D,
// complex64 or complex128, any smoother and cycle.
//
// The coarse levels (129 x 129 nodes and below on the benchmark grids) hold too little work to
// fill the GPU, so as separate launches each costs a launch latency plus a few dependent
// phases, and on one thread block they are bound by one SM's issue rate.  Here a cluster of
// NC thread blocks (8 or 16 SMs) keeps every level's b, u, t, diagonal and coefficients in its
// distributed shared memory.  Rows run along the slowest axis: a row is a grid line of nx nodes
// in 2D and a plane of nx x ny nodes in 3D.  Block r owns the interior rows B_l[r] ..
// B_l[r+1]-1 of level l,
// the slabs nested across levels (B_{l+1}[r] = (B_l[r] + 1) / 2), so that the full weighting of
// an owned coarse row and the prolongation onto an owned fine row only touch rows that the
// block owns or the two rows next to its slab.  Each block keeps those two rows as halo rows
// of u and t; whoever writes the first or last row of its slab also stores the value into the
// neighbouring slab's halo (a store to distributed shared memory, which does not wait), and the
// cluster barrier between phases publishes it.  Every read inside a phase is then a local
// shared-memory read; a dependent read of another block's shared memory costs about as much as
// a whole cluster barrier.  Same arithmetic as the per-level kernels in kernels_mg.cu:
// omega-Jacobi (ping-pong) or omega-red-black sweeps, residual and full weighting, bi- or
// trilinear prolongation, exact coarsest solve by the dense inverse.
//
// complex128 levels are bound by the FP64 units (two lanes per SM and clock), so their sweeps
// are written for few operations: u' = (1 - omega) u + (omega / D) (b - offdiagonal part), with
// omega / D formed once per handle (22 operations per node in 2D instead of about 55 with the
// diagonal assembled and divided by at every node), and a red-black colour takes only its own
// nodes.
//
// What bounds it: the latency of its dependent phases (a cluster barrier and a few shared-memory
// round trips, about 0.8 us each) in complex64, and 16 SMs' FP64 units in complex128.  Measured per
// cycle against a single block with the same levels in its shared memory (and, in complex128, its sweeps
// with a division at every node): 129^2 complex64 V(2,2) 71.7 -> 24.6 us, 641^2 complex128 F cycle (nine
// tails) 2396 -> 755 us, 257^3 complex64 876 -> 757 us.
#include <cooperative_groups.h>

#include <algorithm>

#include "helm_internal.h"

namespace cg = cooperative_groups;

namespace {

constexpr int CT_THREADS = CT_BLOCK_THREADS;

template <typename R> struct CLevel {
    typedef typename CT<R>::T C;
    const C *cf[3];         // global coefficient triples per axis (x, y, z)
    const R *k2;            // global k^2
    C bk, c;
    int nx, ny;             // nodes along x, and along y (3D; 1 in 2D): a row holds nx * ny nodes
    int B[MAX_CT_BLOCKS + 1];     // block r owns interior rows B[r] .. B[r+1]-1 (possibly none)
    unsigned ob, ou, ot, ok, oi, ocx, ocy, ocs;  // byte offsets in shared memory (same in every block);
                                            // ok: the diagonal of M at the owned nodes, oi: its
                                            // reciprocal (formed once; complex128: times omega);
                                            // ocx, ocy (3D): in-row coefficients; ocs: the slow
                                            // axis' coefficients of the owned rows
};

template <typename R> struct CArgs {
    typedef typename CT<R>::T C;
    CLevel<R> lv[MAX_CT_LEVELS];
    int nlev, nu_c, nu1, nu2, rb, zero, gf, gc;
    unsigned total;  // bytes of dynamic shared memory
    R omega;
    const C *minv;   // nu_c x nu_c, row-major (global)
    const C *b_top;  // top level's right-hand side (global)
    C *u_top;        // top level's result; initial guess when !zero (global)
    unsigned obc;         // compact coarsest right-hand side
    unsigned ominv;       // this block's rows of minv (mrow per warp), staged in the prologue
    int mrow;             // 0: minv is read from global memory in the dense phase
    const float4 *img;    // initial shared memory of every block (rank r at r * total / 16), or null
};

struct Ctx {
    unsigned char *sm;
    int rank, nc;
};

// A level as the phases use it: the scalars in registers (a phase's shared-memory stores could
// alias the launch arguments, which live in shared memory too, and would force reloads), this
// block's slab [j0, j1), and the slab bounds of every block (B, in shared memory) for the rare
// accesses to other blocks' rows.
struct LV {
    int nx, ny, S, j0, j1;  // S = nodes of a row
    unsigned ob, ou, ot, ok, oi, ocx, ocy, ocs;
    const int *B;
};
template <typename R> __device__ __forceinline__ LV lv_of(const Ctx &X, const CLevel<R> &L) {
    LV v;
    v.nx = L.nx;
    v.ny = L.ny;
    v.S = L.nx * L.ny;
    v.j0 = L.B[X.rank];
    v.j1 = L.B[X.rank + 1];
    v.ob = L.ob; v.ou = L.ou; v.ot = L.ot; v.ok = L.ok; v.oi = L.oi; v.ocx = L.ocx; v.ocy = L.ocy; v.ocs = L.ocs;
    v.B = L.B;
    return v;
}

// Row j of the level array at offset off in a block's slot layout: slot j - B[c] + 1, so slot
// 0 and slot rows + 1 are the halo rows (a boundary row's halo is never written: zeros).
// This block's row j, for j0 - 1 <= j <= j1:
template <typename C> __device__ __forceinline__ C *lrow(const Ctx &X, const LV &L, unsigned off, int j) {
    return (C *)(X.sm + off) + (size_t)(j - L.j0 + 1) * L.S;
}
// block c's row j (another block's through distributed shared memory)
template <typename C> __device__ __forceinline__ C *crow(const Ctx &X, const LV &L, unsigned off, int j, int c) {
    if (c == X.rank) return lrow<C>(X, L, off, j);
    C *p = (C *)(X.sm + off) + (size_t)(j - L.B[c] + 1) * L.S;
    return cg::this_cluster().map_shared_rank(p, (unsigned)c);
}
__device__ __forceinline__ int owner_of(const LV &L, int nc, int j) {
    int c = 0;
    while (c + 1 < nc && L.B[c + 1] <= j) c++;
    return c;
}

// u(j, q) = v for row j owned by block `owner`, and the same value into every other block whose
// window of rows (B[c] - 1 .. B[c+1]) holds row j: the blocks just above the owner's slab whose
// slabs end at row j (empty ones, then the nearest non-empty one) when j is the owner's first
// row, and likewise below when j is its last row.
template <typename C>
__device__ __forceinline__ void put(const Ctx &X, const LV &L, unsigned off, int j, int q, C v, int owner) {
    const bool own = owner == X.rank;
    const int b0 = own ? L.j0 : L.B[owner], b1 = own ? L.j1 : L.B[owner + 1];
    crow<C>(X, L, off, j, owner)[q] = v;
    if (j == b0)
        for (int p = owner - 1; p >= 0 && L.B[p + 1] == j; p--) crow<C>(X, L, off, j, p)[q] = v;
    if (j == b1 - 1)
        for (int r = owner + 1; r < X.nc && L.B[r] == j + 1; r++) crow<C>(X, L, off, j, r)[q] = v;
}

__device__ __forceinline__ void csync() { cg::this_cluster().sync(); }

// q / m for 0 <= q < 2^21 as (q + 1/2) / m rounded down in FP32: exact, since the quotient is at
// least 1 / (2 m) away from an integer (levels of a tail stay far below that size).
__device__ __forceinline__ int quot(int q, float rm) { return __float2int_rz(((float)q + 0.5f) * rm); }

// f(j, q, i, y) for every owned interior node (row j, node q = i + nx y in it), one node per
// thread and pass (consecutive threads along x).
template <int DIM, typename F>
__device__ __forceinline__ void for_owned(const Ctx &X, const LV &L, F f) {
    const int m = L.nx - 2;
    const float rm = 1.0f / (float)m;
    if constexpr (DIM == 2) {
        const int total = (L.j1 - L.j0) * m;
        for (int t = threadIdx.x; t < total; t += blockDim.x) {
            const int r = quot(t, rm), i = 1 + t - r * m;
            f(L.j0 + r, i, i, 0);
        }
    } else {
        const int my = L.ny - 2, total = (L.j1 - L.j0) * my * m;
        const float rmy = 1.0f / (float)my;
        for (int t = threadIdx.x; t < total; t += blockDim.x) {
            const int r = quot(t, rm), i = 1 + t - r * m, k = quot(r, rmy), y = 1 + r - k * my;
            f(L.j0 + k, i + L.nx * y, i, y);
        }
    }
}
// The same for the nodes of one colour only (colour 0: even i + j (+ k)).
template <int DIM, typename F>
__device__ __forceinline__ void for_colour(const Ctx &X, const LV &L, int colour, F f) {
    const int m = (L.nx - 1) / 2, last = L.nx - 2;
    const float rm = 1.0f / (float)m;
    const int my = DIM == 3 ? L.ny - 2 : 1, total = (L.j1 - L.j0) * my * m;
    const float rmy = 1.0f / (float)my;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        const int r = quot(t, rm), k = DIM == 3 ? quot(r, rmy) : r, y = DIM == 3 ? 1 + r - k * my : 0;
        const int j = L.j0 + k, i = 2 * (t - r * m) + 1 + ((1 + j + y + colour) & 1);
        if (i <= last) f(j, i + (DIM == 3 ? L.nx * y : 0), i, y);
    }
}

// The diagonal of M at an owned node, formed once (bk k^2 + c + the centre coefficients), and its
// reciprocal (complex128: omega / diagonal).
template <typename C> __device__ __forceinline__ C diag_at(const Ctx &X, const LV &L, int j, int q) {
    return ((const C *)(X.sm + L.ok))[(size_t)(j - L.j0) * L.S + q];
}
template <typename C> __device__ __forceinline__ C dinv_at(const Ctx &X, const LV &L, int j, int q) {
    return ((const C *)(X.sm + L.oi))[(size_t)(j - L.j0) * L.S + q];
}

// The off-diagonal part of (M u) at node (j, q) from this block's rows of the array at offset u
// (j - 1 and j + 1 may be halo rows); complex128: acc0 minus that part.
template <typename C, int DIM>
__device__ __forceinline__ C offdiag_at(const Ctx &X, const LV &L, unsigned u, int j, int q, int i, int y, C acc0) {
    const C *cx = (const C *)(X.sm + L.ocx), *cs = (const C *)(X.sm + L.ocs);
    const int li = j - L.j0;
    const C *un = lrow<C>(X, L, u, j - 1), *uc = lrow<C>(X, L, u, j), *us = lrow<C>(X, L, u, j + 1);
    if constexpr (sizeof(acc0) == sizeof(double2)) {
        const C w0 = cx[3 * i], e0 = cx[3 * i + 2], w2 = cs[3 * li], e2 = cs[3 * li + 2];
        C acc = axis_sub<false>(w0, e0, uc[q - 1], uc[q + 1], acc0);
        if constexpr (DIM == 3) {
            const C *cy = (const C *)(X.sm + L.ocy);
            const C w1 = cy[3 * y], e1 = cy[3 * y + 2];
            acc = axis_sub<false>(w1, e1, uc[q - L.nx], uc[q + L.nx], acc);
        }
        return axis_sub<false>(w2, e2, un[q], us[q], acc);
    }
    C acc = cmul(cx[3 * i], uc[q - 1]);
    acc = cfma(cx[3 * i + 2], uc[q + 1], acc);
    if constexpr (DIM == 3) {
        const C *cy = (const C *)(X.sm + L.ocy);
        acc = cfma(cy[3 * y], uc[q - L.nx], acc);
        acc = cfma(cy[3 * y + 2], uc[q + L.nx], acc);
    }
    acc = cfma(cs[3 * li], un[q], acc);
    return cfma(cs[3 * li + 2], us[q], acc);
}
// One relaxed update at node (j, q) of the iterate at offset u.
template <typename R, int DIM>
__device__ __forceinline__ typename CT<R>::T relax_at(const Ctx &X, const LV &L, unsigned u, int j, int q, int i, int y,
                                                      R om) {
    typedef typename CT<R>::T C;
    const C b = lrow<C>(X, L, L.ob, j)[q], uc = lrow<C>(X, L, u, j)[q], di = dinv_at<C>(X, L, j, q);
    const C off = offdiag_at<C, DIM>(X, L, u, j, q, i, y, b);
    if constexpr (sizeof(R) == sizeof(double)) {
        // (1 - omega) u + (omega / D) (b - offdiagonal part)
        return cfma(di, off, cscale(uc, R(1) - om));
    } else {
        const C mu = cfma(diag_at<C>(X, L, j, q), uc, off);
        return cadd(uc, cscale(cmul(csub(b, mu), di), om));
    }
}

// The start of a visit from zero at an owned node whose right-hand side b has just been written, in the
// same phase (the first sweep from zero is pointwise, so it needs no phase of its own): the first
// Jacobi sweep into t, or the first colour of the first red-black sweep (the other colour 0) into u, or
// u = 0 without pre-sweeps.
template <typename R>
__device__ __forceinline__ void start_zero(const Ctx &X, const LV &L, const CArgs<R> *A, int j, int q, int i, int y,
                                           typename CT<R>::T b) {
    typedef typename CT<R>::T C;
    C v = mk(R(0), R(0));
    if (A->nu1 > 0 && !(A->rb && ((i + y + j) & 1))) {
        v = cmul(b, dinv_at<C>(X, L, j, q));
        if constexpr (sizeof(R) == sizeof(float)) v = cscale(v, A->omega);
    }
    put(X, L, A->nu1 > 0 && !A->rb ? L.ot : L.ou, j, q, v, X.rank);
}

// The phases of the cycle.  Each is one out-of-line function over a level index, so that the
// kernel's code stays small (inlining every phase at every depth multiplies it by the levels
// and smoothing steps and runs out of the instruction cache); each ends with a cluster barrier.

// nu sweeps on level l from *cur (partner *oth); started: start_zero has done the pointwise part of the
// first one.  Returns the new pair.
template <typename R, int DIM>
__device__ __noinline__ uint2 ph_smooth(Ctx X, const CArgs<R> *A, int l, int nu, uint2 co, bool started) {
    const LV L = lv_of(X, A->lv[l]);
    const R om = A->omega;
    if (A->rb) {
        for (int h = started ? 1 : 0; h < 2 * nu; h++) {
            // in place: this colour's neighbours (the other colour) are not written here
            const unsigned u = co.x;
            for_colour<DIM>(X, L, h & 1, [&](int j, int q, int i, int y) {
                put(X, L, u, j, q, relax_at<R, DIM>(X, L, u, j, q, i, y, om), X.rank);
            });
            csync();
        }
        return co;
    }
    if (started && nu > 0) co = make_uint2(co.y, co.x);
    for (int s = started ? 1 : 0; s < nu; s++) {
        const unsigned src = co.x, dst = co.y;
        for_owned<DIM>(X, L, [&](int j, int q, int i, int y) {
            put(X, L, dst, j, q, relax_at<R, DIM>(X, L, src, j, q, i, y, om), X.rank);
        });
        csync();
        co = make_uint2(dst, src);
    }
    return co;
}

// (1, 2, 1) along x at node q of row r
template <typename C> __device__ __forceinline__ C w121(const C *r, int q) {
    typedef decltype(r->x) R;
    return cadd(cadd(r[q - 1], r[q + 1]), cscale(r[q], R(2)));
}
// (1, 2, 1) along x, and in 3D along y (stride nx)
template <typename C, int DIM> __device__ __forceinline__ C w121_row(const C *r, int q, int nx) {
    typedef decltype(r->x) R;
    if constexpr (DIM == 2) return w121(r, q);
    else return cadd(cadd(w121(r, q - nx), w121(r, q + nx)), cscale(w121(r, q), R(2)));
}

// Residual of level l (iterate u) into r, then full weighting into level l + 1's b (the fine
// rows 2J-1 .. 2J+1 of an owned coarse row J are owned or halo rows: nested slabs) and the start of
// that level's visit from zero.
// first: u is one sweep from zero, so that D u = omega b (red-black: omega (b - offdiagonal part) at the
// second colour) and complex128 needs no diagonal term.
template <typename R, int DIM>
__device__ __noinline__ void ph_restrict(Ctx X, const CArgs<R> *A, int l, unsigned u, unsigned r, bool first) {
    typedef typename CT<R>::T C;
    const LV L = lv_of(X, A->lv[l]), Lc = lv_of(X, A->lv[l + 1]);
    const R q1 = R(1) - A->omega;
    const bool rb = A->rb != 0, inner = l + 2 < A->nlev;  // the coarsest level is solved, not smoothed
    for_owned<DIM>(X, L, [&](int j, int q, int i, int y) {
        const C b = lrow<C>(X, L, L.ob, j)[q];
        C v;
        if constexpr (sizeof(R) == sizeof(double)) {
            if (!first) v = csub(offdiag_at<C, DIM>(X, L, u, j, q, i, y, b), cmul(diag_at<C>(X, L, j, q), lrow<C>(X, L, u, j)[q]));
            else if (rb && ((i + y + j) & 1)) v = cscale(offdiag_at<C, DIM>(X, L, u, j, q, i, y, b), q1);
            else v = offdiag_at<C, DIM>(X, L, u, j, q, i, y, cscale(b, q1));
        } else {
            v = csub(b, cfma(diag_at<C>(X, L, j, q), lrow<C>(X, L, u, j)[q], offdiag_at<C, DIM>(X, L, u, j, q, i, y, b)));
        }
        put(X, L, r, j, q, v, X.rank);
    });
    csync();
    for_owned<DIM>(X, Lc, [&](int J, int Q, int I, int Y) {
        const C *r0 = lrow<C>(X, L, r, 2 * J - 1), *r1 = lrow<C>(X, L, r, 2 * J), *r2 = lrow<C>(X, L, r, 2 * J + 1);
        const int q = 2 * I + (DIM == 3 ? L.nx * 2 * Y : 0);
        const C a0 = w121_row<C, DIM>(r0, q, L.nx), a1 = w121_row<C, DIM>(r1, q, L.nx), a2 = w121_row<C, DIM>(r2, q, L.nx);
        const C b = cscale(cadd(cadd(a0, a2), cscale(a1, R(2))), DIM == 3 ? R(1.0 / 64.0) : R(0.0625));
        lrow<C>(X, Lc, Lc.ob, J)[Q] = b;
        if (inner) start_zero<R>(X, Lc, A, J, Q, I, Y, b);
    });
    csync();
}

// Bi- or trilinear prolongation of level l + 1's u (coarse rows j/2 and (j+1)/2: owned or halo
// rows of the coarse slab), added to level l's iterate u.
template <typename R, int DIM>
__device__ __noinline__ void ph_prolong(Ctx X, const CArgs<R> *A, int l, unsigned u) {
    typedef typename CT<R>::T C;
    const LV L = lv_of(X, A->lv[l]), Lc = lv_of(X, A->lv[l + 1]);
    for_owned<DIM>(X, L, [&](int j, int q, int i, int y) {
        const C *ea = lrow<C>(X, Lc, Lc.ou, j >> 1), *eb = lrow<C>(X, Lc, Lc.ou, (j + 1) >> 1);
        const int ia = i >> 1, ib = (i + 1) >> 1;
        C e;
        if constexpr (DIM == 2) {
            e = cadd(cadd(ea[ia], ea[ib]), cadd(eb[ia], eb[ib]));
        } else {
            const int ya = Lc.nx * (y >> 1), yb = Lc.nx * ((y + 1) >> 1);
            e = cadd(cadd(cadd(ea[ya + ia], ea[ya + ib]), cadd(ea[yb + ia], ea[yb + ib])),
                     cadd(cadd(eb[ya + ia], eb[ya + ib]), cadd(eb[yb + ia], eb[yb + ib])));
        }
        put(X, L, u, j, q, cadd(lrow<C>(X, L, u, j)[q], cscale(e, DIM == 3 ? R(0.125) : R(0.25))), X.rank);
    });
    csync();
}

template <typename R, int DIM>
__device__ __noinline__ void ph_copy(Ctx X, const CArgs<R> *A, int l, unsigned dst, unsigned src) {
    typedef typename CT<R>::T C;
    const LV L = lv_of(X, A->lv[l]);
    for_owned<DIM>(X, L, [&](int j, int q, int, int) { put(X, L, dst, j, q, lrow<C>(X, L, src, j)[q], X.rank); });
    csync();
}

// Row and in-row node of unknown c (natural order) of a level.
template <int DIM> __device__ __forceinline__ void unknown_at(const LV &L, int c, int &j, int &q) {
    const int mx = L.nx - 2;
    if constexpr (DIM == 2) {
        j = 1 + c / mx;
        q = 1 + c % mx;
    } else {
        const int my = L.ny - 2, r = c / mx;
        j = 1 + r / my;
        q = 1 + c % mx + L.nx * (1 + r % my);
    }
}

// Exact coarsest solve: every block gathers the whole right-hand side, computes its share of
// the rows of Minv b (one warp per row) and stores each result in the owning block's u (and
// the halos that hold its row).
template <typename R, int DIM>
__device__ __noinline__ void ph_dense(Ctx X, const CArgs<R> *A, int l) {
    typedef typename CT<R>::T C;
    const LV L = lv_of(X, A->lv[l]);
    C *bc = (C *)(X.sm + A->obc);
    const int nu = A->nu_c;
    for (int c = threadIdx.x; c < nu; c += blockDim.x) {
        int j, q;
        unknown_at<DIM>(L, c, j, q);
        bc[c] = crow<C>(X, L, L.ob, j, owner_of(L, X.nc, j))[q];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int r = X.rank * nw + warp, k = 0; r < nu; r += X.nc * nw, k++) {
        const C *mrow = A->mrow ? (const C *)(X.sm + A->ominv) + (size_t)(warp * A->mrow + k) * nu
                                : A->minv + (size_t)r * nu;
        C acc = mk(R(0), R(0));
#pragma unroll 4
        for (int c = lane; c < nu; c += 32) acc = cfma(mrow[c], bc[c], acc);
        for (int off = 16; off > 0; off >>= 1) {
            acc.x += __shfl_down_sync(0xffffffffu, acc.x, off);
            acc.y += __shfl_down_sync(0xffffffffu, acc.y, off);
        }
        if (lane == 0) {
            int j, q;
            unknown_at<DIM>(L, r, j, q);
            put(X, L, L.ou, j, q, acc, owner_of(L, X.nc, j));
        }
    }
    csync();
}

// This block's rows of the coarsest inverse into shared memory (the rows ph_dense gives each
// warp), before the kernel waits on its predecessor.
template <typename R>
__device__ __noinline__ void ph_stage_minv(Ctx X, const CArgs<R> *A) {
    typedef typename CT<R>::T C;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5, nu = A->nu_c;
    C *dst = (C *)(X.sm + A->ominv);
    for (int r = X.rank * nw + warp, k = 0; r < nu; r += X.nc * nw, k++)
        for (int c = lane; c < nu; c += 32) dst[(size_t)(warp * A->mrow + k) * nu + c] = A->minv[(size_t)r * nu + c];
}

// Level LVL of the cycle (compile-time depth); the result ends in the level's u.
template <typename R, int DIM, int LVL>
__device__ __noinline__ void ct_cycle(Ctx X, const CArgs<R> *A, bool zero, int gf, int gc) {
    const CLevel<R> &L = A->lv[LVL];
    if (LVL == A->nlev - 1) {
        ph_dense<R, DIM>(X, A, LVL);
        return;
    }
    if constexpr (LVL + 1 < MAX_CT_LEVELS) {
        uint2 co = ph_smooth<R, DIM>(X, A, LVL, A->nu1, make_uint2(L.ou, L.ot), zero);
        ph_restrict<R, DIM>(X, A, LVL, co.x, co.y, zero && A->nu1 == 1);
        if (LVL + 1 == A->nlev - 1) {
            ph_dense<R, DIM>(X, A, LVL + 1);
        } else {
            // first visit from zero with (gf, gc), later ones from the iterate with (gc, gf)
            for (int k = 1; k <= gc; k++) ct_cycle<R, DIM, LVL + 1>(X, A, k == 1, k == 1 ? gf : gc, k == 1 ? gc : gf);
        }
        ph_prolong<R, DIM>(X, A, LVL, co.x);
        co = ph_smooth<R, DIM>(X, A, LVL, A->nu2, co, false);
        if (co.x != L.ou) ph_copy<R, DIM>(X, A, LVL, L.ou, co.x);
    }
}

// The block's shared memory before the cycle: zeros, the staged coefficients, the diagonal
// bk k^2 + c + centre coefficients of the owned rows and the block's rows of the coarsest
// inverse.  X.sm may point to global memory (the image that k_ctail_image builds once).
template <typename R, int DIM>
__device__ __noinline__ void ct_init(Ctx X, const CArgs<R> *A) {
    typedef typename CT<R>::T C;
    for (unsigned q = threadIdx.x; q < A->total / 16; q += blockDim.x) ((float4 *)X.sm)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    for (int l = 0; l < A->nlev; l++) {
        const CLevel<R> &L = A->lv[l];
        const int j0 = L.B[X.rank], j1 = L.B[X.rank + 1];
        C *cx = (C *)(X.sm + L.ocx), *cs = (C *)(X.sm + L.ocs);
        for (int q = threadIdx.x; q < 3 * L.nx; q += blockDim.x) cx[q] = L.cf[0][q];
        if constexpr (DIM == 3) {
            C *cy = (C *)(X.sm + L.ocy);
            for (int q = threadIdx.x; q < 3 * L.ny; q += blockDim.x) cy[q] = L.cf[1][q];
        }
        for (int q = threadIdx.x; q < 3 * (j1 - j0); q += blockDim.x) cs[q] = L.cf[DIM - 1][3 * j0 + q];
    }
    __syncthreads();
    for (int l = 0; l < A->nlev; l++) {
        const CLevel<R> &L = A->lv[l];
        const int j0 = L.B[X.rank], j1 = L.B[X.rank + 1], S = L.nx * L.ny;
        const C *cx = (const C *)(X.sm + L.ocx), *cs = (const C *)(X.sm + L.ocs);
        C *dg = (C *)(X.sm + L.ok), *di = (C *)(X.sm + L.oi);
        for (int p = threadIdx.x; p < (j1 - j0) * S; p += blockDim.x) {
            const int li = p / S, q = p - li * S, i = q % L.nx;
            const R k2 = L.k2[(size_t)j0 * S + p];
            C cc = cadd(cx[3 * i + 1], cs[3 * li + 1]);
            if constexpr (DIM == 3) cc = cadd(cc, ((const C *)(X.sm + L.ocy))[3 * (q / L.nx) + 1]);
            const C d = cadd(cc, cadd(cscale(L.bk, k2), L.c));
            dg[p] = d;
            // (a boundary node's entries are never read)
            di[p] = cinv(d);
            if constexpr (sizeof(R) == sizeof(double)) di[p] = cscale(di[p], A->omega);
        }
    }
    if (A->mrow) ph_stage_minv(X, A);
    __syncthreads();
}

// Builds the initial shared memory of every block of the cluster tail in global memory (one
// block per rank, no cluster): the tail then starts with one copy instead of three dependent
// rounds of loads.
template <typename R, int DIM>
__global__ void __launch_bounds__(CT_THREADS, 1) k_ctail_image(const __grid_constant__ CArgs<R> A0, unsigned char *img) {
    Ctx X{img + (size_t)blockIdx.x * A0.total, (int)blockIdx.x, (int)gridDim.x};
    ct_init<R, DIM>(X, &A0);
}

// The cycle on the staged levels: the top level's right-hand side (and guess) in, its result out.
template <typename R, int DIM>
__device__ __forceinline__ void ct_run(const Ctx &X, const CArgs<R> *A) {
    typedef typename CT<R>::T C;
    const LV T = lv_of(X, A->lv[0]);
    // the operator data above is not written by earlier kernels; b_top and u_top are
    pdl_wait();
    // every block's initial fill precedes any store into its halos
    csync();
    for_owned<DIM>(X, T, [&](int j, int q, int i, int y) {
        const size_t p = (size_t)q + (size_t)T.S * j;
        const C b = A->b_top[p];
        lrow<C>(X, T, T.ob, j)[q] = b;
        if (A->zero) start_zero<R>(X, T, A, j, q, i, y, b);
        else put(X, T, T.ou, j, q, A->u_top[p], X.rank);
    });
    csync();
    ct_cycle<R, DIM, 0>(X, A, A->zero != 0, A->gf, A->gc);
    for_owned<DIM>(X, T, [&](int j, int q, int, int) { A->u_top[(size_t)q + (size_t)T.S * j] = lrow<C>(X, T, T.ou, j)[q]; });
}

template <typename R, int DIM>
__global__ void __launch_bounds__(CT_THREADS, 1) k_mg_ctail(const __grid_constant__ CArgs<R> A0) {
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char ct_smem[];
    __shared__ CArgs<R> As;
    cg::cluster_group cl = cg::this_cluster();
    Ctx X{ct_smem, (int)cl.block_rank(), (int)cl.num_blocks()};
    {
        const int *src = reinterpret_cast<const int *>(&A0);
        int *dst = reinterpret_cast<int *>(&As);
        for (int q = threadIdx.x; q < (int)(sizeof(CArgs<R>) / sizeof(int)); q += blockDim.x) dst[q] = src[q];
    }
    const CArgs<R> *A = &As;
    if (A0.img) {
        const float4 *src = A0.img + (size_t)X.rank * (A0.total / 16);
        block_copy16((float4 *)ct_smem, src, A0.total / 16);
        __syncthreads();
    } else {
        __syncthreads();
        ct_init<R, DIM>(X, A);
    }
    ct_run<R, DIM>(X, A);
}

// Batched cluster tail (2D complex64): cluster z runs problem z's tail (blockIdx.z is shared by
// every block of a cluster, so a cluster returns as a whole when its problem is inactive).  The
// launch arguments A0 are the levels' common layout; the problem's pointers come from its table
// entry, and its blocks start from the problem's prebuilt image.
__global__ void __launch_bounds__(CT_THREADS, 1) k_mg_ctail_b(const __grid_constant__ CArgs<float> A0,
                                                           const BTail *__restrict__ tab, int j) {
    pdl_trigger();
    const BTail &E = tab[blockIdx.z];
    if (*E.active == 0) return;
    extern __shared__ __align__(16) unsigned char ct_smem[];
    __shared__ CArgs<float> As;
    cg::cluster_group cl = cg::this_cluster();
    Ctx X{ct_smem, (int)cl.block_rank(), (int)cl.num_blocks()};
    {
        const int *src = reinterpret_cast<const int *>(&A0);
        int *dst = reinterpret_cast<int *>(&As);
        for (int q = threadIdx.x; q < (int)(sizeof(CArgs<float>) / sizeof(int)); q += blockDim.x) dst[q] = src[q];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int l = 0; l < As.nlev; l++) {
            As.lv[l].cf[0] = E.cx[l];
            As.lv[l].cf[1] = E.cy[l];
            As.lv[l].k2 = E.k2[l];
        }
        As.minv = E.minv;
        As.b_top = E.b_top;
        As.u_top = E.u_top + (size_t)j * E.ustride;
        As.img = (const float4 *)E.img;
    }
    __syncthreads();
    const CArgs<float> *A = &As;
    {
        const float4 *src = A->img + (size_t)X.rank * (A->total / 16);
        block_copy16((float4 *)ct_smem, src, A->total / 16);
        __syncthreads();
    }
    ct_run<float, 2>(X, A);
}

}  // namespace

// n: nodes per axis of every level; rows along axis dim - 1.
bool mg_ctail_bounds(int dim, int nlev, const int (*n)[3], int nc, int (*B)[MAX_CT_BLOCKS + 1]) {
    if (nc < 1 || nc > MAX_CT_BLOCKS) return false;
    const int s = dim - 1;
    for (int l = 0; l < nlev; l++) {
        if (n[l][s] < 3) return false;
        if (l + 1 < nlev && (n[l][s] % 2 == 0 || n[l + 1][s] != (n[l][s] + 1) / 2)) return false;
    }
    const int rows = (n[0][s] - 2 + nc - 1) / nc;
    for (int r = 0; r <= nc; r++) B[0][r] = std::min(1 + r * rows, n[0][s] - 1);
    for (int l = 1; l < nlev; l++)
        for (int r = 0; r <= nc; r++) B[l][r] = (B[l - 1][r] + 1) / 2;
    return true;
}

int mg_ctail_minv_rows(int nc, int nu_c) { return (nu_c + nc * (CT_THREADS / 32) - 1) / (nc * (CT_THREADS / 32)); }
size_t mg_ctail_minv_stage_bytes(int nc, int nu_c, size_t es) {
    const size_t b = (size_t)(CT_THREADS / 32) * mg_ctail_minv_rows(nc, nu_c) * nu_c * es;
    return b <= 64 * 1024 ? b : 0;
}

// Shared-memory layout of the cluster tail (identical in every block): per level b, u, t
// ((rmax + 2) rows each: the owned rows between two halo rows; rmax = the most rows a block
// owns), the diagonal of M and its reciprocal (rmax rows each), the in-row axes' coefficients and
// the slow axis' of the owned rows (3 rmax); then the compact coarsest right-hand side and the
// block's staged rows of the coarsest inverse (ominv).  es: bytes of a value.  Levels that are not
// nested (odd along the rows' axis, halved) get a size no launch accepts.
size_t mg_ctail_layout(int dim, size_t es, int nlev, const int (*n)[3], int nc, int nu_c, unsigned (*off)[8],
                       unsigned *obc, unsigned *ominv) {
    auto al = [](size_t b) { return (b + 15) & ~(size_t)15; };
    int B[MAX_CT_LEVELS][MAX_CT_BLOCKS + 1];
    if (nlev < 1 || nlev > MAX_CT_LEVELS || !mg_ctail_bounds(dim, nlev, n, nc, B)) return ~(size_t)0;
    size_t p = 0;
    for (int l = 0; l < nlev; l++) {
        const size_t S = (size_t)n[l][0] * (dim == 3 ? n[l][1] : 1);
        if (S > (1u << 16)) return ~(size_t)0;
        int rmax = 0;
        for (int r = 0; r < nc; r++) rmax = std::max(rmax, B[l][r + 1] - B[l][r]);
        const size_t vec = al((rmax + 2) * S * es);
        if (p + 3 * vec > CT_SMEM_BYTES) return ~(size_t)0;
        off[l][0] = (unsigned)p; p += vec;                                             // b
        off[l][1] = (unsigned)p; p += vec;                                             // u
        off[l][2] = (unsigned)p; p += vec;                                             // t
        off[l][3] = (unsigned)p; p += al(rmax * S * es);                               // diagonal
        off[l][4] = (unsigned)p; p += al(rmax * S * es);                               // its reciprocal
        off[l][5] = (unsigned)p; p += al((size_t)3 * n[l][0] * es);                    // x coefficients
        off[l][6] = (unsigned)p; p += dim == 3 ? al((size_t)3 * n[l][1] * es) : 0;     // y coefficients (3D)
        off[l][7] = (unsigned)p; p += al((size_t)3 * rmax * es);                       // slow axis' coefficients
    }
    *obc = (unsigned)p;
    p += al((size_t)nu_c * es);
    *ominv = (unsigned)p;
    p += al(mg_ctail_minv_stage_bytes(nc, nu_c, es));
    return p;
}

// The launch arguments of a cluster tail over nlev levels on nc blocks (0 bytes: not possible).
template <typename R>
static size_t ct_args(int dim, int nlev, const DevOp<R> *ops, const typename CT<R>::T *minv, int nu_c, R omega, int nc,
                      CArgs<R> &A) {
    if (nlev < 2 || nlev > MAX_CT_LEVELS || (nc != 8 && nc != 16)) return 0;
    int n[MAX_CT_LEVELS][3];
    for (int l = 0; l < nlev; l++)
        for (int a = 0; a < 3; a++) n[l][a] = ops[l].n[a];
    unsigned off[MAX_CT_LEVELS][8], obc = 0, ominv = 0;
    const size_t es = sizeof(typename CT<R>::T);
    const size_t bytes = mg_ctail_layout(dim, es, nlev, n, nc, nu_c, off, &obc, &ominv);
    if (bytes > CT_SMEM_BYTES) return 0;
    int B[MAX_CT_LEVELS][MAX_CT_BLOCKS + 1];
    if (!mg_ctail_bounds(dim, nlev, n, nc, B)) return 0;
    A = CArgs<R>{};
    for (int l = 0; l < nlev; l++) {
        CLevel<R> &L = A.lv[l];
        for (int a = 0; a < 3; a++) L.cf[a] = ops[l].coef[a];
        L.k2 = ops[l].k2;
        L.bk = ops[l].bk;
        L.c = ops[l].c;
        L.nx = n[l][0];
        L.ny = dim == 3 ? n[l][1] : 1;
        for (int r = 0; r <= MAX_CT_BLOCKS; r++) L.B[r] = B[l][std::min(r, nc)];
        L.ob = off[l][0]; L.ou = off[l][1]; L.ot = off[l][2]; L.ok = off[l][3]; L.oi = off[l][4];
        L.ocx = off[l][5]; L.ocy = off[l][6]; L.ocs = off[l][7];
    }
    A.nlev = nlev;
    A.nu_c = nu_c;
    A.omega = omega;
    A.minv = minv;
    A.obc = obc;
    A.ominv = ominv;
    A.mrow = mg_ctail_minv_stage_bytes(nc, nu_c, es) ? mg_ctail_minv_rows(nc, nu_c) : 0;
    A.total = (unsigned)bytes;
    return bytes;
}

template <typename R>
cudaError_t build_mg_ctail_image(int dim, int nlev, const DevOp<R> *ops, const typename CT<R>::T *minv, int nu_c,
                                 R omega, int nc, void **out, cudaStream_t s) {
    *out = nullptr;
    CArgs<R> A;
    const size_t bytes = ct_args<R>(dim, nlev, ops, minv, nu_c, omega, nc, A);
    if (!bytes) return cudaErrorInvalidValue;
    void *img = nullptr;
    cudaError_t e = cudaMalloc(&img, bytes * nc);
    if (e != cudaSuccess) return e;
    if (dim == 3) k_ctail_image<R, 3><<<nc, CT_THREADS, 0, s>>>(A, (unsigned char *)img);
    else k_ctail_image<R, 2><<<nc, CT_THREADS, 0, s>>>(A, (unsigned char *)img);
    if ((e = cudaGetLastError()) != cudaSuccess) {
        cudaFree(img);
        return e;
    }
    *out = img;
    return cudaSuccess;
}
template cudaError_t build_mg_ctail_image<float>(int, int, const DevOp<float> *, const float2 *, int, float, int,
                                                 void **, cudaStream_t);
template cudaError_t build_mg_ctail_image<double>(int, int, const DevOp<double> *, const double2 *, int, double, int,
                                                  void **, cudaStream_t);

// Attributes that a cluster launch of the kernel needs (set on the current device).
template <typename K> static cudaError_t cluster_attributes(K kernel, int nc) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CT_SMEM_BYTES);
    if (e == cudaSuccess && nc > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

// Launch configuration of `count` clusters of nc blocks (attributes stored in at[2]).
static cudaLaunchConfig_t cluster_config(int nc, int count, size_t bytes, cudaStream_t s, cudaLaunchAttribute *at,
                                         bool pdl) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(nc, 1, count);
    cfg.blockDim = dim3(CT_THREADS, 1, 1);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = nc;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 2 : 1;
    return cfg;
}

template <typename R, int DIM>
static cudaError_t launch_ct(int nc, size_t bytes, const CArgs<R> &A, cudaStream_t s) {
    static bool attr[2] = {false, false};
    const int ai = nc == 16;
    if (!attr[ai]) {
        const cudaError_t e = cluster_attributes(k_mg_ctail<R, DIM>, nc);
        if (e != cudaSuccess) return e;
        attr[ai] = true;
    }
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t cfg = cluster_config(nc, 1, bytes, s, at, pdl_enabled());
    return cudaLaunchKernelEx(&cfg, k_mg_ctail<R, DIM>, A);
}

template <typename R>
cudaError_t launch_mg_ctail(int dim, int nlev, const DevOp<R> *ops, const typename CT<R>::T *b_top,
                            typename CT<R>::T *u_top, const typename CT<R>::T *minv, int nu_c, int nu1, int nu2, int rb,
                            R omega, int zero, int gf, int gc, int nc, const void *img, cudaStream_t s) {
    CArgs<R> A;
    const size_t bytes = ct_args<R>(dim, nlev, ops, minv, nu_c, omega, nc, A);
    if (!bytes) return cudaErrorInvalidValue;
    A.nu1 = nu1;
    A.nu2 = nu2;
    A.rb = rb;
    A.zero = zero;
    A.b_top = b_top;
    A.u_top = u_top;
    A.gf = gf;
    A.gc = gc;
    A.img = (const float4 *)img;
    return dim == 3 ? launch_ct<R, 3>(nc, bytes, A, s) : launch_ct<R, 2>(nc, bytes, A, s);
}
template cudaError_t launch_mg_ctail<float>(int, int, const DevOp<float> *, const float2 *, float2 *, const float2 *,
                                            int, int, int, int, float, int, int, int, int, const void *, cudaStream_t);
template cudaError_t launch_mg_ctail<double>(int, int, const DevOp<double> *, const double2 *, double2 *,
                                             const double2 *, int, int, int, int, double, int, int, int, int,
                                             const void *, cudaStream_t);

// Batched tail over count problems whose tail levels have the shapes of ops (every problem's
// own pointers and prebuilt image in tab); one cluster of nc blocks per problem.
cudaError_t launch_mg_ctail_batch(int nlev, const DevOp<float> *ops, int nu_c, int nu1, int nu2, int rb, float omega,
                                  int gf, int gc, int nc, int count, const BTail *tab, int j, cudaStream_t s) {
    if (count < 1 || count > 65535) return cudaErrorInvalidValue;
    CArgs<float> A;
    const size_t bytes = ct_args<float>(2, nlev, ops, nullptr, nu_c, omega, nc, A);
    if (!bytes) return cudaErrorInvalidValue;
    A.nu1 = nu1;
    A.nu2 = nu2;
    A.rb = rb;
    A.zero = 1;
    A.gf = gf;
    A.gc = gc;
    static bool attr[2] = {false, false};
    const int ai = nc == 16;
    if (!attr[ai]) {
        const cudaError_t e = cluster_attributes(k_mg_ctail_b, nc);
        if (e != cudaSuccess) return e;
        attr[ai] = true;
    }
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t cfg = cluster_config(nc, count, bytes, s, at, pdl_enabled());
    return cudaLaunchKernelEx(&cfg, k_mg_ctail_b, A, tab, j);
}

// Clusters of nc blocks with the given shared memory that the device can run at once (0: the
// configuration cannot be launched).
template <typename R>
int mg_ctail_max_clusters(int dim, int nc, size_t bytes) {
    if (bytes > CT_SMEM_BYTES) return 0;
    auto count = [&](auto kernel) {
        if (cluster_attributes(kernel, nc) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        cudaLaunchAttribute at[2];
        cudaLaunchConfig_t cfg = cluster_config(nc, 1, bytes, 0, at, false);
        int c = 0;
        if (cudaOccupancyMaxActiveClusters(&c, kernel, &cfg) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        return c;
    };
    return dim == 3 ? count(k_mg_ctail<R, 3>) : count(k_mg_ctail<R, 2>);
}
template int mg_ctail_max_clusters<float>(int, int, size_t);
template int mg_ctail_max_clusters<double>(int, int, size_t);
