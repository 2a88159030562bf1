// Stencil and multigrid kernels for the ECS Helmholtz operators (sm_103a).
//
// Operator (Section 3.2 FD formula for unequal complex widths, summed over axes, with the
// operator coefficients of Section 5 folded in):
//   (M x)_p = sum_axes (cw x_{p-e} + cc x_p + ce x_{p+e}) + (bk k2_p + c) x_p.
// Multigrid components (Section 4.2): omega-Jacobi, omega-red-black Jacobi, full-weighting
// restriction fused with the residual, bi/trilinear prolongation fused with the correction,
// and the exact coarsest solve (Algorithm 1 step (0)) as a dense-inverse product.
//
// Layout: interleaved complex node arrays, x fastest, boundary included (never written).
// Threads: 2D blocks of 32 x 8 over (i, j); in 3D every thread marches a chunk of k planes
// keeping the x[p - nx ny], x[p], x[p + nx ny] column in registers.  Every launch covers the
// interior only, so no thread touches a boundary node's value except as a stencil neighbour.
#include "helm_internal.h"
#include "restrict_turns.h"

namespace {

constexpr int BX = 32, BY = 8, KCHUNK = 8;

template <typename R> struct OpView {
    typedef typename CT<R>::T C;
    const C *__restrict__ cx;
    const C *__restrict__ cy;
    const C *__restrict__ cz;
    const R *__restrict__ k2;
    const C *__restrict__ dinv;
    C bk, c;
    int nx, ny, nz;
    const int *gate;  // see DevOp::gate
};

template <typename R> __host__ __device__ OpView<R> view(const DevOp<R> &op) {
    OpView<R> v;
    v.cx = op.coef[0]; v.cy = op.coef[1]; v.cz = op.coef[2];
    v.k2 = op.k2; v.dinv = op.dinv; v.bk = op.bk; v.c = op.c; v.gate = op.gate;
    v.nx = op.n[0]; v.ny = op.n[1]; v.nz = op.n[2];
    return v;
}

// Off-diagonal part of the stencil at p (neighbours along x and y; z handled by callers that
// march in k).
template <typename R, int DIM, typename CX>
__device__ __forceinline__ typename CT<R>::T offdiag(const OpView<R> &o, const CX *__restrict__ x, size_t p, int i,
                                                    int j, int k, typename CT<R>::T xm_z, typename CT<R>::T xp_z) {
    typedef typename CT<R>::T C;
    const size_t sy = (size_t)o.nx;
    C acc = cmul(__ldg(&o.cx[3 * i]), to_c(x[p - 1], R()));
    acc = cfma(__ldg(&o.cx[3 * i + 2]), to_c(x[p + 1], R()), acc);
    acc = cfma(__ldg(&o.cy[3 * j]), to_c(x[p - sy], R()), acc);
    acc = cfma(__ldg(&o.cy[3 * j + 2]), to_c(x[p + sy], R()), acc);
    if (DIM == 3) {
        acc = cfma(__ldg(&o.cz[3 * k]), xm_z, acc);
        acc = cfma(__ldg(&o.cz[3 * k + 2]), xp_z, acc);
    }
    return acc;
}

// (M x)_p and the diagonal entry.
template <typename R, int DIM, typename CX>
__device__ __forceinline__ typename CT<R>::T stencil(const OpView<R> &o, const CX *__restrict__ x, size_t p,
                                                    int i, int j, int k, typename CT<R>::T xm_z,
                                                    typename CT<R>::T xc, typename CT<R>::T xp_z,
                                                    typename CT<R>::T &diag) {
    typedef typename CT<R>::T C;
    const C acc = offdiag<R, DIM>(o, x, p, i, j, k, xm_z, xp_z);
    C d = cadd(__ldg(&o.cx[3 * i + 1]), __ldg(&o.cy[3 * j + 1]));
    if (DIM == 3) d = cadd(d, __ldg(&o.cz[3 * k + 1]));
    d = cadd(d, cadd(cscale(o.bk, o.k2[p]), o.c));
    diag = d;
    return cfma(d, xc, acc);
}

// (M x)_p for a point whose z neighbours are loaded here (used by the restriction kernel).
template <typename R, int DIM, typename CX>
__device__ __forceinline__ typename CT<R>::T apply_point(const OpView<R> &o, const CX *__restrict__ x, int i, int j,
                                                        int k, typename CT<R>::T &diag) {
    typedef typename CT<R>::T C;
    const size_t sz = (size_t)o.nx * o.ny;
    const size_t p = (size_t)i + (size_t)o.nx * ((size_t)j + (size_t)o.ny * k);
    C xm = mk(R(0), R(0)), xp = mk(R(0), R(0));
    if (DIM == 3) { xm = to_c(x[p - sz], R()); xp = to_c(x[p + sz], R()); }
    return stencil<R, DIM, CX>(o, x, p, i, j, k, xm, to_c(x[p], R()), xp, diag);
}

// Thread preamble: interior (i, j) and the k range of this thread.
#define INTERIOR_IJ(o)                                              \
    const int i = blockIdx.x * BX + threadIdx.x + 1;                \
    const int j = blockIdx.y * BY + threadIdx.y + 1;                \
    if (i > (o).nx - 2 || j > (o).ny - 2) return;                   \
    int k0 = 0, k1 = 1;                                             \
    if (DIM == 3) {                                                 \
        k0 = blockIdx.z * KCHUNK + 1;                               \
        k1 = min(k0 + KCHUNK, (o).nz - 1);                          \
    }                                                               \
    const size_t sz = (size_t)(o).nx * (o).ny;                      \
    size_t p = (size_t)i + (size_t)(o).nx * ((size_t)j + (size_t)(o).ny * k0);

// y = M x, or with RES y = b - M x; each thread marches kc planes in 3D with its x and y coefficients
// in registers.  complex128 is bound by the FP64 units (two lanes per SM and clock): 36 operations per
// node in 3D, but 16 where every axis is outside the layers, since those coefficients of A are real.
// Each warp picks the form by axis (x: all its columns, y: its row, z: runs of its planes), outside the
// loop, so that every form is a loop of its own.  Measured, A x in complex128 on 225 x 193 x 161 nodes: 406 us with
// every term complex, 318 us so (543 us with the form chosen by a branch at every node).
template <typename R, int DIM, typename CX, typename CB, bool RES, bool RX, bool RY, bool RZ>
__device__ __forceinline__ void apply_march(const OpView<R> &o, const CB *__restrict__ b, const CX *__restrict__ x,
                                            typename CT<R>::T *__restrict__ y, int i, int j, int k0, int k1) {
    typedef typename CT<R>::T C;
    constexpr bool RD = RX && RY && RZ;
    const size_t sy = (size_t)o.nx, sz = sy * o.ny;
    size_t p = (size_t)i + sy * ((size_t)j + (size_t)o.ny * k0);
    const C cwx = __ldg(&o.cx[3 * i]), cex = __ldg(&o.cx[3 * i + 2]), cwy = __ldg(&o.cy[3 * j]), cey = __ldg(&o.cy[3 * j + 2]);
    const C dxy = cadd(cadd(__ldg(&o.cx[3 * i + 1]), __ldg(&o.cy[3 * j + 1])), o.c);
    C xm = mk(R(0), R(0)), xc = to_c(x[p], R()), xp = xm;
    if (DIM == 3) xm = to_c(x[p - sz], R());
    for (int k = k0; k < k1; k++, p += sz) {
        if (DIM == 3) xp = to_c(x[p + sz], R());
        const R kq = o.k2[p];
        C d = dxy, acc = mk(R(0), R(0));
        if (DIM == 3) {
            const C ccz = __ldg(&o.cz[3 * k + 1]);
            d = RD ? mk(d.x + ccz.x, R(0)) : cadd(d, ccz);
            acc = axis_add<RZ>(__ldg(&o.cz[3 * k]), __ldg(&o.cz[3 * k + 2]), xm, xp, acc);
        }
        acc = axis_add<RX>(cwx, cex, to_c(x[p - 1], R()), to_c(x[p + 1], R()), acc);
        acc = axis_add<RY>(cwy, cey, to_c(x[p - sy], R()), to_c(x[p + sy], R()), acc);
        d.x = fma(o.bk.x, kq, d.x);
        if (RD) {
            acc = mk(fma(d.x, xc.x, acc.x), fma(d.x, xc.y, acc.y));
        } else {
            d.y = fma(o.bk.y, kq, d.y);
            acc = cfma(d, xc, acc);
        }
        y[p] = RES ? csub(to_c(b[p], R()), acc) : acc;
        if (DIM == 3) { xm = xc; xc = xp; }
    }
}

template <typename R, int DIM, typename CX, typename CB, bool RES>
__global__ void __launch_bounds__(BX *BY) k_apply(OpView<R> o, const CB *__restrict__ b, const CX *__restrict__ x,
                                                  typename CT<R>::T *__restrict__ y, int kc) {
    pdl_enter();
    if (RES && o.gate && *o.gate) return;
    const int i = blockIdx.x * BX + threadIdx.x + 1;
    const int j = blockIdx.y * BY + threadIdx.y + 1;
    if (i > o.nx - 2 || j > o.ny - 2) return;
    int k0 = 0, k1 = 1;
    if (DIM == 3) {
        k0 = blockIdx.z * kc + 1;
        k1 = min(k0 + kc, o.nz - 1);
    }
    if constexpr (sizeof(R) == sizeof(double)) {
        auto real3 = [](const double2 *t) {
            return is_zero(__ldg(&t[0].y)) && is_zero(__ldg(&t[1].y)) && is_zero(__ldg(&t[2].y));
        };
        if (is_zero(o.bk.y) && is_zero(o.c.y)) {
            const bool rx = __all_sync(__activemask(), real3(o.cx + 3 * i)), ry = real3(o.cy + 3 * j);
            if constexpr (DIM == 2) {
                if (rx && ry) return apply_march<R, DIM, CX, CB, RES, true, true, true>(o, b, x, y, i, j, 0, 1);
                if (rx) return apply_march<R, DIM, CX, CB, RES, true, false, true>(o, b, x, y, i, j, 0, 1);
                if (ry) return apply_march<R, DIM, CX, CB, RES, false, true, true>(o, b, x, y, i, j, 0, 1);
            } else {
                // runs of planes that are all real or all not
                for (int k = k0, e; k < k1; k = e) {
                    const bool rz = real3(o.cz + 3 * k);
                    e = k + 1;
                    while (e < k1 && real3(o.cz + 3 * e) == rz) e++;
                    if (rx && ry && rz) apply_march<R, DIM, CX, CB, RES, true, true, true>(o, b, x, y, i, j, k, e);
                    else if (rx && ry) apply_march<R, DIM, CX, CB, RES, true, true, false>(o, b, x, y, i, j, k, e);
                    else if (rx && rz) apply_march<R, DIM, CX, CB, RES, true, false, true>(o, b, x, y, i, j, k, e);
                    else if (ry && rz) apply_march<R, DIM, CX, CB, RES, false, true, true>(o, b, x, y, i, j, k, e);
                    else if (rx) apply_march<R, DIM, CX, CB, RES, true, false, false>(o, b, x, y, i, j, k, e);
                    else if (ry) apply_march<R, DIM, CX, CB, RES, false, true, false>(o, b, x, y, i, j, k, e);
                    else if (rz) apply_march<R, DIM, CX, CB, RES, false, false, true>(o, b, x, y, i, j, k, e);
                    else apply_march<R, DIM, CX, CB, RES, false, false, false>(o, b, x, y, i, j, k, e);
                }
                return;
            }
        }
        apply_march<R, DIM, CX, CB, RES, false, false, false>(o, b, x, y, i, j, k0, k1);
    } else {
        // bound by memory: the coefficients come from L1 at every node, which leaves the loads of a
        // plane more room (257 x 225 x 257 nodes: 70.5 us with the x and y coefficients in registers, 67.6 so)
        typedef typename CT<R>::T C;
        const size_t sz = (size_t)o.nx * o.ny;
        size_t p = (size_t)i + (size_t)o.nx * ((size_t)j + (size_t)o.ny * k0);
        C xm = mk(R(0), R(0)), xc = to_c(x[p], R()), xp = mk(R(0), R(0)), d;
        if (DIM == 3) xm = to_c(x[p - sz], R());
        for (int k = k0; k < k1; k++, p += sz) {
            if (DIM == 3) xp = to_c(x[p + sz], R());
            const C v = stencil<R, DIM>(o, x, p, i, j, k, xm, xc, xp, d);
            y[p] = RES ? csub(to_c(b[p], R()), v) : v;
            if (DIM == 3) { xm = xc; xc = xp; }
        }
    }
}

// omega-Jacobi: every unknown from the previous iterate (ping-pong buffers).
template <typename R, int DIM, typename CB, bool ZERO>
__global__ void __launch_bounds__(BX *BY) k_jacobi(OpView<R> o, R omega, const CB *__restrict__ b, const typename CT<R>::T *__restrict__ u,
                                                   typename CT<R>::T *__restrict__ un) {
    pdl_enter();
    if (o.gate && *o.gate) return;
    typedef typename CT<R>::T C;
    INTERIOR_IJ(o);
    if (ZERO) {
        for (int k = k0; k < k1; k++, p += sz) {
            if constexpr (sizeof(R) == sizeof(double)) {
                un[p] = cmul(to_c(b[p], R()), o.dinv[p]);
                continue;
            }
            C d;
            // diagonal only: the stencil of the zero vector
            d = cadd(cadd(__ldg(&o.cx[3 * i + 1]), __ldg(&o.cy[3 * j + 1])), cadd(cscale(o.bk, o.k2[p]), o.c));
            if (DIM == 3) d = cadd(d, __ldg(&o.cz[3 * k + 1]));
            un[p] = cscale(cmul(to_c(b[p], R()), cinv(d)), omega);
        }
        return;
    }
    C xm = mk(R(0), R(0)), xc = u[p], xp = mk(R(0), R(0));
    if (DIM == 3) xm = u[p - sz];
    for (int k = k0; k < k1; k++, p += sz) {
        if (DIM == 3) xp = u[p + sz];
        if constexpr (sizeof(R) == sizeof(double)) {
            const C r = csub(to_c(b[p], R()), offdiag<R, DIM>(o, u, p, i, j, k, xm, xp));
            un[p] = cfma(o.dinv[p], r, cscale(xc, R(1) - omega));
        } else {
            C d;
            C mu = stencil<R, DIM>(o, u, p, i, j, k, xm, xc, xp, d);
            C res = csub(to_c(b[p], R()), mu);
            un[p] = cadd(xc, cscale(cmul(res, cinv(d)), omega));
        }
        if (DIM == 3) { xm = xc; xc = xp; }
    }
}

// 3D omega-Jacobi: k_jacobi's arithmetic in the same order, with the x and y coefficient
// triples loaded once per thread, the (z - 1, z, z + 1) column in registers, and the next plane's
// operands (four in-plane neighbours, z + 2, b, k^2) loaded while this plane is computed.
// KC: fine planes per thread (shorter chunks on small grids give more blocks; at most 16 against
// at most 8 on 257^3: 690 against 694 us per cycle).  ZERO with a complex128 b
// in a complex64 cycle: the sweep also writes b rounded to complex64 to b_out.
template <typename R, typename CB, bool ZERO, int KC>
__global__ void __launch_bounds__(BX *BY) k_jacobi3(OpView<R> o, R omega, const CB *__restrict__ b,
                                                    const typename CT<R>::T *__restrict__ u,
                                                    typename CT<R>::T *__restrict__ un,
                                                    typename CT<R>::T *__restrict__ b_out) {
    pdl_enter();
    const int gv = gate_value(o.gate);
    typedef typename CT<R>::T C;
    const int i = blockIdx.x * BX + threadIdx.x + 1;
    const int j = blockIdx.y * BY + threadIdx.y + 1;
    if (i > o.nx - 2 || j > o.ny - 2) return;
    const int k0 = blockIdx.z * KC + 1, k1 = min(k0 + KC, o.nz - 1);
    const size_t sz = (size_t)o.nx * o.ny;
    size_t p = (size_t)i + (size_t)o.nx * ((size_t)j + (size_t)o.ny * k0);
    const size_t sy = (size_t)o.nx;
    const C cwx = __ldg(&o.cx[3 * i]), ccx = __ldg(&o.cx[3 * i + 1]), cex = __ldg(&o.cx[3 * i + 2]);
    const C cwy = __ldg(&o.cy[3 * j]), ccy = __ldg(&o.cy[3 * j + 1]), cey = __ldg(&o.cy[3 * j + 2]);
    C bq = to_c(b[p], R());
    if constexpr (sizeof(R) == sizeof(double)) {
        // complex128: bound by the FP64 units, so the sweep takes omega / D as formed once
        // (34 operations per node instead of about 67)
        C wq = o.dinv[p];
        if (gv) return;
        if (ZERO) {
            for (int k = k0; k < k1; k++, p += sz) un[p] = cmul(to_c(b[p], R()), o.dinv[p]);
            return;
        }
        C xm = u[p - sz], xc = u[p], xp = u[p + sz];
        for (int k = k0; k < k1; k++, p += sz) {
            C xp2 = xp, bn = bq, wn = wq;
            const C xw = u[p - 1], xe = u[p + 1], xs = u[p - sy], xn = u[p + sy];
            if (k + 1 < k1) {
                xp2 = u[p + 2 * sz];
                bn = to_c(b[p + sz], R());
                wn = o.dinv[p + sz];
            }
            C acc = cmul(cwx, xw);
            acc = cfma(cex, xe, acc);
            acc = cfma(cwy, xs, acc);
            acc = cfma(cey, xn, acc);
            acc = cfma(__ldg(&o.cz[3 * k]), xm, acc);
            acc = cfma(__ldg(&o.cz[3 * k + 2]), xp, acc);
            un[p] = cfma(wq, csub(bq, acc), cscale(xc, R(1) - omega));
            xm = xc;
            xc = xp;
            xp = xp2; bq = bn; wq = wn;
        }
        return;
    } else {
    R kq = o.k2[p];
    if (gv) return;
    if (ZERO) {
        const C dxy = cadd(ccx, ccy);
        for (int k = k0; k < k1; k++, p += sz) {
            C bn = bq;
            R kn = kq;
            if (k + 1 < k1) {
                bn = to_c(b[p + sz], R());
                kn = o.k2[p + sz];
            }
            const C d = cadd(cadd(dxy, cadd(cscale(o.bk, kq), o.c)), __ldg(&o.cz[3 * k + 1]));
            if (sizeof(CB) != sizeof(C)) b_out[p] = bq;  // b is complex128: keep what the sweep used
            un[p] = cscale(cmul(bq, cinv(d)), omega);
            bq = bn;
            kq = kn;
        }
        return;
    }
    C xm = u[p - sz], xc = u[p], xp = u[p + sz];
    C xw = u[p - 1], xe = u[p + 1], xs = u[p - sy], xn = u[p + sy];
    for (int k = k0; k < k1; k++, p += sz) {
        C xw2 = xw, xe2 = xe, xs2 = xs, xn2 = xn, xp2 = xp, bn = bq;
        R kn = kq;
        if (k + 1 < k1) {
            const size_t q = p + sz;
            xw2 = u[q - 1];
            xe2 = u[q + 1];
            xs2 = u[q - sy];
            xn2 = u[q + sy];
            xp2 = u[q + sz];
            bn = to_c(b[q], R());
            kn = o.k2[q];
        }
        // the lines two planes ahead into L2 (257^3: 690 us per cycle with them, 734 without; further
        // ahead or in the residual kernel no gain)
        if (k + 2 < k1 && (threadIdx.x & 15) == 0) {
            const size_t q = p + 2 * sz;
            l2_prefetch(&u[q + sz]);
            l2_prefetch(&b[q]);
            l2_prefetch(&o.k2[q]);
        }
        C acc = cmul(cwx, xw);
        acc = cfma(cex, xe, acc);
        C d = ccx;
        acc = cfma(cwy, xs, acc);
        acc = cfma(cey, xn, acc);
        d = cadd(d, ccy);
        const C czw = __ldg(&o.cz[3 * k]), czc = __ldg(&o.cz[3 * k + 1]), cze = __ldg(&o.cz[3 * k + 2]);
        acc = cfma(czw, xm, acc);
        acc = cfma(cze, xp, acc);
        d = cadd(d, czc);
        d = cadd(d, cadd(cscale(o.bk, kq), o.c));
        const C mu = cfma(d, xc, acc);
        const C res = csub(bq, mu);
        un[p] = cadd(xc, cscale(cmul(res, cinv(d)), omega));
        xm = xc;
        xc = xp;
        xw = xw2; xe = xe2; xs = xs2; xn = xn2; xp = xp2; bq = bn; kq = kn;
    }
    }  // complex64
}

// one colour of omega-red-black Jacobi, in place: threads map to every other x node and march kc
// planes.  FROM: the iterate on entry is given (RB_ANY), zero everywhere and not read (RB_ZERO: the
// first colour of a sweep from zero is pointwise), or zero on this colour, or omega = 1, and not read
// there (RB_NO_OWN: the second colour of a sweep from zero, any colour with omega = 1).  complex128 takes omega / D as formed once (see k_jacobi3).
// Measured, 193 x 129 x 97 complex128 V(1,1) cycle: 1318 us with the diagonal assembled and divided by
// at every node, a zero fill before the first sweep and chunks of 8 planes on every level, 719 us so.
enum { RB_ANY, RB_ZERO, RB_NO_OWN };
template <typename R, int DIM, typename CB, int FROM>
__global__ void __launch_bounds__(BX *BY) k_rb(OpView<R> o, R omega, const CB *__restrict__ b, typename CT<R>::T *u, int colour,
                                               int kc) {
    pdl_enter();
    if (o.gate && *o.gate) return;
    typedef typename CT<R>::T C;
    const int t = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y + 1;
    if (j > o.ny - 2) return;
    int k0 = 0, k1 = 1;
    if (DIM == 3) { k0 = blockIdx.z * kc + 1; k1 = min(k0 + kc, o.nz - 1); }
    const size_t sz = (size_t)o.nx * o.ny;
#pragma unroll 2
    for (int k = k0; k < k1; k++) {
        const int i = 2 * t + 1 + ((1 + j + k + colour) & 1);
        if (i > o.nx - 2) continue;
        const size_t p = (size_t)i + (size_t)o.nx * ((size_t)j + (size_t)o.ny * k);
        C xm = mk(R(0), R(0)), xp = xm, xc = xm, w, acc = xm;
        if (FROM != RB_ZERO && DIM == 3) { xm = u[p - sz]; xp = u[p + sz]; }
        if (FROM == RB_ANY) xc = u[p];
        if constexpr (sizeof(R) == sizeof(double)) {
            w = o.dinv[p];
        } else {
            C d = cadd(__ldg(&o.cx[3 * i + 1]), __ldg(&o.cy[3 * j + 1]));
            if (DIM == 3) d = cadd(d, __ldg(&o.cz[3 * k + 1]));
            w = cscale(cinv(cadd(d, cadd(cscale(o.bk, o.k2[p]), o.c))), omega);
        }
        C r = to_c(b[p], R());
        if (FROM != RB_ZERO) r = csub(r, offdiag<R, DIM>(o, u, p, i, j, k, xm, xp));
        u[p] = FROM == RB_ANY ? cfma(w, r, cscale(xc, R(1) - omega)) : cmul(w, r);
    }
}

// rc[I] = sum_{d in {-1,0,1}^DIM} prod w(d) (b - M u)[2I + d],  w(0) = 1/2, w(+-1) = 1/4.
template <typename R, int DIM, typename CB>
__global__ void __launch_bounds__(BX *BY) k_residual_restrict(OpView<R> o, const CB *__restrict__ b, const typename CT<R>::T *__restrict__ u,
                                                              typename CT<R>::T *__restrict__ rc, int ncx, int ncy, int ncz) {
    pdl_enter();
    if (o.gate && *o.gate) return;
    typedef typename CT<R>::T C;
    const int I = blockIdx.x * BX + threadIdx.x + 1;
    const int J = blockIdx.y * BY + threadIdx.y + 1;
    if (I > ncx - 2 || J > ncy - 2) return;
    int K0 = 0, K1 = 1;
    if (DIM == 3) { K0 = blockIdx.z * KCHUNK + 1; K1 = min(K0 + KCHUNK, ncz - 1); }
    for (int K = K0; K < K1; K++) {
        C acc = mk(R(0), R(0));
        const int dk0 = DIM == 3 ? -1 : 0, dk1 = DIM == 3 ? 1 : 0;
        for (int dk = dk0; dk <= dk1; dk++) {
            const R wk = DIM == 3 ? (dk == 0 ? R(0.5) : R(0.25)) : R(1);
            const int k = DIM == 3 ? 2 * K + dk : 0;
#pragma unroll
            for (int dj = -1; dj <= 1; dj++) {
                const R wj = wk * (dj == 0 ? R(0.5) : R(0.25));
                const int j = 2 * J + dj;
#pragma unroll
                for (int di = -1; di <= 1; di++) {
                    const R w = wj * (di == 0 ? R(0.5) : R(0.25));
                    const int i = 2 * I + di;
                    const size_t p = (size_t)i + (size_t)o.nx * ((size_t)j + (size_t)o.ny * k);
                    C d;
                    C mu = apply_point<R, DIM>(o, u, i, j, k, d);
                    acc = cadd(acc, cscale(csub(to_c(b[p], R()), mu), w));
                }
            }
        }
        rc[(size_t)I + (size_t)ncx * ((size_t)J + (size_t)ncy * K)] = acc;
    }
}

// uf[q] += average of ec over coarse nodes floor(q/2), ceil(q/2) along every axis.
template <typename R, int DIM>
__global__ void __launch_bounds__(BX *BY) k_prolong_add(int nx, int ny, int nz, const typename CT<R>::T *__restrict__ ec,
                                                        typename CT<R>::T *__restrict__ uf,
                                                        const int *__restrict__ gate) {
    pdl_enter();
    if (gate && *gate) return;
    typedef typename CT<R>::T C;
    const int i = blockIdx.x * BX + threadIdx.x + 1;
    const int j = blockIdx.y * BY + threadIdx.y + 1;
    if (i > nx - 2 || j > ny - 2) return;
    const int ncx = (nx + 1) / 2, ncy = (ny + 1) / 2;
    int k0 = 0, k1 = 1;
    if (DIM == 3) { k0 = blockIdx.z * KCHUNK + 1; k1 = min(k0 + KCHUNK, nz - 1); }
    const int i0 = i >> 1, i1 = (i + 1) >> 1, j0 = j >> 1, j1 = (j + 1) >> 1;
    for (int k = k0; k < k1; k++) {
        const int kk0 = DIM == 3 ? k >> 1 : 0, kk1 = DIM == 3 ? (k + 1) >> 1 : 0;
        C acc = mk(R(0), R(0));
        int cnt = 0;
        for (int kk = kk0; kk <= kk1; kk++)
            for (int jj = j0; jj <= j1; jj++)
                for (int ii = i0; ii <= i1; ii++) {
                    acc = cadd(acc, ec[(size_t)ii + (size_t)ncx * ((size_t)jj + (size_t)ncy * kk)]);
                    cnt++;
                }
        const size_t p = (size_t)i + (size_t)nx * ((size_t)j + (size_t)ny * k);
        uf[p] = cadd(uf[p], cscale(acc, R(1) / R(cnt)));
    }
}

// 3D residual + full weighting, each fine residual computed once.  A block owns R3_TX x R3_TY
// coarse nodes in (x, y) and kc coarse planes (at most R3_KC); one thread per fine node of the region those
// coarse nodes weigh ((2 R3_TX + 1) x (2 R3_TY + 1)) marches the block's fine planes
// 2 K0 - 1 .. 2 K1 - 1 like k_jacobi3 (coefficients in registers, the u column (z - 1, z, z + 1)
// in registers, the next plane's operands loaded while this plane is computed).  Each thread weighs its
// own residuals by (1, 2, 1) along z in registers; once per coarse plane the weighted plane goes through
// shared memory and the coarse nodes' threads apply (1, 2, 1) in x and y.  The four groups of four warps
// take turns at that sum: a group waits for the plane in its own turn only and merely arrives at the
// barrier in the others' (restrict_turns.h), so that the sum does not hold up the march of the other
// warps.  Five shared planes for the four turns: every warp then waits in a turn of its own between a
// group's reads of a plane and its own next store into it.  (257^3 complex64: 120 us
// per launch on the finest level and 690 us per cycle; 702 us with every warp waiting at every plane.)  An
// odd fine plane 2K + 1 completes coarse plane K and starts K + 1.  Fine nodes outside the grid's interior
// hold zero residuals.  Same weights as k_residual_restrict, applied per axis.
constexpr int R3_TX = 16, R3_TY = 8, R3_KC = 8;
constexpr int R3_FW = 2 * R3_TX + 1, R3_FH = 2 * R3_TY + 1;  // fine region
constexpr int R3_NT = ((R3_FW * R3_FH + 31) / 32) * 32;       // threads: one per region node
template <typename R> constexpr size_t r3_smem_bytes(int planes) {
    return (size_t)planes * R3_FW * R3_FH * sizeof(typename CT<R>::T);
}

template <typename R, typename CB>
__global__ void __launch_bounds__(R3_NT, sizeof(R) == sizeof(float) ? 2 : 1)
    k_resrestrict3(OpView<R> o, const CB *__restrict__ b, const typename CT<R>::T *__restrict__ u,
                   typename CT<R>::T *__restrict__ rc, int ncx, int ncy, int ncz, int kc) {
    pdl_enter();
    const int gv = gate_value(o.gate);
    typedef typename CT<R>::T C;
    extern __shared__ __align__(16) unsigned char r3_smem[];
    C(*rbuf)[R3_FH][R3_FW] = reinterpret_cast<C(*)[R3_FH][R3_FW]>(r3_smem);
    const int nx = o.nx, ny = o.ny;
    const int I0 = 1 + blockIdx.x * R3_TX, J0 = 1 + blockIdx.y * R3_TY;
    const int K0 = 1 + blockIdx.z * kc, K1 = min(K0 + kc, ncz - 1);
    const int t = threadIdx.x, lx = t % R3_FW, ly = t / R3_FW;
    const int x = 2 * I0 - 1 + lx, y = 2 * J0 - 1 + ly;
    // region nodes inside the grid's interior compute residuals; the others hold zeros
    const bool region = t < R3_FW * R3_FH, res = region && x <= nx - 2 && y <= ny - 2;
    const size_t sy = (size_t)nx, sz = (size_t)nx * ny;
    const int zs = 2 * K0 - 1, ze = 2 * K1 - 1;
    const C zero = mk(R(0), R(0));
    C cwx = zero, cex = zero, cwy = zero, cey = zero, dxy = zero;
    C xm = zero, xc = zero, xp = zero, xw = zero, xe = zero, xs = zero, xn = zero, bq = zero;
    R kq = R(0);
    size_t p = (size_t)x + sy * y + sz * zs;
    if (res) {
        cwx = __ldg(&o.cx[3 * x]); cex = __ldg(&o.cx[3 * x + 2]);
        cwy = __ldg(&o.cy[3 * y]); cey = __ldg(&o.cy[3 * y + 2]);
        dxy = cadd(cadd(__ldg(&o.cx[3 * x + 1]), __ldg(&o.cy[3 * y + 1])), o.c);
        xm = u[p - sz]; xc = u[p]; xp = u[p + sz];
        xw = u[p - 1]; xe = u[p + 1]; xs = u[p - sy]; xn = u[p + sy];
        bq = to_c(b[p], R());
        kq = o.k2[p];
    }
    if (gv) return;  // the same value in every thread: no barrier is left waiting
    // the coarse node this thread sums in its warp group's turns (warps 0 .. 15)
    const int group = r3_group(t >> 5), cn = t & 127, cx = cn % R3_TX, cy = cn / R3_TX, I = I0 + cx, J = J0 + cy;
    const bool own = t < 512 && I <= ncx - 2 && J <= ncy - 2;
    C acc = zero;  // z sum of this fine column for the current coarse plane
    for (int z = zs; z <= ze; z++, p += sz) {
        C r = zero;
        if (res) {
            C xw2 = xw, xe2 = xe, xs2 = xs, xn2 = xn, xp2 = xp, bn = bq;
            R kn = kq;
            if (z < ze) {
                const size_t q = p + sz;
                xw2 = u[q - 1];
                xe2 = u[q + 1];
                xs2 = u[q - sy];
                xn2 = u[q + sy];
                xp2 = u[q + sz];
                bn = to_c(b[q], R());
                kn = o.k2[q];
            }
            C a2 = cmul(cwx, xw);
            a2 = cfma(cex, xe, a2);
            a2 = cfma(cwy, xs, a2);
            a2 = cfma(cey, xn, a2);
            a2 = cfma(__ldg(&o.cz[3 * z]), xm, a2);
            a2 = cfma(__ldg(&o.cz[3 * z + 2]), xp, a2);
            const C ccz = __ldg(&o.cz[3 * z + 1]);
            const C d = mk(fma(o.bk.x, kq, dxy.x + ccz.x), fma(o.bk.y, kq, dxy.y + ccz.y));
            r = csub(bq, cfma(d, xc, a2));
            xm = xc;
            xc = xp;
            xw = xw2; xe = xe2; xs = xs2; xn = xn2; xp = xp2; bq = bn; kq = kn;
        }
        if (!(z & 1)) {
            acc = mk(fma(R(2), r.x, acc.x), fma(R(2), r.y, acc.y));
            continue;
        }
        // fine plane 2K + 1 (K = (z - 1) / 2) completes coarse plane K and starts K + 1
        const int K = (z - 1) >> 1;
        if (K >= K0) {
            const int turn = r3_turn(K - K0);
            C(*buf)[R3_FW] = rbuf[r3_plane(K - K0)];
            if (region) buf[ly][lx] = cadd(acc, r);
            if (turn != group) {
                asm volatile("bar.arrive %0, %1;" ::"r"(1 + turn), "n"(R3_NT) : "memory");
            } else {
                asm volatile("bar.sync %0, %1;" ::"r"(1 + turn), "n"(R3_NT) : "memory");
                if (own) {
                    // (1, 2, 1) along x on the three fine rows 2J - 1 .. 2J + 1, then along y
                    C a[3];
#pragma unroll
                    for (int dy = 0; dy < 3; dy++) {
                        const C *row = &buf[2 * cy + dy][2 * cx];
                        a[dy] = cadd(cadd(row[0], row[2]), cscale(row[1], R(2)));
                    }
                    rc[(size_t)I + (size_t)ncx * ((size_t)J + (size_t)ncy * K)] =
                        cscale(cadd(cadd(a[0], a[2]), cscale(a[1], R(2))), R(1.0 / 64.0));
                }
            }
        }
        acc = r;
    }
}

// 3D residual + full weighting after a red-black sweep with omega = 1, whose second colour (odd
// i + j + k) ends with zero residuals: only the first colour's residuals are formed, one thread per
// red node of a plane of the region (the same tiles as k_resrestrict3), and the weights take only
// them.  first: the sweep was the first from zero, so D u = b at the red nodes and their residual is
// minus the off-diagonal part.  Bound by the FP64 units in complex128: 28 (first) or 36 operations for
// half of the nodes.
// Measured, 193 x 129 x 97 complex128 V(1,1) cycle: 719 us with every residual formed (277 us of it on
// the finest level), 505 us so.
constexpr int R3R_HW = R3_TX + 1, R3R_NT = ((R3R_HW * R3_FH + 31) / 32) * 32;
template <typename R, typename CB>
__global__ void __launch_bounds__(R3R_NT, 2)
    k_resrestrict3_red(OpView<R> o, const CB *__restrict__ b, const typename CT<R>::T *__restrict__ u,
                       typename CT<R>::T *__restrict__ rc, int ncx, int ncy, int ncz, int kc, int first) {
    pdl_enter();
    if (o.gate && *o.gate) return;
    typedef typename CT<R>::T C;
    extern __shared__ __align__(16) unsigned char r3_smem[];
    C(*rbuf)[R3_FH][R3_FW] = reinterpret_cast<C(*)[R3_FH][R3_FW]>(r3_smem);
    const int I0 = 1 + blockIdx.x * R3_TX, J0 = 1 + blockIdx.y * R3_TY;
    const int K0 = 1 + blockIdx.z * kc, K1 = min(K0 + kc, ncz - 1);
    const int t = threadIdx.x, X0 = 2 * I0 - 1, ly = t / R3R_HW, y = 2 * J0 - 1 + ly;
    const size_t sy = (size_t)o.nx, sz = sy * o.ny;
    const int zs = 2 * K0 - 1, ze = 2 * K1 - 1;
    // a buffer holds planes of one parity, so its red nodes are the same in every plane: the rest
    // (black, or outside the interior) stays zero
    for (int q = t; q < 2 * R3_FH * R3_FW; q += R3R_NT) (&rbuf[0][0][0])[q] = mk(R(0), R(0));
    __syncthreads();
    const bool row = t < R3R_HW * R3_FH && y <= o.ny - 2;
    C cwy = mk(R(0), R(0)), ccy = cwy, cey = cwy;
    if (row) { cwy = __ldg(&o.cy[3 * y]); ccy = __ldg(&o.cy[3 * y + 1]); cey = __ldg(&o.cy[3 * y + 2]); }
    const int cx = t % R3_TX, cy = t / R3_TX, I = I0 + cx, J = J0 + cy;
    const bool own = t < R3_TX * R3_TY && I <= ncx - 2 && J <= ncy - 2;
    C acc = mk(R(0), R(0));
    for (int z = zs; z <= ze; z++) {
        const int lx = 2 * (t - ly * R3R_HW) + ((X0 + y + z) & 1), x = X0 + lx;
        if (row && lx < R3_FW && x <= o.nx - 2) {
            const size_t p = (size_t)x + sy * y + sz * z;
            C a2 = cmul(__ldg(&o.cx[3 * x]), u[p - 1]);
            a2 = cfma(__ldg(&o.cx[3 * x + 2]), u[p + 1], a2);
            a2 = cfma(cwy, u[p - sy], a2);
            a2 = cfma(cey, u[p + sy], a2);
            a2 = cfma(__ldg(&o.cz[3 * z]), u[p - sz], a2);
            a2 = cfma(__ldg(&o.cz[3 * z + 2]), u[p + sz], a2);
            if (first) {
                a2 = mk(-a2.x, -a2.y);
            } else {
                C d = cadd(cadd(__ldg(&o.cx[3 * x + 1]), ccy), __ldg(&o.cz[3 * z + 1]));
                d = cadd(d, cadd(cscale(o.bk, o.k2[p]), o.c));
                a2 = csub(to_c(b[p], R()), cfma(d, u[p], a2));
            }
            rbuf[z & 1][ly][lx] = a2;
        }
        __syncthreads();
        if (own) {
            const C(*rr)[R3_FW] = rbuf[z & 1];
            const int fx = 2 * cx + 1, fy = 2 * cy + 1;  // region position of fine node (2I, 2J)
            if (z & 1) {
                // odd plane: the red nodes are the four side neighbours (weight 2)
                const C v = cscale(cadd(cadd(rr[fy][fx - 1], rr[fy][fx + 1]), cadd(rr[fy - 1][fx], rr[fy + 1][fx])), R(2));
                const int K = (z - 1) >> 1;
                if (K >= K0) rc[(size_t)I + (size_t)ncx * ((size_t)J + (size_t)ncy * K)] = cscale(cadd(acc, v), R(1.0 / 64.0));
                acc = v;
            } else {
                // even plane: the centre (weight 4) and the four corners, doubled along z
                const C v = cadd(cadd(rr[fy - 1][fx - 1], rr[fy - 1][fx + 1]), cadd(rr[fy + 1][fx - 1], rr[fy + 1][fx + 1]));
                const C c = rr[fy][fx];
                acc = mk(fma(R(2), fma(R(4), c.x, v.x), acc.x), fma(R(2), fma(R(4), c.y, v.y), acc.y));
            }
        }
    }
}

// 3D prolongation + correction in closed form: uf[p] += 1/8 of the sum of ec at the eight corners
// (floor / ceil of i/2, j/2, k/2), coincident corners repeated, i.e. the average over the distinct
// coarse nodes of k_prolong_add.  Each thread marches kc fine planes.
// The same for the nodes with odd i + j + k only (threads map to every other x node): before a red-black sweep
// with omega = 1, whose first colour does not use its old values.
template <typename R>
__global__ void __launch_bounds__(BX *BY) k_prolong3_black(int nx, int ny, int nz, const typename CT<R>::T *__restrict__ ec,
                                                           typename CT<R>::T *__restrict__ uf, int kc,
                                                           const int *__restrict__ gate) {
    pdl_enter();
    if (gate && *gate) return;
    typedef typename CT<R>::T C;
    const int t = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y + 1;
    if (j > ny - 2) return;
    const int ncx = (nx + 1) / 2, ncy = (ny + 1) / 2;
    const int k0 = blockIdx.z * kc + 1, k1 = min(k0 + kc, nz - 1);
    const size_t csy = (size_t)ncx, csz = (size_t)ncx * ncy, ja = csy * (j >> 1), jb = csy * ((j + 1) >> 1);
#pragma unroll 2
    for (int k = k0; k < k1; k++) {
        const int i = 2 * t + 1 + ((j + k) & 1);
        if (i > nx - 2) continue;
        const size_t p = (size_t)i + (size_t)nx * ((size_t)j + (size_t)ny * k);
        const int ia = i >> 1, ib = (i + 1) >> 1;
        auto corner_sum = [&](int c) {
            const C *e = ec + csz * c;
            return cadd(cadd(e[ja + ia], e[ja + ib]), cadd(e[jb + ia], e[jb + ib]));
        };
        const C uq = uf[p], sa = corner_sum(k >> 1);
        if (k & 1) uf[p] = cadd(uq, cscale(cadd(sa, corner_sum((k + 1) >> 1)), R(0.125)));
        else uf[p] = cadd(uq, cscale(sa, R(0.25)));
    }
}

template <typename R>
__global__ void __launch_bounds__(BX *BY) k_prolong3(int nx, int ny, int nz, const typename CT<R>::T *__restrict__ ec,
                                                     typename CT<R>::T *__restrict__ uf, int kc,
                                                     const int *__restrict__ gate) {
    pdl_enter();
    const int gv = gate_value(gate);
    typedef typename CT<R>::T C;
    const int i = blockIdx.x * BX + threadIdx.x + 1;
    const int j = blockIdx.y * BY + threadIdx.y + 1;
    if (i > nx - 2 || j > ny - 2) return;
    const int ncx = (nx + 1) / 2, ncy = (ny + 1) / 2;
    const int k0 = blockIdx.z * kc + 1, k1 = min(k0 + kc, nz - 1);
    const size_t csy = (size_t)ncx, csz = (size_t)ncx * ncy;
    const size_t c00 = (size_t)(i >> 1) + csy * (j >> 1), c10 = (size_t)((i + 1) >> 1) + csy * (j >> 1);
    const size_t c01 = (size_t)(i >> 1) + csy * ((j + 1) >> 1), c11 = (size_t)((i + 1) >> 1) + csy * ((j + 1) >> 1);
    // S(c): the four in-plane corners' sum on coarse plane c; fine plane k takes S(k >> 1) and
    // S((k + 1) >> 1), so every coarse plane is summed once and the next one is loaded while the
    // current fine plane is written
    auto corner_sum = [&](int c) {
        const size_t z = csz * c;
        return cadd(cadd(ec[c00 + z], ec[c10 + z]), cadd(ec[c01 + z], ec[c11 + z]));
    };
    C sa = corner_sum(k0 >> 1), sb = corner_sum((k0 + 1) >> 1);
    size_t p = (size_t)i + (size_t)nx * ((size_t)j + (size_t)ny * k0);
    C uq = uf[p];
    if (gv) return;
    for (int k = k0; k < k1; k++, p += (size_t)nx * ny) {
        C sn = sb, un = uq;
        if (k + 1 < k1) {
            un = uf[p + (size_t)nx * ny];
            // three planes ahead into L2 (257^3: 690 us per cycle with it, 702 without)
            if (k + 3 < k1 && (threadIdx.x & 15) == 0) l2_prefetch(&uf[p + 3 * (size_t)nx * ny]);
            if (((k + 2) >> 1) != ((k + 1) >> 1)) sn = corner_sum((k + 2) >> 1);
        }
        uf[p] = cadd(uq, cscale(cadd(sa, sb), R(0.125)));
        // next fine plane: (k + 1) >> 1 is this plane's upper coarse plane
        sa = sb;
        sb = sn;
        uq = un;
    }
}

// Exact coarsest solve as u = Minv b on the unknowns (interior nodes in natural order); one
// warp per row, fixed-order lane partial sums reduced by shuffles.
template <typename R>
__global__ void k_dense_solve(int nx, int ny, int nz, int dim, int nu, const typename CT<R>::T *__restrict__ minv,
                              const typename CT<R>::T *__restrict__ b, typename CT<R>::T *__restrict__ u) {
    pdl_enter();
    typedef typename CT<R>::T C;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= nu) return;
    const int mx = nx - 2, my = ny - 2;
    C acc = mk(R(0), R(0));
    for (int c = lane; c < nu; c += 32) {
        const int ci = c % mx, cj = (c / mx) % my, ck = dim == 3 ? c / (mx * my) : -1;
        const size_t q = (size_t)(ci + 1) + (size_t)nx * ((size_t)(cj + 1) + (size_t)ny * (ck + 1));
        acc = cfma(minv[(size_t)warp * nu + c], b[q], acc);
    }
    for (int off = 16; off > 0; off >>= 1) {
        acc.x += __shfl_down_sync(0xffffffffu, acc.x, off);
        acc.y += __shfl_down_sync(0xffffffffu, acc.y, off);
    }
    if (lane == 0) {
        const int ri = warp % mx, rj = (warp / mx) % my, rk = dim == 3 ? warp / (mx * my) : -1;
        u[(size_t)(ri + 1) + (size_t)nx * ((size_t)(rj + 1) + (size_t)ny * (rk + 1))] = acc;
    }
    (void)nz;
}

template <typename CI, typename CO>
__global__ void k_convert(size_t n, const CI *__restrict__ in, CO *__restrict__ out) {
    pdl_enter();
    typedef decltype(out->x) RO;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x)
        out[q] = to_c(in[q], RO());
}

template <typename C> __global__ void k_zero(size_t n, C *x) {
    pdl_enter();
    typedef decltype(x->x) R;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x)
        x[q] = mk(R(0), R(0));
}

// ------------------------------------------------------------------------------ temporal blocking
// 2D omega-Jacobi with two sweeps, several sweeps per shared-memory tile.  Each block owns a
// tile of TCX x TCY coarse nodes and the fine nodes x in [2 I0 - 1, 2 I0 + 2 TCX - 1) (same in
// y), and works on the fine region R3 = [2 I0 - 3, 2 I0 + 2 TCX + 1], the owned nodes plus a
// 3-node halo: two sweeps and a residual each consume one halo layer.  Nodes outside the
// interior of the grid are held at zero (Dirichlet).  Same arithmetic as k_jacobi /
// k_residual_restrict / k_prolong_add, in one launch per phase of the cycle instead of three.
// The tile shape is a template parameter; the host picks one per level (tuning).
// Threads of a block of the blocked kernels for a region of n nodes: the fewest passes over the
// region with at most 512 threads, then the fewest warps for that many passes (a fixed 256 left a
// nearly empty last pass on some tiles: 777 = 3 x 256 + 9).
constexpr int tile_threads(int n) { return ((n + (n + 511) / 512 - 1) / ((n + 511) / 512) + 31) / 32 * 32; }

template <int TCX, int TCY> struct Tile {
    static constexpr int RW = 2 * TCX + 5, RH = 2 * TCY + 5;  // R3 extent
    static constexpr int NT = tile_threads(RW * RH);           // threads per block
    static constexpr int NP = (RW * RH + NT - 1) / NT;          // passes of a phase
    struct Coef {
        float2 x[RW][3], y[RH][3];
    };
    struct Pre {
        Coef tc;
        float2 b[RH][RW];
        float2 di[RH][RW];  // 1 / diagonal
        float2 u1[RH][RW];  // first sweep, later the residual
        float2 u2[RH][RW];
    };
    struct Post {
        Coef tc;
        float2 b[RH][RW];
        float2 di[RH][RW];  // 1 / diagonal
        float2 u3[RH][RW];
        float2 u4[RH][RW];
    };
};

// 1 / D at the region nodes of this thread, node k of for_region_k in dv[k] (0 off the interior).
template <int RW, int RH, int ST, int NP>
__device__ __forceinline__ void tile_dinv(const OpView<float> &o, int X0, int Y0, float2 (&dv)[NP]) {
#pragma unroll
    for (int k = 0; k < NP; k++) {
        const int q = threadIdx.x + ST * k, sy = q / RW, x = X0 + q - sy * RW, y = Y0 + sy;
        dv[k] = (q < RW * RH && x >= 1 && x <= o.nx - 2 && y >= 1 && y <= o.ny - 2) ? __ldg(&o.dinv[(size_t)x + (size_t)o.nx * y])
                                                                                : make_float2(0.f, 0.f);
    }
}
// f(sx, sy, k) for every node of an RW x RH region, ST threads, node q = tid + ST k in row-major order.
template <int RW, int RH, int ST, int NP, typename F>
__device__ __forceinline__ void for_region_k(F f) {
#pragma unroll
    for (int k = 0; k < NP; k++) {
        const int q = threadIdx.x + ST * k, sy = q / RW;
        if (q < RW * RH) f(q - sy * RW, sy, k);
    }
}

// Loads the operator's coefficient triples of the region's columns and rows.
template <int RW, int RH, typename TC>
__device__ __forceinline__ void tile_coef(const OpView<float> &o, int X0, int Y0, TC &tc) {
    for (int q = threadIdx.x; q < RW * 3; q += blockDim.x) {
        const int sx = q / 3, t = q % 3, x = X0 + sx;
        tc.x[sx][t] = (x >= 1 && x <= o.nx - 2) ? o.cx[3 * x + t] : make_float2(0.f, 0.f);
    }
    for (int q = threadIdx.x; q < RH * 3; q += blockDim.x) {
        const int sy = q / 3, t = q % 3, y = Y0 + sy;
        tc.y[sy][t] = (y >= 1 && y <= o.ny - 2) ? o.cy[3 * y + t] : make_float2(0.f, 0.f);
    }
}

// (M u)_s and the diagonal at region node (sx, sy) from shared-memory u (row stride RW).
template <int RW, typename TC>
__device__ __forceinline__ float2 tile_stencil(const TC &tc, const float2 (*u)[RW], int sx, int sy, float k2,
                                               float2 bk, float2 c, float2 &d) {
    float2 acc = cmul(tc.x[sx][0], u[sy][sx - 1]);
    acc = cfma(tc.x[sx][2], u[sy][sx + 1], acc);
    acc = cfma(tc.y[sy][0], u[sy - 1][sx], acc);
    acc = cfma(tc.y[sy][2], u[sy + 1][sx], acc);
    d = cadd(cadd(tc.x[sx][1], tc.y[sy][1]), cadd(cscale(bk, k2), c));
    return cfma(d, u[sy][sx], acc);
}

// Off-diagonal part of (M u)_s at region node (sx, sy).
template <int RW, typename TC>
__device__ __forceinline__ float2 tile_offdiag(const TC &tc, const float2 (*u)[RW], int sx, int sy) {
    float2 acc = cmul(tc.x[sx][0], u[sy][sx - 1]);
    acc = cfma(tc.x[sx][2], u[sy][sx + 1], acc);
    acc = cfma(tc.y[sy][0], u[sy - 1][sx], acc);
    return cfma(tc.y[sy][2], u[sy + 1][sx], acc);
}
// One omega-Jacobi update at region node (sx, sy): u + omega ((b - offdiag) / d - u).
template <int RW, typename TC>
__device__ __forceinline__ float2 tile_jacobi(const TC &tc, const float2 (*u)[RW], const float2 (*b)[RW],
                                              const float2 (*di)[RW], int sx, int sy, float omega) {
    const float2 uc = u[sy][sx];
    const float2 t = cmul(csub(b[sy][sx], tile_offdiag<RW>(tc, u, sx, sy)), di[sy][sx]);
    return cadd(uc, cscale(csub(t, uc), omega));
}

// f(sx, sy) for every node of an RW x RH region, ST threads, node q = tid + ST k in row-major
// order (the region coordinates advance incrementally).
template <int RW, int RH, int ST, typename F>
__device__ __forceinline__ void for_region(F f) {
    constexpr int N = RW * RH, DX = ST % RW, DY = ST / RW;
    int sx = threadIdx.x % RW, sy = threadIdx.x / RW;
    for (int q = threadIdx.x; q < N; q += ST) {
        f(sx, sy);
        sx += DX;
        sy += DY;
        if (sx >= RW) {
            sx -= RW;
            sy++;
        }
    }
}

// Diagonal of M at region node (sx, sy) from the staged coefficients and k^2.
template <typename TC>
__device__ __forceinline__ float2 tile_diag(const TC &tc, int sx, int sy, float k2, float2 bk, float2 c) {
    return cadd(cadd(tc.x[sx][1], tc.y[sy][1]), cadd(cscale(bk, k2), c));
}

// u = two omega-Jacobi sweeps from u = 0 for M u = b, written on the owned fine nodes; then
// rc = FW(b - M u) on the owned coarse nodes.  Blocks whose region lies inside the grid's
// interior skip the per-node boundary tests.
// (bx, by): the tile of coarse nodes this block owns.
// CB double2: b is a complex128 vector; its owned nodes rounded to complex64 go to b_out too.
// EARLY: the caller has not yet waited for the kernel before it in the stream: the operator's data
// (coefficients and 1 / D, which no kernel writes) is loaded before the wait (1025^2 complex64 cycle, eager:
// 69.6 us, with the loads after it 74.8; its FGMRES solve in replayed graphs 20.4 against 20.8 ms).  The batched kernels fill the
// chip and keep the plain order.
template <int TCX, int TCY, bool EARLY, typename CB>
__device__ __forceinline__ void pre2_restrict_tile(const OpView<float> &o, float omega, const CB *__restrict__ b,
                                                   float2 *__restrict__ u, float2 *__restrict__ rc, int ncx, int ncy,
                                                   int bx, int by, const int *gate = nullptr,
                                                   float2 *__restrict__ b_out = nullptr) {
    typedef Tile<TCX, TCY> TL;
    constexpr int RW = TL::RW, RH = TL::RH;
    extern __shared__ __align__(16) unsigned char pre_smem[];
    __shared__ int gate_s;  // the gate flag, published by the first block barrier
    typename TL::Pre &T = *reinterpret_cast<typename TL::Pre *>(pre_smem);
    const int I0 = 1 + bx * TCX, J0 = 1 + by * TCY;
    const int X0 = 2 * I0 - 3, Y0 = 2 * J0 - 3;
    const int nx = o.nx, ny = o.ny;
    const bool full = X0 >= 1 && X0 + RW - 1 <= nx - 2 && Y0 >= 1 && Y0 + RH - 1 <= ny - 2;
    auto inside = [&](int x, int y) { return full || (x >= 1 && x <= nx - 2 && y >= 1 && y <= ny - 2); };
    // the coefficients are first used by the second sweep: one barrier publishes them with b,
    // 1 / D and the first sweep
    tile_coef<RW, RH>(o, X0, Y0, T.tc);
    float2 dv[TL::NP];
    if (EARLY) {
        tile_dinv<RW, RH, TL::NT>(o, X0, Y0, dv);
        pdl_enter();
    }
    if (threadIdx.x == 0) gate_s = gate_value(gate);
    // load b; sweep 1 from zero (pointwise): u1 = omega b / D
    for_region_k<RW, RH, TL::NT, TL::NP>([&](int sx, int sy, int k) {
        const int x = X0 + sx, y = Y0 + sy;
        float2 bv = make_float2(0.f, 0.f), di = EARLY ? dv[k] : make_float2(0.f, 0.f);
        if (inside(x, y)) {
            const size_t p = (size_t)x + (size_t)nx * y;
            bv = to_c(b[p], 0.f);
            if (!EARLY) di = o.dinv[p];
        }
        T.b[sy][sx] = bv;
        T.di[sy][sx] = di;
        T.u1[sy][sx] = cscale(cmul(bv, di), omega);
    });
    __syncthreads();
    if (gate_s) return;
    // sweep 2 on R3 shrunk by one
    for_region<RW, RH, TL::NT>([&](int sx, int sy) {
        float2 v = make_float2(0.f, 0.f);
        if (sx >= 1 && sx < RW - 1 && sy >= 1 && sy < RH - 1 && inside(X0 + sx, Y0 + sy))
            v = tile_jacobi<RW>(T.tc, T.u1, T.b, T.di, sx, sy, omega);
        T.u2[sy][sx] = v;
    });
    __syncthreads();
    // owned fine nodes of the smoothed iterate, and the residual on R3 shrunk by two
    for_region<RW, RH, TL::NT>([&](int sx, int sy) {
        const int x = X0 + sx, y = Y0 + sy;
        const bool in = inside(x, y);
        if (in && sx >= 2 && sx < 2 + 2 * TCX && sy >= 2 && sy < 2 + 2 * TCY) {
            u[(size_t)x + (size_t)nx * y] = T.u2[sy][sx];
            if (sizeof(CB) == sizeof(double2)) b_out[(size_t)x + (size_t)nx * y] = T.b[sy][sx];
        }
        float2 r = make_float2(0.f, 0.f);
        if (in && sx >= 2 && sx < RW - 2 && sy >= 2 && sy < RH - 2) {
            const float2 d = cinv_fast(T.di[sy][sx]);
            r = csub(csub(T.b[sy][sx], tile_offdiag<RW>(T.tc, T.u2, sx, sy)), cmul(d, T.u2[sy][sx]));
        }
        T.u1[sy][sx] = r;
    });
    __syncthreads();
    // full weighting on the owned coarse nodes: fine node 2I is region node 2(I - I0) + 3
    for (int q = threadIdx.x; q < TCX * TCY; q += blockDim.x) {
        const int cx = q % TCX, cy = q / TCX, I = I0 + cx, J = J0 + cy;
        if (I > ncx - 2 || J > ncy - 2) continue;
        const int sx = 2 * cx + 3, sy = 2 * cy + 3;
        const float2 *r0 = &T.u1[sy - 1][sx], *r1 = &T.u1[sy][sx], *r2 = &T.u1[sy + 1][sx];
        // (1,2,1)/4 along x on each of the three rows, then (1,2,1)/4 along y
        const float2 a0 = cadd(cadd(r0[-1], r0[1]), cscale(r0[0], 2.f));
        const float2 a1 = cadd(cadd(r1[-1], r1[1]), cscale(r1[0], 2.f));
        const float2 a2 = cadd(cadd(r2[-1], r2[1]), cscale(r2[0], 2.f));
        rc[(size_t)I + (size_t)ncx * J] = cscale(cadd(cadd(a0, a2), cscale(a1, 2.f)), 0.0625f);
    }
}

template <int TCX, int TCY, typename CB>
__global__ void __launch_bounds__(Tile<TCX, TCY>::NT, 4) k_pre2_restrict(OpView<float> o, float omega, const CB *__restrict__ b,
                                                       float2 *__restrict__ u, float2 *__restrict__ rc, int ncx,
                                                       int ncy, float2 *__restrict__ b_out) {
    pre2_restrict_tile<TCX, TCY, true>(o, omega, b, u, rc, ncx, ncy, blockIdx.x, blockIdx.y, o.gate, b_out);
}

// u_out <- two omega-Jacobi sweeps of (u_in + P ec), on the owned fine nodes.  u_in and u_out
// are different arrays: blocks read their halo of u_in while other blocks write u_out.
// Bilinear interpolation in closed form: P ec at fine node (x, y) is the mean of the four
// coarse values at (floor/ceil(x/2), floor/ceil(y/2)), coincident ones repeated.
template <int TCX, int TCY, bool EARLY>
__device__ __forceinline__ void prolong_post2_tile(const OpView<float> &o, float omega, const float2 *__restrict__ b,
                                                   const float2 *__restrict__ u_in, float2 *__restrict__ u,
                                                   const float2 *__restrict__ ec, int ncx, int ncy, int bx, int by,
                                                   const int *gate = nullptr) {
    typedef Tile<TCX, TCY> TL;
    constexpr int RW = TL::RW, RH = TL::RH;
    extern __shared__ __align__(16) unsigned char post_smem[];
    __shared__ int gate_s;  // the gate flag, published by the first block barrier
    typename TL::Post &T = *reinterpret_cast<typename TL::Post *>(post_smem);
    const int I0 = 1 + bx * TCX, J0 = 1 + by * TCY;
    const int X0 = 2 * I0 - 3, Y0 = 2 * J0 - 3;
    const int nx = o.nx, ny = o.ny;
    const bool full = X0 >= 1 && X0 + RW - 1 <= nx - 2 && Y0 >= 1 && Y0 + RH - 1 <= ny - 2;
    auto inside = [&](int x, int y) { return full || (x >= 1 && x <= nx - 2 && y >= 1 && y <= ny - 2); };
    // the coefficients are first used by the first sweep: one barrier publishes them with b,
    // 1 / D and u + P ec, whose coarse values each node reads itself (the four corner nodes
    // floor/ceil(x / 2), floor/ceil(y / 2) of an interior fine node lie in the coarse grid)
    tile_coef<RW, RH>(o, X0, Y0, T.tc);
    float2 dv[TL::NP];
    if (EARLY) {
        tile_dinv<RW, RH, TL::NT>(o, X0, Y0, dv);
        pdl_enter();
    }
    if (threadIdx.x == 0) gate_s = gate_value(gate);
    // u3 = u + P ec on the region
    for_region_k<RW, RH, TL::NT, TL::NP>([&](int sx, int sy, int k) {
        const int x = X0 + sx, y = Y0 + sy;
        float2 bv = make_float2(0.f, 0.f), v = make_float2(0.f, 0.f), di = EARLY ? dv[k] : make_float2(0.f, 0.f);
        if (inside(x, y)) {
            const size_t p = (size_t)x + (size_t)nx * y;
            bv = b[p];
            if (!EARLY) di = o.dinv[p];
            const size_t ya = (size_t)ncx * (y >> 1), yb = (size_t)ncx * ((y + 1) >> 1);
            const int xa = x >> 1, xb = (x + 1) >> 1;
            const float2 e = cadd(cadd(ec[ya + xa], ec[ya + xb]), cadd(ec[yb + xa], ec[yb + xb]));
            v = cadd(u_in[p], cscale(e, 0.25f));
        }
        T.b[sy][sx] = bv;
        T.di[sy][sx] = di;
        T.u3[sy][sx] = v;
    });
    __syncthreads();
    if (gate_s) return;
    // sweep 1 on R3 shrunk by one
    for_region<RW, RH, TL::NT>([&](int sx, int sy) {
        float2 v = make_float2(0.f, 0.f);
        if (sx >= 1 && sx < RW - 1 && sy >= 1 && sy < RH - 1 && inside(X0 + sx, Y0 + sy))
            v = tile_jacobi<RW>(T.tc, T.u3, T.b, T.di, sx, sy, omega);
        T.u4[sy][sx] = v;
    });
    __syncthreads();
    // sweep 2 on the owned fine nodes
    for (int q = threadIdx.x; q < 4 * TCX * TCY; q += blockDim.x) {
        const int sx = 2 + q % (2 * TCX), sy = 2 + q / (2 * TCX), x = X0 + sx, y = Y0 + sy;
        if (!inside(x, y)) continue;
        u[(size_t)x + (size_t)nx * y] = tile_jacobi<RW>(T.tc, T.u4, T.b, T.di, sx, sy, omega);
    }
}

template <int TCX, int TCY>
__global__ void __launch_bounds__(Tile<TCX, TCY>::NT, 4) k_prolong_post2(OpView<float> o, float omega, const float2 *__restrict__ b,
                                                       const float2 *__restrict__ u_in, float2 *__restrict__ u,
                                                       const float2 *__restrict__ ec, int ncx, int ncy) {
    prolong_post2_tile<TCX, TCY, true>(o, omega, b, u_in, u, ec, ncx, ncy, blockIdx.x, blockIdx.y, o.gate);
}

// Batched forms (many problems, one launch): blockIdx.z picks the table entry, whose level has
// the same nodes in every entry of one launch; entries whose problem is inactive return at once.
template <int TCX, int TCY>
__global__ void __launch_bounds__(Tile<TCX, TCY>::NT, 4) k_pre2_restrict_b(const BLevel *__restrict__ tab, float omega) {
    pdl_enter();
    const BLevel &E = tab[blockIdx.z];
    if (*E.active == 0) return;
    const OpView<float> o = view(E.op);
    pre2_restrict_tile<TCX, TCY, false>(o, omega, E.b, E.t, E.coarse, (o.nx + 1) / 2, (o.ny + 1) / 2, blockIdx.x, blockIdx.y);
}

template <int TCX, int TCY>
__global__ void __launch_bounds__(Tile<TCX, TCY>::NT, 4) k_prolong_post2_b(const BLevel *__restrict__ tab, float omega, int j) {
    pdl_enter();
    const BLevel &E = tab[blockIdx.z];
    if (*E.active == 0) return;
    const OpView<float> o = view(E.op);
    prolong_post2_tile<TCX, TCY, false>(o, omega, E.b, E.t, E.u + (size_t)j * E.ustride, E.coarse, (o.nx + 1) / 2,
                                 (o.ny + 1) / 2, blockIdx.x, blockIdx.y);
}

// Planes per thread of a 3D z-marching kernel: kmax, halved while the grid would have fewer than
// `target` blocks (small levels: more, shorter chains instead of a few long ones).
static int z_chunk(size_t tiles_xy, int planes, int kmax, size_t target) {
    int kc = kmax;
    while (kc > 1 && tiles_xy * cdiv(planes, kc) < target) kc /= 2;
    return kc;
}

// Planes per thread of an A x in 3D.  complex64: as above.  complex128 holds 100 registers, two blocks
// per SM, and is bound by the FP64 units, so what counts is the block-planes of the busiest SM: whole
// rounds of two blocks, each of kc planes and about 0.8 of one for its coefficients.  Measured, kc = 8 /
// 4 / 2 / 1: 65 x 57 x 73 nodes - / 19.5 / - / 21.2 us, 81^3 36.2 / - / 37.9 / 44.0, 97^3 61.3 / 50.5 / 53.3 / -,
// 129 x 97 x 113 80.6 / 73.8 / 78.3 / -, 129^3 111.7 / 108.6 / - / -, 161 x 129 x 161 162 / 165 / - / -, 193 x 161 x 193 276 / 288 / - / -.  (The
// residual and the red-black sweep keep the shorter chunks: with this rule a red-black cycle on 193 x
// 129 x 97 nodes took 518 instead of 469 us.)
template <typename R> static int apply_chunk(size_t tiles_xy, int planes) {
    if (sizeof(R) == sizeof(float)) return z_chunk(tiles_xy, planes, KCHUNK, 152 * 10);
    int best = 1;
    double least = 1e30;
    for (int kc = KCHUNK; kc >= 1; kc /= 2) {
        const double cost = (double)cdiv(tiles_xy * cdiv(planes, kc), 2 * 152) * (kc + 0.8);
        if (cost < least) {
            least = cost;
            best = kc;
        }
    }
    return best;
}

dim3 grid_for(const int n[3], int dim) {
    return dim3(cdiv(n[0] - 2, BX), cdiv(n[1] - 2, BY), dim == 3 ? cdiv(n[2] - 2, KCHUNK) : 1);
}

}  // namespace

// ------------------------------------------------------------------------------ launchers
template <typename R, typename CX>
cudaError_t launch_apply(const DevOp<R> &op, int dim, const CX *x, typename CT<R>::T *y, cudaStream_t s) {
    dim3 g = grid_for(op.n, dim), b(BX, BY);
    const int kc = dim == 3 ? apply_chunk<R>((size_t)g.x * g.y, op.n[2] - 2) : 1;
    if (dim == 3) g.z = cdiv(op.n[2] - 2, kc);
    const CX *none = nullptr;
    if (dim == 3) launch_pdl(k_apply<R, 3, CX, CX, false>, g, b, 0, s, view(op), none, x, y, kc);
    else launch_pdl(k_apply<R, 2, CX, CX, false>, g, b, 0, s, view(op), none, x, y, kc);
    return cudaGetLastError();
}

template <typename R, typename CB>
cudaError_t launch_residual(const DevOp<R> &op, int dim, const CB *bb, const typename CT<R>::T *u,
                            typename CT<R>::T *r, cudaStream_t s) {
    typedef typename CT<R>::T C;
    dim3 g = grid_for(op.n, dim), b(BX, BY);
    const int kc = dim == 3 ? z_chunk((size_t)g.x * g.y, op.n[2] - 2, KCHUNK, 152 * 10) : 1;
    if (dim == 3) g.z = cdiv(op.n[2] - 2, kc);
    if (dim == 3) launch_pdl(k_apply<R, 3, C, CB, true>, g, b, 0, s, view(op), bb, u, r, kc);
    else launch_pdl(k_apply<R, 2, C, CB, true>, g, b, 0, s, view(op), bb, u, r, kc);
    return cudaGetLastError();
}

template <typename R, typename CB>
cudaError_t launch_jacobi(const DevOp<R> &op, int dim, R omega, const CB *bb, const typename CT<R>::T *u_in,
                          typename CT<R>::T *u_out, cudaStream_t s) {
    dim3 g = grid_for(op.n, dim), b(BX, BY);
    if (dim == 3) {
        const int kc = z_chunk((size_t)g.x * g.y, op.n[2] - 2, 2 * KCHUNK, 152 * 10);
        g.z = cdiv(op.n[2] - 2, kc);
        typename CT<R>::T *none = nullptr;
        auto go = [&](auto kernel) { return launch_pdl(kernel, g, b, 0, s, view(op), omega, bb, u_in, u_out, none); };
        if (u_in == nullptr) {
            switch (kc) {
            case 16: go(k_jacobi3<R, CB, true, 16>); break;
            case 8: go(k_jacobi3<R, CB, true, 8>); break;
            case 4: go(k_jacobi3<R, CB, true, 4>); break;
            case 2: go(k_jacobi3<R, CB, true, 2>); break;
            default: go(k_jacobi3<R, CB, true, 1>); break;
            }
        } else {
            switch (kc) {
            case 16: go(k_jacobi3<R, CB, false, 16>); break;
            case 8: go(k_jacobi3<R, CB, false, 8>); break;
            case 4: go(k_jacobi3<R, CB, false, 4>); break;
            case 2: go(k_jacobi3<R, CB, false, 2>); break;
            default: go(k_jacobi3<R, CB, false, 1>); break;
            }
        }
    } else if (u_in == nullptr) {
        launch_pdl(k_jacobi<R, 2, CB, true>, g, b, 0, s, view(op), omega, bb, u_in, u_out);
    } else {
        launch_pdl(k_jacobi<R, 2, CB, false>, g, b, 0, s, view(op), omega, bb, u_in, u_out);
    }
    return cudaGetLastError();
}

cudaError_t launch_jacobi3_first(const DevOp<float> &op, float omega, const double2 *v, float2 *b_out, float2 *u_out,
                                 cudaStream_t s) {
    const int dim = 3;
    dim3 g = grid_for(op.n, dim), b(BX, BY);
    const int kc = z_chunk((size_t)g.x * g.y, op.n[2] - 2, KCHUNK, 152 * 10);
    g.z = cdiv(op.n[2] - 2, kc);
    const float2 *none = nullptr;
    auto go = [&](auto kernel) { return launch_pdl(kernel, g, b, 0, s, view(op), omega, v, none, u_out, b_out); };
    switch (kc) {
    case 8: go(k_jacobi3<float, double2, true, 8>); break;
    case 4: go(k_jacobi3<float, double2, true, 4>); break;
    case 2: go(k_jacobi3<float, double2, true, 2>); break;
    default: go(k_jacobi3<float, double2, true, 1>); break;
    }
    return cudaGetLastError();
}

template <typename R, typename CB>
cudaError_t launch_rb(const DevOp<R> &op, int dim, R omega, const CB *bb, typename CT<R>::T *u, int colour, int zero,
                      cudaStream_t s) {
    dim3 g(cdiv((op.n[0] - 1) / 2, BX), cdiv(op.n[1] - 2, BY)), b(BX, BY);
    // planes per thread: chunks of 8 left most of the chip idle on small levels (33 us a colour)
    const int kc = dim == 3 ? z_chunk((size_t)g.x * g.y, op.n[2] - 2, KCHUNK, 152 * 10) : 1;
    if (dim == 3) g.z = cdiv(op.n[2] - 2, kc);
    auto go = [&](auto kernel) { return launch_pdl(kernel, g, b, 0, s, view(op), omega, bb, u, colour, kc); };
    const bool no_own = zero || omega == R(1);
    if (dim == 3) {
        if (zero && colour == 0) go(k_rb<R, 3, CB, RB_ZERO>);
        else if (no_own) go(k_rb<R, 3, CB, RB_NO_OWN>);
        else go(k_rb<R, 3, CB, RB_ANY>);
    } else {
        if (zero && colour == 0) go(k_rb<R, 2, CB, RB_ZERO>);
        else if (no_own) go(k_rb<R, 2, CB, RB_NO_OWN>);
        else go(k_rb<R, 2, CB, RB_ANY>);
    }
    return cudaGetLastError();
}

template <typename R, typename CB>
cudaError_t launch_residual_restrict(const DevOp<R> &op, int dim, const CB *bb, const typename CT<R>::T *u,
                                     typename CT<R>::T *rc, cudaStream_t s, bool red, bool first) {
    int nc[3] = {(op.n[0] + 1) / 2, (op.n[1] + 1) / 2, dim == 3 ? (op.n[2] + 1) / 2 : 1};
    if (red && dim == 3) {
        dim3 g(cdiv(nc[0] - 2, R3_TX), cdiv(nc[1] - 2, R3_TY), 1);
        const int kc = z_chunk((size_t)g.x * g.y, nc[2] - 2, R3_KC, 152 * 4);
        g.z = cdiv(nc[2] - 2, kc);
        launch_pdl(k_resrestrict3_red<R, CB>, g, R3R_NT, r3_smem_bytes<R>(2), s, view(op), bb, u, rc, nc[0], nc[1], nc[2],
                   kc, first ? 1 : 0);
        return cudaGetLastError();
    }
    if (dim == 3 && (size_t)op.n[0] * op.n[1] < ((size_t)1 << 31)) {  // 32-bit in-plane offsets
        constexpr size_t smem = r3_smem_bytes<R>(R3_PLANES);
        static_assert(smem <= 48 * 1024, "");
        dim3 g(cdiv(nc[0] - 2, R3_TX), cdiv(nc[1] - 2, R3_TY), 1);
        const int kc = z_chunk((size_t)g.x * g.y, nc[2] - 2, R3_KC, 152 * 4);
        g.z = cdiv(nc[2] - 2, kc);
        launch_pdl(k_resrestrict3<R, CB>, g, R3_NT, smem, s, view(op), bb, u, rc, nc[0], nc[1], nc[2], kc);
        return cudaGetLastError();
    }
    dim3 g = grid_for(nc, dim), b(BX, BY);
    if (dim == 3) launch_pdl(k_residual_restrict<R, 3, CB>, g, b, 0, s, view(op), bb, u, rc, nc[0], nc[1], nc[2]);
    else launch_pdl(k_residual_restrict<R, 2, CB>, g, b, 0, s, view(op), bb, u, rc, nc[0], nc[1], nc[2]);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_prolong_add(const int nf[3], int dim, const typename CT<R>::T *ec, typename CT<R>::T *uf,
                               cudaStream_t s, const int *gate, bool black) {
    dim3 g = grid_for(nf, dim), b(BX, BY);
    if (dim == 3 && black) {
        g.x = cdiv((nf[0] - 1) / 2, BX);
        const int kc = z_chunk((size_t)g.x * g.y, nf[2] - 2, KCHUNK, 152 * 10);
        g.z = cdiv(nf[2] - 2, kc);
        launch_pdl(k_prolong3_black<R>, g, b, 0, s, nf[0], nf[1], nf[2], ec, uf, kc, gate);
    } else if (dim == 3) {
        const int kc = z_chunk((size_t)g.x * g.y, nf[2] - 2, KCHUNK, 152 * 10);
        g.z = cdiv(nf[2] - 2, kc);
        launch_pdl(k_prolong3<R>, g, b, 0, s, nf[0], nf[1], nf[2], ec, uf, kc, gate);
    } else {
        launch_pdl(k_prolong_add<R, 2>, g, b, 0, s, nf[0], nf[1], 1, ec, uf, gate);
    }
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_dense_solve(const int n[3], int dim, int nu, const typename CT<R>::T *minv,
                               const typename CT<R>::T *b, typename CT<R>::T *u, cudaStream_t s) {
    const int threads = 256, warps = threads / 32;
    launch_pdl(k_dense_solve<R>, cdiv(nu, warps), threads, 0, s, n[0], n[1], dim == 3 ? n[2] : 1, dim, nu, minv, b, u);
    return cudaGetLastError();
}

// Tile shapes (coarse nodes per block) of the temporally blocked kernels, by tile index (the
// wavefront, HELM_TILE_WAVE, has none).
static const int kTiles[HELM_TILE_COUNT][2] = {{32, 8}, {16, 16}, {16, 8}, {64, 4}, {0, 0}, {8, 8}};

bool fused_jacobi2_ok(const int n[3], int dim, int tile) {
    if (tile == HELM_TILE_WAVE) return wave_jacobi2_ok(n, dim);
    if (tile < 0 || tile >= HELM_TILE_COUNT) return false;
    if (dim != 2 || (n[0] - 1) % 2 || (n[1] - 1) % 2) return false;
    const int ncx = (n[0] + 1) / 2, ncy = (n[1] + 1) / 2;
    // the last tile's owned range must reach the last interior node: a tile row or column
    // that ends exactly at the grid's edge would leave node n - 2 unowned
    return ncx >= 3 && ncy >= 3 && (ncx - 2) % kTiles[tile][0] != 0 && (ncy - 2) % kTiles[tile][1] != 0;
}

template <int TCX, int TCY, typename CB>
static cudaError_t pre2_t(const DevOp<float> &op, float omega, const CB *b, float2 *u_out, float2 *rc, float2 *b_out,
                          cudaStream_t s) {
    const int ncx = (op.n[0] + 1) / 2, ncy = (op.n[1] + 1) / 2;
    constexpr size_t smem = sizeof(typename Tile<TCX, TCY>::Pre);
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_pre2_restrict<TCX, TCY, CB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    dim3 g(cdiv(ncx - 2, TCX), cdiv(ncy - 2, TCY));
    launch_pdl(k_pre2_restrict<TCX, TCY, CB>, g, Tile<TCX, TCY>::NT, smem, s, view(op), omega, b, u_out, rc, ncx, ncy, b_out);
    return cudaGetLastError();
}

template <int TCX, int TCY>
static cudaError_t post2_t(const DevOp<float> &op, float omega, const float2 *b, const float2 *u_in, float2 *u_out,
                           const float2 *ec, cudaStream_t s) {
    const int ncx = (op.n[0] + 1) / 2, ncy = (op.n[1] + 1) / 2;
    constexpr size_t smem = sizeof(typename Tile<TCX, TCY>::Post);
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_prolong_post2<TCX, TCY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    dim3 g(cdiv(ncx - 2, TCX), cdiv(ncy - 2, TCY));
    launch_pdl(k_prolong_post2<TCX, TCY>, g, Tile<TCX, TCY>::NT, smem, s, view(op), omega, b, u_in, u_out, ec, ncx,
               ncy);
    return cudaGetLastError();
}

template <typename CB>
static cudaError_t pre2_tile(const DevOp<float> &op, int tile, float omega, const CB *b, float2 *u_out, float2 *rc,
                             float2 *b_out, cudaStream_t s) {
    switch (tile) {
    case 0: return pre2_t<32, 8>(op, omega, b, u_out, rc, b_out, s);
    case 1: return pre2_t<16, 16>(op, omega, b, u_out, rc, b_out, s);
    case 2: return pre2_t<16, 8>(op, omega, b, u_out, rc, b_out, s);
    case HELM_TILE_8x8: return pre2_t<8, 8>(op, omega, b, u_out, rc, b_out, s);
    default: return pre2_t<64, 4>(op, omega, b, u_out, rc, b_out, s);
    }
}

cudaError_t launch_pre2_restrict(const DevOp<float> &op, int tile, float omega, const float2 *b, float2 *u_out,
                                 float2 *rc, cudaStream_t s) {
    if (!fused_jacobi2_ok(op.n, 2, tile) || (tile != HELM_TILE_WAVE && !op.dinv)) return cudaErrorInvalidValue;
    if (tile == HELM_TILE_WAVE) return launch_pre2_wave(op, omega, b, u_out, rc, s);
    return pre2_tile(op, tile, omega, b, u_out, rc, (float2 *)nullptr, s);
}

cudaError_t launch_pre2_restrict_c128(const DevOp<float> &op, int tile, float omega, const double2 *v, float2 *b_out,
                                      float2 *u_out, float2 *rc, cudaStream_t s) {
    if (!fused_jacobi2_ok(op.n, 2, tile) || tile == HELM_TILE_WAVE || !op.dinv) return cudaErrorInvalidValue;
    return pre2_tile(op, tile, omega, v, u_out, rc, b_out, s);
}

cudaError_t launch_prolong_post2(const DevOp<float> &op, int tile, float omega, const float2 *b, const float2 *u_in,
                                 float2 *u_out, const float2 *ec, cudaStream_t s) {
    if (!fused_jacobi2_ok(op.n, 2, tile) || (tile != HELM_TILE_WAVE && !op.dinv)) return cudaErrorInvalidValue;
    switch (tile) {
    case HELM_TILE_WAVE: return launch_post2_wave(op, omega, b, u_in, u_out, ec, s);
    case 0: return post2_t<32, 8>(op, omega, b, u_in, u_out, ec, s);
    case 1: return post2_t<16, 16>(op, omega, b, u_in, u_out, ec, s);
    case 2: return post2_t<16, 8>(op, omega, b, u_in, u_out, ec, s);
    case HELM_TILE_8x8: return post2_t<8, 8>(op, omega, b, u_in, u_out, ec, s);
    default: return post2_t<64, 4>(op, omega, b, u_in, u_out, ec, s);
    }
}

template <int TCX, int TCY>
static cudaError_t pre2_b_t(int n0, int n1, int count, const BLevel *tab, float omega, cudaStream_t s) {
    const int ncx = (n0 + 1) / 2, ncy = (n1 + 1) / 2;
    constexpr size_t smem = sizeof(typename Tile<TCX, TCY>::Pre);
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_pre2_restrict_b<TCX, TCY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    dim3 g(cdiv(ncx - 2, TCX), cdiv(ncy - 2, TCY), count);
    launch_pdl(k_pre2_restrict_b<TCX, TCY>, g, Tile<TCX, TCY>::NT, smem, s, tab, omega);
    return cudaGetLastError();
}

template <int TCX, int TCY>
static cudaError_t post2_b_t(int n0, int n1, int count, const BLevel *tab, float omega, int j, cudaStream_t s) {
    const int ncx = (n0 + 1) / 2, ncy = (n1 + 1) / 2;
    constexpr size_t smem = sizeof(typename Tile<TCX, TCY>::Post);
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_prolong_post2_b<TCX, TCY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    dim3 g(cdiv(ncx - 2, TCX), cdiv(ncy - 2, TCY), count);
    launch_pdl(k_prolong_post2_b<TCX, TCY>, g, Tile<TCX, TCY>::NT, smem, s, tab, omega, j);
    return cudaGetLastError();
}

cudaError_t launch_pre2_restrict_batch(const int n[3], int tile, int count, const BLevel *tab, float omega,
                                       cudaStream_t s) {
    if (count < 1 || count > 65535 || tile == HELM_TILE_WAVE || !fused_jacobi2_ok(n, 2, tile)) return cudaErrorInvalidValue;
    switch (tile) {
    case 0: return pre2_b_t<32, 8>(n[0], n[1], count, tab, omega, s);
    case 1: return pre2_b_t<16, 16>(n[0], n[1], count, tab, omega, s);
    case 2: return pre2_b_t<16, 8>(n[0], n[1], count, tab, omega, s);
    case HELM_TILE_8x8: return pre2_b_t<8, 8>(n[0], n[1], count, tab, omega, s);
    default: return pre2_b_t<64, 4>(n[0], n[1], count, tab, omega, s);
    }
}

cudaError_t launch_prolong_post2_batch(const int n[3], int tile, int count, const BLevel *tab, float omega, int j,
                                       cudaStream_t s) {
    if (count < 1 || count > 65535 || tile == HELM_TILE_WAVE || !fused_jacobi2_ok(n, 2, tile)) return cudaErrorInvalidValue;
    switch (tile) {
    case 0: return post2_b_t<32, 8>(n[0], n[1], count, tab, omega, j, s);
    case 1: return post2_b_t<16, 16>(n[0], n[1], count, tab, omega, j, s);
    case 2: return post2_b_t<16, 8>(n[0], n[1], count, tab, omega, j, s);
    case HELM_TILE_8x8: return post2_b_t<8, 8>(n[0], n[1], count, tab, omega, j, s);
    default: return post2_b_t<64, 4>(n[0], n[1], count, tab, omega, j, s);
    }
}

template <typename CI, typename CO>
cudaError_t launch_convert(size_t n, const CI *in, CO *out, cudaStream_t s) {
    launch_pdl(k_convert<CI, CO>, (unsigned)std::min<size_t>(cdiv(n, 256), 152 * 16), 256, 0, s, n, in, out);
    return cudaGetLastError();
}

template <typename C> cudaError_t launch_zero(size_t n, C *x, cudaStream_t s) {
    launch_pdl(k_zero<C>, (unsigned)std::min<size_t>(cdiv(n, 256), 152 * 16), 256, 0, s, n, x);
    return cudaGetLastError();
}

#define INST_R(R)                                                                                               \
    template cudaError_t launch_residual<R, CT<R>::T>(const DevOp<R> &, int, const CT<R>::T *, const CT<R>::T *, \
                                                       CT<R>::T *, cudaStream_t);                               \
    template cudaError_t launch_jacobi<R, CT<R>::T>(const DevOp<R> &, int, R, const CT<R>::T *, const CT<R>::T *, \
                                                     CT<R>::T *, cudaStream_t);                                 \
    template cudaError_t launch_rb<R, CT<R>::T>(const DevOp<R> &, int, R, const CT<R>::T *, CT<R>::T *, int,     \
                                                 int, cudaStream_t);                                            \
    template cudaError_t launch_residual_restrict<R, CT<R>::T>(const DevOp<R> &, int, const CT<R>::T *,          \
                                                                const CT<R>::T *, CT<R>::T *, cudaStream_t, bool, \
                                                                bool);                                          \
    template cudaError_t launch_prolong_add<R>(const int *, int, const CT<R>::T *, CT<R>::T *, cudaStream_t,      \
                                               const int *, bool);                                             \
    template cudaError_t launch_dense_solve<R>(const int *, int, int, const CT<R>::T *, const CT<R>::T *,        \
                                                CT<R>::T *, cudaStream_t);
INST_R(float)
INST_R(double)
template cudaError_t launch_apply<double, double2>(const DevOp<double> &, int, const double2 *, double2 *, cudaStream_t);
template cudaError_t launch_apply<double, float2>(const DevOp<double> &, int, const float2 *, double2 *, cudaStream_t);
template cudaError_t launch_apply<float, float2>(const DevOp<float> &, int, const float2 *, float2 *, cudaStream_t);
template cudaError_t launch_convert<double2, float2>(size_t, const double2 *, float2 *, cudaStream_t);
template cudaError_t launch_convert<float2, double2>(size_t, const float2 *, double2 *, cudaStream_t);
template cudaError_t launch_convert<double2, double2>(size_t, const double2 *, double2 *, cudaStream_t);
template cudaError_t launch_convert<float2, float2>(size_t, const float2 *, float2 *, cudaStream_t);
template cudaError_t launch_zero<double2>(size_t, double2 *, cudaStream_t);
template cudaError_t launch_zero<float2>(size_t, float2 *, cudaStream_t);

// ------------------------------------------------------------------------------ 1 / diagonal
namespace {
template <typename R> __global__ void k_diag_inv(OpView<R> o, int dim, R omega, typename CT<R>::T *__restrict__ dinv) {
    pdl_enter();
    typedef typename CT<R>::T C;
    const size_t sz = (size_t)o.nx * o.ny, n = sz * (dim == 3 ? o.nz : 1);
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < n; p += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(p / sz), x = (int)(p % o.nx), y = (int)(p % sz / o.nx);
        C v = mk(R(0), R(0));
        if (x >= 1 && x <= o.nx - 2 && y >= 1 && y <= o.ny - 2 && (dim == 2 || (k >= 1 && k <= o.nz - 2))) {
            C d = cadd(o.cx[3 * x + 1], o.cy[3 * y + 1]);
            if (dim == 3) d = cadd(d, o.cz[3 * k + 1]);
            d = cadd(d, cadd(cscale(o.bk, o.k2[p]), o.c));
            v = cinv(d);
            if constexpr (sizeof(R) == sizeof(double)) v = cscale(v, omega);
        }
        dinv[p] = v;
    }
}
}  // namespace

template <typename R>
cudaError_t launch_diag_inv(const DevOp<R> &op, int dim, R omega, typename CT<R>::T *dinv, cudaStream_t s) {
    const size_t n = (size_t)op.n[0] * op.n[1] * (dim == 3 ? op.n[2] : 1);
    launch_pdl(k_diag_inv<R>, (unsigned)std::min<size_t>(cdiv(n, 256), 152 * 8), 256, 0, s, view(op), dim, omega, dinv);
    return cudaGetLastError();
}
template cudaError_t launch_diag_inv<float>(const DevOp<float> &, int, float, float2 *, cudaStream_t);
template cudaError_t launch_diag_inv<double>(const DevOp<double> &, int, double, double2 *, cudaStream_t);
