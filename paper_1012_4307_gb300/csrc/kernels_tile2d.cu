// One level's way down and its way up of a 2D cycle in one launch each, for either precision,
// omega-Jacobi or omega-red-black, one or two sweeps, from zero or from a guess:
//   pre:  u_out = sweeps of M u = b (from zero or u_in), rc = FW(b - M u_out)
//   post: u_out = sweeps of (u_in + P ec)
// (the complex64 V(2,2) omega-Jacobi cycle from zero has kernels of its own, k_pre2_restrict and
// k_prolong_post2 in kernels_mg.cu, whose tiles are compile-time constants).
//
// What bounds it: in complex128 the FP64 units (two lanes per SM and clock), so the arithmetic is
// the one with the fewest operations: a sweep is u' = (1 - omega) u + (omega / D) (b - off) with
// omega / D formed once per handle (24 operations per node; about 55 with the diagonal assembled
// and divided by in every sweep), and each fine residual is formed once per tile instead of once
// for each of the coarse nodes it weighs on (9 residuals per coarse node, 2.25 per fine node, in a
// serial chain that took 20 us even on the smallest levels).  Small levels are bound by the latency
// of their launches and phases: two launches per visit instead of four or five.
//
// A block owns tcx x tcy coarse nodes and the fine nodes 2 I0 - 1 .. 2 I0 + 2 tcx - 2 (same in y),
// and keeps the iterate of its region (the owned nodes and the halo that the sweeps and the residual
// consume) in shared memory; b, omega / D and k^2 are read from global memory where they are used
// (each once or twice per node).  Every phase runs over the part of its range inside the grid as a
// flat index, so that no lane idles on halo columns (a masked lane costs as much FP64 time as a
// live one); a red-black half-sweep takes only its own colour's nodes.  Sizes are launch arguments:
// the code is the same for every tile.
// Measured on GB300: 641^2 complex128 F cycle with one sweep each way 755 -> 599 us, Bi-CGSTAB on 385^2
// (two such cycles an iteration) 57.5 -> 42.0 ms; with the residual after one sweep from zero formed
// without the diagonal and real coefficients taken as real (block-uniform), 599 -> 538 us; with the
// coefficients staged before the wait for the kernel ahead, 525 -> 511 us.
#include <algorithm>

#include "helm_internal.h"

namespace {

template <typename R> struct T2 {
    typedef typename CT<R>::T C;
    const C *cx, *cy;   // coefficient triples
    const R *k2;
    const C *di;        // complex128: omega / diagonal; complex64: 1 / diagonal
    C bk, c;
    R omega;
    int nx, ny, ncx, ncy;
    int tcx, tcy;       // coarse nodes per tile
    int nu, zero, s;    // sweeps, start from zero, stencil steps the sweeps take
    const C *b, *u_in;
    C *u_out, *rc;      // rc: pre only
    const C *ec;        // post only
    const int *gate;
};

// q / m rounded down for 0 <= q < 2^20 (see the cluster tail).
__device__ __forceinline__ int quot(int q, float rm) { return __float2int_rz(((float)q + 0.5f) * rm); }

struct Range {
    int x0, x1, y0, y1;  // inclusive; empty when x1 < x0 or y1 < y0
};
// f(x, y) for every node of the range, flat over the block
template <typename F> __device__ __forceinline__ void over(const Range &r, F f) {
    const int w = r.x1 - r.x0 + 1, n = w * (r.y1 - r.y0 + 1);
    if (w <= 0) return;
    const float rw = 1.0f / (float)w;
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
        const int y = quot(q, rw);
        f(r.x0 + q - y * w, r.y0 + y);
    }
}
// ... of one colour (0: even x + y)
template <typename F> __device__ __forceinline__ void over_colour(const Range &r, int colour, F f) {
    const int w = (r.x1 - r.x0 + 2) / 2, n = w * (r.y1 - r.y0 + 1);
    if (r.x1 < r.x0) return;
    const float rw = 1.0f / (float)w;
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
        const int yy = quot(q, rw), y = r.y0 + yy;
        const int x = r.x0 + ((r.x0 + y + colour) & 1) + 2 * (q - yy * w);
        if (x <= r.x1) f(x, y);
    }
}

// The block's view of its region in shared memory: node (x, y) at (x - X0) + W (y - Y0).
template <typename R> struct Region {
    typedef typename CT<R>::T C;
    const T2<R> &A;
    int X0, Y0, W, H;
    C *cx, *cy, *ua, *ub;
    bool real;  // complex128: the off-diagonal coefficients of every column and row of the region are real
    __device__ __forceinline__ int at(int x, int y) const { return (x - X0) + W * (y - Y0); }
    // [x0 - e, x1 + e] x [y0 - e, y1 + e] inside the grid's interior
    __device__ __forceinline__ Range grow(const Range &r, int e) const {
        return Range{max(r.x0 - e, 1), min(r.x1 + e, A.nx - 2), max(r.y0 - e, 1), min(r.y1 + e, A.ny - 2)};
    }
    // coefficients and a zero iterate; ends with a block barrier
    __device__ __forceinline__ void stage() {
        int im = sizeof(R) == sizeof(float);
        for (int q = threadIdx.x; q < 3 * W; q += blockDim.x) {
            const int x = X0 + q / 3;
            cx[q] = (x >= 1 && x <= A.nx - 2) ? __ldg(&A.cx[3 * X0 + q]) : mk(R(0), R(0));
            im |= q % 3 != 1 && !is_zero(cx[q].y);
        }
        for (int q = threadIdx.x; q < 3 * H; q += blockDim.x) {
            const int y = Y0 + q / 3;
            cy[q] = (y >= 1 && y <= A.ny - 2) ? __ldg(&A.cy[3 * Y0 + q]) : mk(R(0), R(0));
            im |= q % 3 != 1 && !is_zero(cy[q].y);
        }
        for (int q = threadIdx.x; q < 2 * W * H; q += blockDim.x) ua[q] = mk(R(0), R(0));  // ua, then ub
        real = !__syncthreads_or(im);
    }
    // b minus the off-diagonal part of M u at (x, y)
    template <bool REAL> __device__ __forceinline__ C rhs_off(const C *u, C b, int x, int y) const {
        const int p = at(x, y), ix = 3 * (x - X0), iy = 3 * (y - Y0);
        return axis_sub<REAL>(cy[iy], cy[iy + 2], u[p - W], u[p + W],
                              axis_sub<REAL>(cx[ix], cx[ix + 2], u[p - 1], u[p + 1], b));
    }
    // one relaxed update: (1 - omega) u + (omega / D) (b - off)
    template <bool REAL> __device__ __forceinline__ C relax(const C *u, int x, int y) const {
        const size_t g = (size_t)x + (size_t)A.nx * y;
        const C b = __ldg(&A.b[g]);
        C w = __ldg(&A.di[g]);
        if constexpr (sizeof(R) == sizeof(float)) w = cscale(w, A.omega);
        return cfma(w, rhs_off<REAL>(u, b, x, y), cscale(u[at(x, y)], R(1) - A.omega));
    }
    __device__ __forceinline__ C relax_zero(int x, int y) const {
        const size_t g = (size_t)x + (size_t)A.nx * y;
        const C v = cmul(__ldg(&A.b[g]), __ldg(&A.di[g]));
        return sizeof(R) == sizeof(float) ? cscale(v, A.omega) : v;
    }
};

template <typename R>
__device__ __forceinline__ Region<R> region(const T2<R> &A, unsigned char *smem, int X0, int Y0, int W, int H) {
    typedef typename CT<R>::T C;
    Region<R> G{A, X0, Y0, W, H, nullptr, nullptr, nullptr, nullptr, false};
    C *p = (C *)smem;
    G.ua = p; p += W * H;
    G.ub = p; p += W * H;
    G.cx = p; p += 3 * W;
    G.cy = p;
    return G;
}

template <typename R, bool RB, bool REAL> __device__ __forceinline__ void tile_pre(const T2<R> &A, const Region<R> &G, const Range &res) {
    typedef typename CT<R>::T C;
    const int I0 = 1 + blockIdx.x * A.tcx, J0 = 1 + blockIdx.y * A.tcy, e = 1 + A.s;
    C *cur = G.ua, *oth = G.ub;
    int left = e;  // the iterate is right on grow(res, left)
    if (!A.zero) {
        over(G.grow(res, left), [&](int x, int y) { cur[G.at(x, y)] = A.u_in[(size_t)x + (size_t)A.nx * y]; });
        __syncthreads();
    }
    for (int k = 0; k < A.nu; k++) {
        const bool z0 = A.zero && k == 0;
        if constexpr (RB) {
            for (int colour = 0; colour < 2; colour++) {
                if (z0 && colour == 0) {
                    over_colour(G.grow(res, left), 0, [&](int x, int y) { cur[G.at(x, y)] = G.relax_zero(x, y); });
                } else {
                    left--;
                    over_colour(G.grow(res, left), colour, [&](int x, int y) { cur[G.at(x, y)] = G.template relax<REAL>(cur, x, y); });
                }
                __syncthreads();
            }
        } else if (z0) {
            over(G.grow(res, left), [&](int x, int y) { cur[G.at(x, y)] = G.relax_zero(x, y); });
            __syncthreads();
        } else {
            left--;
            over(G.grow(res, left), [&](int x, int y) { oth[G.at(x, y)] = G.template relax<REAL>(cur, x, y); });
            __syncthreads();
            C *t = cur;
            cur = oth;
            oth = t;
        }
    }
    // residual (zero off the interior), and the owned nodes of the iterate
    for (int q = threadIdx.x; q < (2 * A.tcx + 1) * (2 * A.tcy + 1); q += blockDim.x) {
        const int w = 2 * A.tcx + 1, yy = quot(q, 1.0f / (float)w), x = res.x0 + q - yy * w, y = res.y0 + yy;
        C r = mk(R(0), R(0));
        if (x <= A.nx - 2 && y <= A.ny - 2) {
            const size_t g = (size_t)x + (size_t)A.nx * y;
            const int p = G.at(x, y);
            const C uc = cur[p];
            if (A.zero && A.nu == 1) {
                // after one sweep from zero D u = omega b (red-black: omega (b - off) at the second
                // colour), so no diagonal is formed: r = (1 - omega) b - off, or (1 - omega) (b - off)
                const C bv = __ldg(&A.b[g]);
                const R q1 = R(1) - A.omega;
                if (RB && ((x + y) & 1)) r = cscale(G.template rhs_off<REAL>(cur, bv, x, y), q1);
                else r = G.template rhs_off<REAL>(cur, cscale(bv, q1), x, y);
            } else {
                const C d = cadd(cadd(G.cx[3 * (x - G.X0) + 1], G.cy[3 * (y - G.Y0) + 1]),
                                 cadd(cscale(A.bk, __ldg(&A.k2[g])), A.c));
                r = csub(G.template rhs_off<REAL>(cur, __ldg(&A.b[g]), x, y), cmul(d, uc));
            }
            if (x < res.x1 && y < res.y1) A.u_out[g] = uc;
        }
        oth[G.at(x, y)] = r;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < A.tcx * A.tcy; q += blockDim.x) {
        const int cy = quot(q, 1.0f / (float)A.tcx), I = I0 + q - cy * A.tcx, J = J0 + cy;
        if (I > A.ncx - 2 || J > A.ncy - 2) continue;
        const C *r1 = oth + G.at(2 * I, 2 * J), *r0 = r1 - G.W, *r2 = r1 + G.W;
        // (1,2,1)/4 along x on each of the three rows, then along y
        const C a0 = cadd(cadd(r0[-1], r0[1]), cscale(r0[0], R(2)));
        const C a1 = cadd(cadd(r1[-1], r1[1]), cscale(r1[0], R(2)));
        const C a2 = cadd(cadd(r2[-1], r2[1]), cscale(r2[0], R(2)));
        A.rc[(size_t)I + (size_t)A.ncx * J] = cscale(cadd(cadd(a0, a2), cscale(a1, R(2))), R(0.0625));
    }
}

template <typename R, bool RB>
__global__ void __launch_bounds__(512) k_tile_pre(const __grid_constant__ T2<R> A) {
    extern __shared__ __align__(16) unsigned char t2_smem[];
    const int I0 = 1 + blockIdx.x * A.tcx, J0 = 1 + blockIdx.y * A.tcy;
    // residuals of the coarse nodes' neighbourhoods: owned fine nodes and one more row and column
    const Range res{2 * I0 - 1, 2 * I0 + 2 * A.tcx - 1, 2 * J0 - 1, 2 * J0 + 2 * A.tcy - 1};
    const int e = 1 + A.s;
    Region<R> G = region<R>(A, t2_smem, res.x0 - e, res.y0 - e, 2 * A.tcx + 1 + 2 * e, 2 * A.tcy + 1 + 2 * e);
    G.stage();  // coefficients only, which no kernel writes: before the wait for the kernel ahead
    pdl_enter();
    if (A.gate && *A.gate) return;
    if constexpr (sizeof(R) == sizeof(double)) {
        if (G.real) {
            tile_pre<R, RB, true>(A, G, res);
            return;
        }
    }
    tile_pre<R, RB, false>(A, G, res);
}

template <typename R, bool RB, bool REAL> __device__ __forceinline__ void tile_post(const T2<R> &A, const Region<R> &G, const Range &own) {
    typedef typename CT<R>::T C;
    const int e = A.s;
    C *cur = G.ua, *oth = G.ub;
    int left = e;
    // u + P ec: the mean of the four coarse values at floor / ceil of x / 2 and y / 2
    over(G.grow(own, left), [&](int x, int y) {
        const size_t ya = (size_t)A.ncx * (y >> 1), yb = (size_t)A.ncx * ((y + 1) >> 1);
        const int xa = x >> 1, xb = (x + 1) >> 1;
        const C c = cadd(cadd(A.ec[ya + xa], A.ec[ya + xb]), cadd(A.ec[yb + xa], A.ec[yb + xb]));
        cur[G.at(x, y)] = cadd(A.u_in[(size_t)x + (size_t)A.nx * y], cscale(c, R(0.25)));
    });
    __syncthreads();
    for (int k = 0; k < A.nu; k++) {
        const bool last = k + 1 == A.nu;
        if constexpr (RB) {
            left--;
            over_colour(G.grow(own, left), 0, [&](int x, int y) { cur[G.at(x, y)] = G.template relax<REAL>(cur, x, y); });
            __syncthreads();
            left--;
            if (last) {
                over_colour(G.grow(own, 0), 1, [&](int x, int y) { A.u_out[(size_t)x + (size_t)A.nx * y] = G.template relax<REAL>(cur, x, y); });
                over_colour(G.grow(own, 0), 0, [&](int x, int y) { A.u_out[(size_t)x + (size_t)A.nx * y] = cur[G.at(x, y)]; });
            } else {
                over_colour(G.grow(own, left), 1, [&](int x, int y) { cur[G.at(x, y)] = G.template relax<REAL>(cur, x, y); });
                __syncthreads();
            }
        } else {
            left--;
            if (last) {
                over(G.grow(own, 0), [&](int x, int y) { A.u_out[(size_t)x + (size_t)A.nx * y] = G.template relax<REAL>(cur, x, y); });
            } else {
                over(G.grow(own, left), [&](int x, int y) { oth[G.at(x, y)] = G.template relax<REAL>(cur, x, y); });
                __syncthreads();
                C *t = cur;
                cur = oth;
                oth = t;
            }
        }
    }
}

template <typename R, bool RB>
__global__ void __launch_bounds__(512) k_tile_post(const __grid_constant__ T2<R> A) {
    extern __shared__ __align__(16) unsigned char t2_smem[];
    const int I0 = 1 + blockIdx.x * A.tcx, J0 = 1 + blockIdx.y * A.tcy;
    const Range own{2 * I0 - 1, 2 * I0 + 2 * A.tcx - 2, 2 * J0 - 1, 2 * J0 + 2 * A.tcy - 2};
    const int e = A.s;
    Region<R> G = region<R>(A, t2_smem, own.x0 - e, own.y0 - e, 2 * A.tcx + 2 * e, 2 * A.tcy + 2 * e);
    G.stage();  // coefficients only, which no kernel writes: before the wait for the kernel ahead
    pdl_enter();
    if (A.gate && *A.gate) return;
    if constexpr (sizeof(R) == sizeof(double)) {
        if (G.real) {
            tile_post<R, RB, true>(A, G, own);
            return;
        }
    }
    tile_post<R, RB, false>(A, G, own);
}

// Coarse nodes per tile: the shape with the least time by the model (blocks per SM, at least one) x
// (nodes of the widest phase).  Large levels take the large tile (least halo), small ones the tile
// that spreads them over the SMs.
void pick_tile(int nx, int ny, int e, int &tcx, int &tcy) {
    static const int shapes[4][2] = {{16, 8}, {8, 8}, {8, 4}, {4, 4}};
    double best = 0;
    tcx = 0;
    for (const auto &t : shapes) {
        const double blocks = (double)cdiv(nx - 2, 2 * t[0]) * cdiv(ny - 2, 2 * t[1]);
        const double cost = std::max(1.0, blocks / 152.0) * (2 * t[0] + 1 + 2 * e) * (2 * t[1] + 1 + 2 * e);
        if (tcx == 0 || cost < 0.97 * best) {
            best = cost;
            tcx = t[0];
            tcy = t[1];
        }
    }
}

template <typename R> T2<R> args(const DevOp<R> &op, R omega, int nu, int rb, int zero) {
    T2<R> A{};
    A.cx = op.coef[0]; A.cy = op.coef[1]; A.k2 = op.k2; A.di = op.dinv; A.bk = op.bk; A.c = op.c;
    A.omega = omega;
    A.nx = op.n[0]; A.ny = op.n[1]; A.ncx = (op.n[0] + 1) / 2; A.ncy = (op.n[1] + 1) / 2;
    A.nu = nu;
    A.zero = zero;
    A.s = (rb ? 2 : 1) * nu - (zero ? 1 : 0);
    A.gate = op.gate;
    return A;
}

template <typename R, void (*KERNEL)(T2<R>)> cudaError_t launch_tile(T2<R> &A, int e, bool pre, cudaStream_t s) {
    pick_tile(A.nx, A.ny, e, A.tcx, A.tcy);
    const int own = pre ? 1 : 0;
    const size_t W = 2 * A.tcx + own + 2 * e, H = 2 * A.tcy + own + 2 * e;
    const size_t smem = (2 * W * H + 3 * (W + H)) * sizeof(typename CT<R>::T);
    static bool attr = false;
    if (!attr) {
        const cudaError_t err = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
        if (err != cudaSuccess) return err;
        attr = true;
    }
    // threads: the fewest passes over the last phase with at most 512, then the fewest warps
    const int n = (2 * A.tcx + own) * (2 * A.tcy + own), passes = cdiv(n, 512);
    const int nt = cdiv(cdiv(n, passes), 32) * 32;
    launch_pdl(KERNEL, dim3(cdiv(A.nx - 2, 2 * A.tcx), cdiv(A.ny - 2, 2 * A.tcy)), dim3(nt), smem, s, A);
    return cudaGetLastError();
}

}  // namespace

bool tile2d_ok(const int n[3], int dim, int nu) { return dim == 2 && nu >= 1 && nu <= 2 && n[0] >= 5 && n[1] >= 5; }

template <typename R>
cudaError_t launch_tile_pre(const DevOp<R> &op, R omega, int nu, int rb, const typename CT<R>::T *b,
                            const typename CT<R>::T *u_in, typename CT<R>::T *u_out, typename CT<R>::T *rc,
                            cudaStream_t s) {
    if (!tile2d_ok(op.n, 2, nu) || !op.dinv || u_in == u_out) return cudaErrorInvalidValue;
    T2<R> A = args<R>(op, omega, nu, rb, u_in ? 0 : 1);
    A.b = b; A.u_in = u_in; A.u_out = u_out; A.rc = rc;
    return rb ? launch_tile<R, k_tile_pre<R, true>>(A, 1 + A.s, true, s)
              : launch_tile<R, k_tile_pre<R, false>>(A, 1 + A.s, true, s);
}
template <typename R>
cudaError_t launch_tile_post(const DevOp<R> &op, R omega, int nu, int rb, const typename CT<R>::T *b,
                             const typename CT<R>::T *u_in, typename CT<R>::T *u_out, const typename CT<R>::T *ec,
                             cudaStream_t s) {
    if (!tile2d_ok(op.n, 2, nu) || !op.dinv || u_in == u_out) return cudaErrorInvalidValue;
    T2<R> A = args<R>(op, omega, nu, rb, 0);
    A.b = b; A.u_in = u_in; A.u_out = u_out; A.ec = ec;
    return rb ? launch_tile<R, k_tile_post<R, true>>(A, A.s, false, s)
              : launch_tile<R, k_tile_post<R, false>>(A, A.s, false, s);
}
#define INST(R)                                                                                                   \
    template cudaError_t launch_tile_pre<R>(const DevOp<R> &, R, int, int, const CT<R>::T *, const CT<R>::T *,    \
                                            CT<R>::T *, CT<R>::T *, cudaStream_t);                                \
    template cudaError_t launch_tile_post<R>(const DevOp<R> &, R, int, int, const CT<R>::T *, const CT<R>::T *,   \
                                             CT<R>::T *, const CT<R>::T *, cudaStream_t);
INST(float)
INST(double)
