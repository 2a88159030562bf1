// Rotation of one column of the Hessenberg matrix by one warp (used by the single and the batched kernel
// of kernels_krylov.cu; the host compiles it too, to run its lanes one after another).
#pragma once

#include "helm_internal.h"

// Complex Givens rotations G = [c s; -conj(s) c] (c real) on column j of the Hessenberg
// matrix (column-major, leading dimension ldh); see Saad, Iterative Methods for Sparse Linear
// Systems, Section 6.5.9 for the real case.
// Called by one warp.  A warp's FP64 instruction takes 64 clocks of its scheduler however few lanes
// are live, so the chain is written for few instructions: the lanes stage column j of H (j + 2
// entries) and the earlier rotations in shared memory; each rotation is three multiply-adds, lanes 0
// .. 3 forming the real and imaginary parts of its two outputs; the new rotation's moduli and
// quotients are formed side by side in different lanes; and est[j] = |g_{j+1}| / ||f|| is est[j-1]
// times the new rotation's |s| = |b| / t.  (One lane doing all of it took 12.8 us per step at j = 13.)
// est_host (may be null): pinned host memory, where est[j] is also stored, so that the host reads
// the estimate once the step's event has fired, with no copy in the step (a device-to-host copy
// node cost about 7 us per step at the end of every replayed step graph).
// tol, stop (may be null): *stop = 1 when est[j] <= *tol or is not a number.
__device__ __forceinline__ void givens_body(double2 *H, int ldh, int j, double *cs, double2 *sn, double2 *g,
                                            const double2 *fnorm_dev, double *est, double *est_host = nullptr,
                                            const double *tol = nullptr, int *stop = nullptr) {
    __shared__ double2 colS[66], snS[64];
    __shared__ double csS[64];
    const int lane = threadIdx.x & 31;
    constexpr unsigned all = 0xffffffffu;
    double2 *col = H + (size_t)ldh * j;
    for (int i = lane; i <= j + 1; i += 32) colS[i] = col[i];
    for (int i = lane; i < j; i += 32) {
        csS[i] = cs[i];
        snS[i] = sn[i];
    }
    const double2 gj = g[j];
    const double fnorm = fnorm_dev->x, before = j > 0 ? est[j - 1] : 0.0;
    __syncwarp();
    double2 a = colS[0];
    __syncwarp();  // every lane holds the entry before lanes 0 and 1 store the rotated one over it
    for (int i = 0; i < j; i++) {
        const double2 b = colS[i + 1], s = snS[i];
        const double c = csS[i];
        // lanes 0, 1: c a + s b;  lanes 2, 3: c b - conj(s) a  (real, imaginary)
        const bool im = lane & 1, second = lane & 2;
        const double2 u = second ? b : a, v = second ? make_double2(-a.x, -a.y) : b;
        const double p = im ? u.y : u.x, q = im ? v.y : v.x;
        double r = im ? v.x : -v.y;
        if (second) r = -r;
        const double o = fma(c, p, fma(s.x, q, s.y * r));
        if (lane < 2) ((double *)&colS[i])[lane] = o;
        a = make_double2(__shfl_sync(all, o, 2), __shfl_sync(all, o, 3));
    }
    const double2 b = colS[j + 1];
    __syncwarp();
    // lane 0: |a|, lane 1: |b|
    const double m = lane == 0 ? hypot(a.x, a.y) : hypot(b.x, b.y);
    const double na = __shfl_sync(all, m, 0), nb = __shfl_sync(all, m, 1);
    const double t = hypot(na, nb);
    // lanes 0 .. 4: c = |a| / t, a / |a|, 1 / t, |s| = |b| / t;  lane 5 (j = 0): |g_0| / ||f||
    const double num = lane == 0 ? na : lane == 1 ? a.x : lane == 2 ? a.y : lane == 3 ? 1.0 : lane == 4 ? nb : fabs(gj.x);
    const double den = lane == 1 || lane == 2 ? na : lane == 5 ? fnorm : t;
    const double quo = num / den;
    double c = __shfl_sync(all, quo, 0);
    const double2 ua = make_double2(__shfl_sync(all, quo, 1), __shfl_sync(all, quo, 2));
    const double rt = __shfl_sync(all, quo, 3);
    double sm = __shfl_sync(all, quo, 4);
    const double e0 = __shfl_sync(all, quo, 5);
    double2 s;
    if (na == 0.0) {
        c = 0.0;
        s = make_double2(1.0, 0.0);
        sm = 1.0;
    } else {
        s = cscale(cmul(ua, make_double2(b.x, -b.y)), rt);
    }
    if (lane == 0) {
        cs[j] = c;
        sn[j] = s;
        colS[j] = cadd(cscale(a, c), cmul(s, b));
        colS[j + 1] = make_double2(0.0, 0.0);
        g[j + 1] = cmul(make_double2(-s.x, s.y), gj);
        g[j] = cscale(gj, c);
        // g_0 = (||r0||, 0)
        const double e = (j > 0 ? before : e0) * sm;
        est[j] = e;
        if (est_host) est_host[j] = e;
        if (stop && !(e > *tol)) *stop = 1;
    }
    __syncwarp();
    for (int i = lane; i <= j + 1; i += 32) col[i] = colS[i];
}
