// Delayed CGS2 (DCGS2) coefficient step (run by the last block of the reduction in kernels_krylov.cu),
// and the last-block protocol that the Krylov passes share.
#pragma once

#include "helm_internal.h"

__device__ __forceinline__ double warp_sum_d(double v) {
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// DCGS2 coefficients of step j (Swirydowicz, Langou, Ananthan, Yang & Thomas,
// "Low synchronization Gram-Schmidt and GMRES algorithms", 2020; Bielich et al. 2022).
// Basis slot j holds x = alpha u: the once-orthogonalised vector of step j - 1, not normalised
// (alpha = alpha2[j].x its norm; slot 0 holds the final v_0 and alpha = 1).  From
// hv[i] = V_i^H x (i <= j; hv[j] = x^H x) and, with has_w, hv[j + 1 + i] = V_i^H w (i <= j):
//   u = sum_{i<j} a_i v_i + nu v_j,  a_i = hv[i] / alpha,  nu = sqrt(hv[j] / alpha^2 - |a|^2)
//   (nu = 1 for j = 0, where slot 0 already holds the final v_0);
//   column j - 1 of H, first-pass entries plus alpha a, gets its final values and
//   H[j][j-1] = alpha nu;
//   column j: c_i = hv[j+1+i] (i < j), H[j][j] = v_j^H w = (hv[2j+1] / alpha - a^H c) / nu;
//   with s = H[j][j] / nu, the update pass forms v_j = (x - sum V_i (alpha a_i)) / (alpha nu)
//   and w' = w - x (s / alpha) - sum V_i (c_i - a_i s): coef[i] = alpha a_i,
//   coef[j+i] = c_i - a_i s, coef[2j] = (1 / (alpha nu), small), coef[2j+1] = s / alpha,
//   where small = 1 when ||alpha a|| <= 2^-18 alpha nu, else 0.
// has_w = 2: the slot j + 1 vector and its inner products come from the unscaled x
// (w' = A M^{-1} x = alpha w, the preconditioner being linear): they are divided by alpha
// here, and coef[2j+2] = (1 / alpha, 0) tells the update pass to scale w' the same way
// (has_w = 1: coef[2j+2] = (1, 0)).
// Warps 0 and 1 of the block call it (j <= 64): warp 1 forms 1 / alpha while warp 0 (lane l takes i = l
// and, past 32 vectors, l + 32) forms the sums.  What it costs is the FP64 instructions of one warp, 64
// clocks of its scheduler each: the three sums go through one transposing butterfly (6 additions
// instead of 15) and the second half of the entries is passed over when there is none.  With that, the
// reduction's own sums transposed and the norm's last sum over the whole block (reduce_norm_block), a
// 1025^2 solve to 1e-10 (101 iterations) went from 20.8 to 20.5 ms.
__device__ __forceinline__ void dcgs2_coef_warps(int j, int has_w, const double2 *hv, const double2 *alpha2,
                                                 double2 *H, int ldh, double2 *coef) {
    __shared__ double ra_shared;
    const int lane = threadIdx.x & 31;
    const double al = j > 0 ? alpha2[j].x : 1.0;
    if (threadIdx.x >= 32) {
        if (lane == 0) ra_shared = 1.0 / al;
        asm volatile("bar.sync 1, 64;" ::: "memory");
        return;
    }
    const int nk = j > 32 ? 2 : 1;
    double2 a[2], c[2];
    double s2 = 0.0, tr = 0.0, ti = 0.0;
#pragma unroll
    for (int k = 0; k < 2; k++) {
        if (k >= nk) break;
        const int i = lane + 32 * k;
        a[k] = i < j ? hv[i] : make_double2(0.0, 0.0);
        c[k] = has_w && i < j ? hv[j + 1 + i] : make_double2(0.0, 0.0);
        s2 = fma(a[k].x, a[k].x, fma(a[k].y, a[k].y, s2));
        // conj(a) c
        tr = fma(a[k].x, c[k].x, fma(a[k].y, c[k].y, tr));
        ti = fma(a[k].x, c[k].y, fma(-a[k].y, c[k].x, ti));
    }
    {
        // lanes 0-7: s2, 16-23: tr, the others: ti
        constexpr unsigned all = 0xffffffffu;
        const bool up = lane & 16, odd = lane & 8;
        double m = (up ? tr : s2) + __shfl_xor_sync(all, up ? s2 : tr, 16);
        ti += __shfl_xor_sync(all, ti, 16);
        m = (odd ? ti : m) + __shfl_xor_sync(all, odd ? m : ti, 8);
        for (int off = 4; off > 0; off >>= 1) m += __shfl_xor_sync(all, m, off);
        s2 = __shfl_sync(all, m, 0);
        tr = __shfl_sync(all, m, 16);
        ti = __shfl_sync(all, m, 8);
    }
    asm volatile("bar.sync 1, 64;" ::: "memory");
    const double ra = ra_shared, rw = has_w == 2 ? ra : 1.0;
    double nu = 1.0;
    if (j > 0) {
        nu = sqrt(fmax((hv[j].x - s2) * (ra * ra), 1e-300));
        double2 *col = H + (size_t)ldh * (j - 1);
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const int i = lane + 32 * k;
            if (k < nk && i < j) col[i] = cadd(col[i], a[k]);  // alpha a_i = hv[i]
        }
        if (lane == 0) col[j] = make_double2(al * nu, 0.0);
    }
    if (!has_w) return;
    const double rt = rw * ra;
    const double2 t = make_double2((hv[2 * j + 1].x - tr) * rt, (hv[2 * j + 1].y - ti) * rt);
    const double rn = 1.0 / nu;
    const double2 hjj = cscale(t, rn);
    const double2 sf = cscale(hjj, rn), sa = cscale(sf, ra);
    double2 *col = H + (size_t)ldh * j;
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const int i = lane + 32 * k;
        if (k < nk && i < j) {
            const double2 ck = cscale(c[k], rw);
            col[i] = ck;
            coef[i] = a[k];
            coef[j + i] = csub(ck, cmul(a[k], sa));
        }
    }
    if (lane == 0) {
        col[j] = hjj;
        // small correction (||alpha a|| <= 2^-18 alpha nu): the update may form sum V_i (alpha a_i)
        // in FP32
        const double xn = al * nu;
        coef[2 * j] = make_double2(rn * ra, s2 <= 0x1p-36 * xn * xn ? 1.0 : 0.0);
        coef[2 * j + 1] = sa;
        coef[2 * j + 2] = make_double2(rw, 0.0);
    }
}

// Last-block-done protocol: every block of a pass has written its partials; the block that takes the
// last ticket (the others return false) reduces them in a fixed order and resets the ticket for the
// next launch.  Deterministic like a reduction kernel of its own.
__device__ __forceinline__ bool last_block(unsigned *ticket, unsigned nblocks) {
    __shared__ bool is_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = atomicAdd(ticket, 1u) == nblocks - 1;
    __syncthreads();
    if (is_last) __threadfence();
    return is_last;
}
// *out = (sqrt(sum of the G partials' real parts), 0), by a block of T threads in a fixed tree.
template <int T>
__device__ __forceinline__ void reduce_norm_block(const double2 *partials, int G, double2 *out) {
    __shared__ double red[T / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double s = 0.0;
#pragma unroll 4
    for (int b = threadIdx.x; b < G; b += T) s += partials[b].x;
    s = warp_sum_d(s);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (warp != 0) return;
    s = red[lane % (T / 32)];
    for (int off = T / 64; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) *out = make_double2(sqrt(s), 0.0);
}
