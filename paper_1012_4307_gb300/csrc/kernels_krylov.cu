// FP64 vector kernels of the outer Krylov solvers (flexible GMRES, Bi-CGSTAB) and the
// adjoint helpers.  All sums use a fixed grid (a function of the vector length only) and a
// fixed reduction tree, so repeated runs give bit-identical results.
//
// Classical Gram-Schmidt runs as two fused passes over the basis:
//   "dot"     h = V^H w and ||w||^2                 (k_mdot_norm, at most 8 basis vectors per block row)
//   "update"  w <- w - V h and ||w'||^2, same sweep (k_update_norm)
// followed by the DGKS test on the device (k_reduce_decide); the optional second pass reuses
// the same kernels, gated by the device flag, so the host never waits for the decision.
// On GB300 the FP64 units (about 2 FMA per SM per clock) bound these kernels, not DRAM.
#include "helm_internal.h"
#include "df_arith.h"
#include "dcgs2_coef.cuh"
#include "givens.cuh"

namespace {

constexpr int NT = 256;           // threads per block
constexpr int MAXBLK = 152 * 4;   // grid cap (4 blocks per SM on 152 SMs)

__device__ __forceinline__ double2 shfl_down2(double2 v, int off) {
    v.x = __shfl_down_sync(0xffffffffu, v.x, off);
    v.y = __shfl_down_sync(0xffffffffu, v.y, off);
    return v;
}

// Block-wide sums of NV complex values per thread (fixed tree: warp shuffles, then warps in
// order); thread t < NV returns sum t in out[t] (other threads: unspecified).
template <int NV>
__device__ __forceinline__ void block_sum(double2 (&v)[NV], double2 *out_shared) {
    __shared__ double2 red[NT / 32][NV];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NV; i++) {
        double2 x = v[i];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) x = cadd(x, shfl_down2(x, off));
        if (lane == 0) red[warp][i] = x;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double2 s = red[0][threadIdx.x];
        for (int w = 1; w < NT / 32; w++) s = cadd(s, red[w][threadIdx.x]);
        out_shared[threadIdx.x] = s;
    }
}

// Sums of N real values per thread over the warp (N a power of two, at most 32) by a transposing
// butterfly: at offsets 16, 8, ... a lane keeps half of its values, sends the other half to the lane
// at that offset and adds what it receives, so the values per lane halve at every level (N - 1 + the
// plain levels additions per lane instead of 5 N; on the FP64 units, where a warp's instruction takes
// 64 clocks of its scheduler, 5 N additions for 9 complex values cost more than the pass itself).
// Lanes l with l % (32 / N) == 0 end with the sum of value idx in v[0].
template <int M, int O, int N> __device__ __forceinline__ void transpose_level(double (&v)[N], int lane, int &idx) {
    if constexpr (M > 1) {
        const bool upper = (lane & O) != 0;
#pragma unroll
        for (int i = 0; i < M / 2; i++) {
            const double keep = upper ? v[i + M / 2] : v[i], send = upper ? v[i] : v[i + M / 2];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
        }
        if (upper) idx += M / 2;
    } else {
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], O);
    }
    if constexpr (O > 1) transpose_level<(M > 1 ? M / 2 : 1), O / 2>(v, lane, idx);
}
template <int N> __device__ __forceinline__ int warp_transpose_sum(double (&v)[N]) {
    int idx = 0;
    transpose_level<N, 16>(v, threadIdx.x & 31, idx);
    return idx;
}

// Block-wide sum of one real value per thread, in thread 0 (fixed tree).
__device__ __forceinline__ double block_sum_real(double v) {
    __shared__ double red[NT / 32];
    double a[1] = {v};
    warp_transpose_sum<1>(a);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a[0];
    __syncthreads();
    double s = red[0];
    if (threadIdx.x == 0)
        for (int w = 1; w < NT / 32; w++) s += red[w];
    return s;
}

// partials[b] = (sum |w[q]|^2, 0)
__global__ void __launch_bounds__(NT) k_norm2(size_t n, const double2 *__restrict__ w, double2 *__restrict__ partials) {
    pdl_enter();
    double acc = 0.0;
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const double2 wq = w[q];
        acc = fma(wq.x, wq.x, fma(wq.y, wq.y, acc));
    }
    acc = block_sum_real(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = make_double2(acc, 0.0);
}

// Pass "dot": partials[i * G + b] = sum_q conj(V_i[q]) w[q] (i < nv), and partials[nv * G + b] =
// (sum |w[q]|^2, 0).  Grid (G, chunks): block row y takes the vectors nv y / chunks ..
// nv (y + 1) / chunks - 1, at most CH, so the rows are even.  Skipped entirely when *gate == 0.
// Bound by the FP64 units (4 fused multiply-adds per vector and node): two blocks per SM, each thread
// many nodes (a grid of one or two nodes per thread spent most of its time in the block sums:
// 513^2, 13 vectors, 89 us per pass under ncu against 23 us of multiply-adds).
template <int CH>
__global__ void __launch_bounds__(NT, 2) k_mdot_norm(size_t n, const double2 *__restrict__ V, size_t ldv, int nv,
                                                     const double2 *__restrict__ w, double2 *__restrict__ partials,
                                                     const int *__restrict__ gate) {
    pdl_enter();
    if (gate && *gate == 0) return;
    __shared__ double red[NT / 32][2 * CH + 1];
    const int chunks = gridDim.y;
    const int i0 = nv * (int)blockIdx.y / chunks;
    const int cnt = nv * ((int)blockIdx.y + 1) / chunks - i0;
    const bool first = blockIdx.y == 0;
    double acc[2 * CH], nn[1] = {0.0};
#pragma unroll
    for (int t = 0; t < 2 * CH; t++) acc[t] = 0.0;
    const double2 *Vc = V + (size_t)i0 * ldv;
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const double2 wq = w[q];
        double2 v[CH];
        const double2 *p = Vc + q;
#pragma unroll
        for (int t = 0; t < CH; t++, p += ldv) v[t] = t < cnt ? *p : make_double2(0.0, 0.0);
        if (first) nn[0] = fma(wq.x, wq.x, fma(wq.y, wq.y, nn[0]));
#pragma unroll
        for (int t = 0; t < CH; t++)
            if (t < cnt) {
                acc[2 * t] = fma(v[t].x, wq.x, fma(v[t].y, wq.y, acc[2 * t]));
                acc[2 * t + 1] = fma(v[t].x, wq.y, fma(-v[t].y, wq.x, acc[2 * t + 1]));
            }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int idx = warp_transpose_sum<2 * CH>(acc);
    if ((lane & (32 / (2 * CH) - 1)) == 0) red[warp][idx] = acc[0];
    if (first) {
        warp_transpose_sum<1>(nn);
        if (lane == 0) red[warp][2 * CH] = nn[0];
    }
    __syncthreads();
    const int t = threadIdx.x, G = gridDim.x;
    if (t < 2 * cnt || (first && t == 2 * CH)) {
        double s = red[0][t];
        for (int x = 1; x < NT / 32; x++) s += red[x][t];
        if (t < 2 * CH) ((double *)(partials + (size_t)(i0 + (t >> 1)) * G + blockIdx.x))[t & 1] = s;
        else partials[(size_t)nv * G + blockIdx.x] = make_double2(s, 0.0);
    }
}

// Pass "update": w -= sum_{i < nv} V_i h_i, then partials[b] = (sum |w|^2, 0).  Gated.
// Bound by the FP64 units (4 multiply-adds per vector and node).  The second Gram-Schmidt pass only
// takes out what rounding left behind: with wnorm (||w|| so far) and ||h|| <= 2^-36 ||w||, the sum over
// the basis is formed in FP32 and subtracted in FP64: its rounding, at most nv 2^-24 ||h|| <= 2^-54 ||w|| for
// 64 vectors, stays below that of the FP64 chain, which rounds w once per vector; a larger correction
// takes the FP64 products.  The coefficients enter the sum divided by the power of two in ||w||, so that
// FP32's range is that of the correction's size relative to w, whatever the units of the problem.
// Measured against FP64 products in both passes (FGMRES(30) and its backward step to 1e-10, 97^2 .. 513^2
// and 49^3 .. 97^3, both precisions, three seeds): solutions 2e-15 .. 4e-14 apart, their errors against
// 64-bit results (1e-12 .. 2e-9, the tolerance's) equal; 513^2 13.88 -> 12.98 ms, 257^2 4.21 -> 4.13, 97^2 2.10 ->
// 2.12, 97^3 19.0 -> 17.7.
__global__ void __launch_bounds__(NT) k_update_norm(size_t n, const double2 *__restrict__ V, size_t ldv, int nv,
                                                    const double2 *__restrict__ h, double2 *__restrict__ w,
                                                    double2 *__restrict__ partials, const int *__restrict__ gate,
                                                    const double2 *__restrict__ wnorm) {
    pdl_enter();
    if (gate && *gate == 0) return;
    __shared__ double2 hs[64];
    __shared__ float2 hf[64];
    __shared__ int small_s;
    // unit = the power of two in ||w||, per = 1 / unit (both normal numbers, or no short form)
    double unit = 0.0, per = 0.0;
    if (wnorm) {
        const int e = (__double2hiint(wnorm->x) >> 20) & 0x7ff;
        if (e >= 1 && e <= 2045) {
            unit = __hiloint2double(e << 20, 0);
            per = __hiloint2double((2046 - e) << 20, 0);
        }
    }
    for (int i = threadIdx.x; i < nv; i += NT) {
        const double2 hi = h[i];
        hs[i] = hi;
        hf[i] = to_c(cscale(hi, per), 0.f);
    }
    if (threadIdx.x == 0) small_s = 0;
    __syncthreads();
    if (unit != 0.0 && threadIdx.x < 32) {
        double s2 = 0.0;
        for (int i = threadIdx.x; i < nv; i += 32) {
            const double2 r = cscale(hs[i], per);
            s2 = fma(r.x, r.x, fma(r.y, r.y, s2));
        }
        s2 = warp_sum_d(s2);
        const double r = wnorm->x * per;  // in [1, 2)
        if (threadIdx.x == 0) small_s = s2 <= 0x1p-72 * r * r;
    }
    __syncthreads();
    double acc = 0.0;
    if (small_s) {
        for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
            double2 wq = w[q];
            float2 c = make_float2(0.f, 0.f);
#pragma unroll 8
            for (int i = 0; i < nv; i++) {
                const float2 v = to_c(V[(size_t)i * ldv + q], 0.f), hh = hf[i];
                c.x = fmaf(v.x, hh.x, fmaf(-v.y, hh.y, c.x));
                c.y = fmaf(v.x, hh.y, fmaf(v.y, hh.x, c.y));
            }
            wq = make_double2(fma(-unit, to_double(c.x), wq.x), fma(-unit, to_double(c.y), wq.y));
            w[q] = wq;
            acc = fma(wq.x, wq.x, fma(wq.y, wq.y, acc));
        }
    } else {
        for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
            double2 wq = w[q];
#pragma unroll 8
            for (int i = 0; i < nv; i++) {
                const double2 v = V[(size_t)i * ldv + q];
                const double2 hh = hs[i];
                wq.x = fma(-v.x, hh.x, fma(v.y, hh.y, wq.x));
                wq.y = fma(-v.x, hh.y, fma(-v.y, hh.x, wq.y));
            }
            w[q] = wq;
            acc = fma(wq.x, wq.x, fma(wq.y, wq.y, acc));
        }
    }
    acc = block_sum_real(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = make_double2(acc, 0.0);
}

// out[i] = sum_b partials[i * nblk + b] in a fixed order for i = blockIdx.x; mode 0 '=',
// 1 '+=', 2 (sqrt(re), 0).  With out2, out2[i] = the plain sum (mode 2: its root) as well.  Gated.
__global__ void k_reduce(const double2 *__restrict__ partials, int nblk, double2 *__restrict__ out, int mode,
                         const int *__restrict__ gate, double *host_out, double2 *__restrict__ out2) {
    pdl_enter();
    if (gate && *gate == 0) return;
    __shared__ double2 sums[1];
    const int i = blockIdx.x;
    double2 s[1] = {make_double2(0.0, 0.0)};
    for (int b = threadIdx.x; b < nblk; b += NT) s[0] = cadd(s[0], partials[(size_t)i * nblk + b]);
    block_sum<1>(s, sums);
    if (threadIdx.x == 0) {
        const double2 t = sums[0];
        double2 r;
        if (mode == 0) r = t;
        else if (mode == 1) r = cadd(out[i], t);
        else r = make_double2(sqrt(t.x), 0.0);
        out[i] = r;
        if (out2) out2[i] = mode == 2 ? r : t;
        if (host_out) host_out[i] = r.x;
    }
}

// DGKS test after one classical Gram-Schmidt pass: the new norm ||w'|| = sqrt(sum partials)
// is written to *hnorm (which held ||w||^2 before the pass) and to *norm; re-orthogonalise (*flag = 1) when
// ||w'|| < eta ||w||, i.e. when the projection cancelled most of w.
__global__ void k_reduce_decide(const double2 *__restrict__ partials, int nblk, double2 *hnorm, int *flag, int *count,
                                double eta, double2 *norm) {
    pdl_enter();
    __shared__ double2 sums[1];
    double2 s[1] = {make_double2(0.0, 0.0)};
    for (int b = threadIdx.x; b < nblk; b += NT) s[0] = cadd(s[0], partials[b]);
    block_sum<1>(s, sums);
    if (threadIdx.x == 0) {
        const double before = sqrt(hnorm->x), after = sqrt(sums[0].x);
        const int redo = !(after >= eta * before);
        *flag = redo;
        if (redo) *count += 1;
        *hnorm = make_double2(after, 0.0);
        *norm = make_double2(after, 0.0);
    }
}

// y = x / scale; with b_out, its complex64 copy too (the next cycle's right-hand side)
__global__ void k_scale_inv(size_t n, const double2 *x, const double2 *__restrict__ scale, double2 *y,
                            float2 *__restrict__ b_out) {
    pdl_enter();
    const double s = scale[0].x;
    const double r = s != 0.0 ? 1.0 / s : 0.0;
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const double2 v = x[q], t = make_double2(v.x * r, v.y * r);
        y[q] = t;
        if (b_out) b_out[q] = to_c(t, 0.f);
    }
}

template <typename CZ>
__global__ void k_combine(size_t n, const CZ *__restrict__ Z, size_t ldz, int nz, const double2 *__restrict__ y,
                          double2 *__restrict__ x) {
    pdl_enter();
    __shared__ double2 ys[64];
    for (int i = threadIdx.x; i < nz; i += NT) ys[i] = y[i];
    __syncthreads();
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        double2 acc = x[q];
        for (int c = 0; c < nz; c++) acc = cfma(ys[c], to_c(Z[(size_t)c * ldz + q], 0.0), acc);
        x[q] = acc;
    }
}

// x += Z y for complex64 Z: the sum over the basis in double-FP32 on the FP32 units (products
// of the exact FP32 z with y split into float pairs are error-free, sums use TwoSum), added to
// x in FP64 once per node.  The FP64 form above is bound by the FP64 units (4 FMA per vector
// and node).
// With alpha, column c >= 1 of Z holds alpha_c z_c (alpha_c = alpha[c].x) and its weight is
// y_c / alpha_c.
__global__ void __launch_bounds__(NT) k_combine_df(size_t n, const float2 *__restrict__ Z, size_t ldz, int nz,
                                                   const double2 *__restrict__ y, const double2 *__restrict__ alpha,
                                                   double2 *__restrict__ x) {
    pdl_enter();
    __shared__ float4 ys[64];  // (re hi, re lo, im hi, im lo)
    for (int i = threadIdx.x; i < nz; i += NT) {
        const double r = (alpha && i > 0) ? 1.0 / alpha[i].x : 1.0;
        const ff a = ff_split(y[i].x * r), b = ff_split(y[i].y * r);
        ys[i] = make_float4(a.hi, a.lo, b.hi, b.lo);
    }
    __syncthreads();
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f;
#pragma unroll 4
        for (int c = 0; c < nz; c++) {
            const float2 z = Z[(size_t)c * ldz + q];
            const float4 y4 = ys[c];
            const ff yr{y4.x, y4.y}, yi{y4.z, y4.w};
            float p, e;
            // re += zr yr - zi yi ; im += zr yi + zi yr
            ff_prod_f(yr, z.x, p, e); ff_acc_prod(sr, cr, p, e);
            ff_prod_f(yi, z.y, p, e); ff_acc_prod(sr, cr, -p, -e);
            ff_prod_f(yi, z.x, p, e); ff_acc_prod(si, ci, p, e);
            ff_prod_f(yr, z.y, p, e); ff_acc_prod(si, ci, p, e);
        }
        const double2 xq = x[q];
        x[q] = make_double2(xq.x + (to_double(sr) + to_double(cr)), xq.y + (to_double(si) + to_double(ci)));
    }
}

__global__ void k_givens(double2 *H, int ldh, int j, double *cs, double2 *sn, double2 *g, const double2 *fnorm_dev,
                         double *est, double *est_host, const double *tol, int *stop) {
    pdl_enter();
    if (threadIdx.x >= 32 || blockIdx.x != 0) return;
    givens_body(H, ldh, j, cs, sn, g, fnorm_dev, est, est_host, tol, stop);
}

__global__ void k_cycle_start(double2 *g, int len, const double2 *beta, int *stop, double *tol_dev, double tol) {
    pdl_enter();
    for (int i = threadIdx.x; i < len; i += blockDim.x) g[i] = i == 0 ? *beta : make_double2(0.0, 0.0);
    if (threadIdx.x == 0) {
        if (stop) *stop = 0;
        if (tol_dev) *tol_dev = tol;
    }
}

// Batched rotation of column j (block z = problem), and the gather of every problem's estimate
// est[j] into out[problem] (-1 for inactive problems); out is pinned host memory, which the host
// reads once the step's event has fired.  A problem whose estimate meets *tol (or is not a
// number) is made inactive at once, so that the steps already queued behind this one skip it
// (the host, reading the same estimate, takes it out of the lockstep).
__global__ void k_givens_b(const BVec *__restrict__ tab, int j, double *out, const double *tol) {
    pdl_enter();
    const BVec &P = tab[blockIdx.z];
    if (threadIdx.x >= 32) return;
    if (*P.active == 0) {
        if (threadIdx.x == 0) out[blockIdx.z] = -1.0;
        return;
    }
    givens_body(P.H, P.ldh, j, P.cs, P.sn, P.g, P.fnorm, P.est);
    if (threadIdx.x == 0) {
        const double e = P.est[j];
        out[blockIdx.z] = e;
        if (tol && !(e > *tol)) *P.active = 0;
    }
}

// The reduction of the two-vector inner-product pass (block v sums value v of the partials in a
// fixed tree) followed, in the last block to finish, by the DCGS2 coefficient
// step of step j (see dcgs2_coef.cuh); the ticket returns to 0.
__device__ __forceinline__ void reduce_dcgs2_body(const double2 *__restrict__ partials, int nblk, double2 *hv,
                                                  unsigned *ticket, int j, const double2 *alpha2, double2 *H, int ldh,
                                                  double2 *coef, int has_w) {
    __shared__ double red[2 * NT / 32];
    const int i = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double2 *p = partials + (size_t)i * nblk;
    double v[2] = {0.0, 0.0};
#pragma unroll 2
    for (int b = threadIdx.x; b < nblk; b += NT) {
        v[0] += p[b].x;
        v[1] += p[b].y;
    }
    const int c = warp_transpose_sum<2>(v);
    if ((lane & 15) == 0) red[2 * warp + c] = v[0];
    __syncthreads();
    if (warp == 0) {
        // lane 2 w + c: component c of warp w
        static_assert(2 * NT / 32 == 16, "");
        double s = red[lane & 15];
        for (int off = 8; off > 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane < 2) ((double *)(hv + i))[lane] = s;
    }
    if (!last_block(ticket, gridDim.x)) return;
    if (threadIdx.x < 64) dcgs2_coef_warps(j, has_w, hv, alpha2, H, ldh, coef);
    if (threadIdx.x == 0) *ticket = 0u;
}

__global__ void k_reduce_dcgs2(const double2 *__restrict__ partials, int nblk, double2 *hv, unsigned *ticket, int j,
                               const double2 *alpha2, double2 *H, int ldh, double2 *coef, int has_w) {
    pdl_enter();
    reduce_dcgs2_body(partials, nblk, hv, ticket, j, alpha2, H, ldh, coef, has_w);
}

// Batched reduction + coefficient step of step j (block z = problem; the problem's dot pass
// had first[z + 1] - first[z] blocks, i.e. that many / groups per value).
__global__ void k_reduce_dcgs2_b(const BVec *__restrict__ tab, const unsigned *__restrict__ first, int groups, int j,
                                 int has_w) {
    pdl_enter();
    const BVec &P = tab[blockIdx.z];
    if (*P.active == 0) return;
    const int nblk = (int)((first[blockIdx.z + 1] - first[blockIdx.z]) / groups);
    reduce_dcgs2_body(P.partials, nblk, P.hv, P.tickets, j, P.alpha2, P.H, P.ldh, P.dcoef, has_w);
}

// y = R^{-1} g for the k x k upper-triangular leading block R of H (column-major, leading
// dimension ldh): R and g are staged in shared memory by the whole block, then one warp
// eliminates column by column (y_r = g_r / R_rr, then g_i -= R_ir y_r for i < r, lanes over i),
// with the reciprocals 1 / R_rr formed beforehand in parallel.
__global__ void __launch_bounds__(NT) k_backsolve(const double2 *H, int ldh, int k, const double2 *g, double2 *y) {
    pdl_enter();
    extern __shared__ double2 bs_smem[];
    double2 *R = bs_smem, *gs = bs_smem + (size_t)k * k;
    for (int q = threadIdx.x; q < k * k; q += blockDim.x) {
        const int c = q / k, r = q - c * k;
        R[q] = r <= c ? H[r + (size_t)ldh * c] : make_double2(0.0, 0.0);
    }
    for (int q = threadIdx.x; q < k; q += blockDim.x) gs[q] = g[q];
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    // the reciprocal diagonal first, all lanes at once; the elimination then only multiplies
    for (int r = lane; r < k; r += 32) R[r + (size_t)k * r] = cinv(R[r + (size_t)k * r]);
    __syncwarp();
    for (int r = k - 1; r >= 0; r--) {
        const double2 yr = cmul(gs[r], R[r + (size_t)k * r]);
        for (int i = lane; i < r; i += 32) gs[i] = csub(gs[i], cmul(R[i + (size_t)k * r], yr));
        if (lane == 0) y[r] = yr;
        __syncwarp();
    }
}

// Bi-CGSTAB scalar block (device): 0 rho, 1 rho_old, 2 alpha, 3 omega, 4 beta, 5 <rh,v>,
// 6 <t,s>, 7 <t,t>, 8 -alpha, 9 -omega, 11 flags (x: breakdown)
__device__ __forceinline__ void bicg_stage(int stage, double2 *sc) {
    const double2 zero = make_double2(0.0, 0.0);
    auto isz = [](double2 v) { return v.x == 0.0 && v.y == 0.0; };
    if (stage == 0) {            // beta = (rho / rho_old) (alpha / omega)
        if (isz(sc[0]) || isz(sc[1]) || isz(sc[3])) { sc[11].x = 1.0; sc[4] = zero; return; }
        sc[4] = cmul(cmul(sc[0], cinv(sc[1])), cmul(sc[2], cinv(sc[3])));
    } else if (stage == 1) {     // alpha = rho / <rh, v>
        if (isz(sc[5])) { sc[11].x = 1.0; sc[2] = zero; sc[8] = zero; return; }
        sc[2] = cmul(sc[0], cinv(sc[5]));
        sc[8] = make_double2(-sc[2].x, -sc[2].y);
    } else if (stage == 2) {     // omega = <t, s> / <t, t>; rho_old = rho
        if (sc[7].x == 0.0) { sc[11].x = 1.0; sc[3] = zero; sc[9] = zero; return; }
        sc[3] = cscale(sc[6], 1.0 / sc[7].x);
        sc[9] = make_double2(-sc[3].x, -sc[3].y);
        sc[1] = sc[0];
        if (isz(sc[3])) sc[11].x = 1.0;
    } else {                     // init: rho_old = alpha = omega = 1, flags = 0
        sc[1] = sc[2] = sc[3] = make_double2(1.0, 0.0);
        sc[11] = zero;
    }
}
__global__ void k_bicg_scalars(int stage, double2 *sc) {
    pdl_enter();
    if (threadIdx.x == 0 && blockIdx.x == 0) bicg_stage(stage, sc);
}

// The vector passes of an iteration, each one launch that also forms the inner products of what it
// writes; the last block to finish sums the blocks' partials in a fixed order and takes the scalar
// step (a dot, its reduction, the scalar kernel, the copy and the update as launches of their own
// took 39 + 5 + 3 + 5 us of a 385^2 iteration's four dots; now five passes an iteration, the two
// norms the host reads stored in pinned memory by the pass that forms them).

// v[0 .. N) summed over the grid into sum[0 .. N) (shared memory) of the last block, which returns
// true; partials: N x gridDim.x doubles.
template <int N>
__device__ __forceinline__ bool grid_sums(double (&v)[N], double *partials, unsigned *ticket, double (&sum)[N]) {
    __shared__ double red[NT / 32][N];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, G = gridDim.x;
    auto block = [&](double (&x)[N]) {
        const int idx = warp_transpose_sum<N>(x);
        if ((lane & (32 / N - 1)) == 0) red[warp][idx] = x[0];
        __syncthreads();
        double s = 0.0;
        if (threadIdx.x < N)
            for (int w = 0; w < NT / 32; w++) s += red[w][threadIdx.x];
        __syncthreads();
        return s;
    };
    const double s = block(v);
    if (threadIdx.x < N) partials[(size_t)threadIdx.x * G + blockIdx.x] = s;
    if (!last_block(ticket, G)) return false;
    double t[N];
#pragma unroll
    for (int k = 0; k < N; k++) {
        t[k] = 0.0;
        for (int b = threadIdx.x; b < G; b += NT) t[k] += __ldcg(&partials[(size_t)k * G + b]);
    }
    const double f = block(t);
    if (threadIdx.x < N) sum[threadIdx.x] = f;
    if (threadIdx.x == 0) *ticket = 0u;
    __syncthreads();
    return true;
}

// STAGE 1: <a, b> = <rh, v>, then alpha.  STAGE 2: <a, b> = <t, s> and <t, t>, then omega.
template <int STAGE>
__global__ void __launch_bounds__(NT) k_bicg_dots(size_t n, const double2 *__restrict__ a, const double2 *__restrict__ b,
                                                  double2 *sc, double *partials, unsigned *ticket) {
    pdl_enter();
    constexpr int N = STAGE == 1 ? 2 : 4;
    __shared__ double sum[N];
    double v[N];
#pragma unroll
    for (int k = 0; k < N; k++) v[k] = 0.0;
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const double2 x = a[q], y = b[q];
        v[0] = fma(x.x, y.x, fma(x.y, y.y, v[0]));
        v[1] = fma(x.x, y.y, fma(-x.y, y.x, v[1]));
        if constexpr (STAGE == 2) v[2] = fma(x.x, x.x, fma(x.y, x.y, v[2]));
    }
    if (!grid_sums<N>(v, partials, ticket, sum) || threadIdx.x != 0) return;
    sc[STAGE == 1 ? 5 : 6] = make_double2(sum[0], sum[1]);
    if constexpr (STAGE == 2) sc[7] = make_double2(sum[2], 0.0);
    bicg_stage(STAGE, sc);
}

// p = r + beta (p - omega v); with b_out, its complex64 copy (the next cycle's right-hand side)
__global__ void k_bicg_p(size_t n, const double2 *__restrict__ r, const double2 *__restrict__ v,
                         const double2 *__restrict__ sc, double2 *__restrict__ p, float2 *__restrict__ b_out) {
    pdl_enter();
    const double2 beta = sc[4], om = sc[3];
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const double2 t = cfma(beta, csub(p[q], cmul(om, v[q])), r[q]);
        p[q] = t;
        if (b_out) b_out[q] = to_c(t, 0.f);
    }
}

// s = r - alpha v and ||s||; host[0] = ||s||, host[1] = the breakdown flag (pinned)
__global__ void __launch_bounds__(NT) k_bicg_s(size_t n, const double2 *__restrict__ r, const double2 *__restrict__ v,
                                               double2 *sc, double2 *__restrict__ so, float2 *__restrict__ b_out,
                                               double *partials, unsigned *ticket, double *host) {
    pdl_enter();
    __shared__ double sum[1];
    const double2 na = sc[8];
    double acc[1] = {0.0};
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const double2 t = cfma(na, v[q], r[q]);
        so[q] = t;
        if (b_out) b_out[q] = to_c(t, 0.f);
        acc[0] = fma(t.x, t.x, fma(t.y, t.y, acc[0]));
    }
    if (!grid_sums<1>(acc, partials, ticket, sum) || threadIdx.x != 0) return;
    host[0] = sqrt(sum[0]);
    host[1] = sc[11].x;
}

// x += alpha y + omega z; r = s - omega t; ||r||, <rh, r> -> the next iteration's rho and beta;
// host[0] = ||r||, host[1] = the breakdown flag before that step (pinned)
template <typename CY>
__global__ void __launch_bounds__(NT) k_bicg_xr(size_t n, const CY *__restrict__ y, const CY *__restrict__ z,
                                                const double2 *__restrict__ s, const double2 *__restrict__ t,
                                                const double2 *__restrict__ rh, double2 *sc, double2 *__restrict__ x,
                                                double2 *__restrict__ r, double *partials, unsigned *ticket, double *host) {
    pdl_enter();
    __shared__ double sum[4];
    const double2 al = sc[2], om = sc[3], no = sc[9];
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        x[q] = cfma(om, to_c(z[q], 0.0), cfma(al, to_c(y[q], 0.0), x[q]));
        const double2 rq = cfma(no, t[q], s[q]), h = rh[q];
        r[q] = rq;
        v[0] = fma(h.x, rq.x, fma(h.y, rq.y, v[0]));
        v[1] = fma(h.x, rq.y, fma(-h.y, rq.x, v[1]));
        v[2] = fma(rq.x, rq.x, fma(rq.y, rq.y, v[2]));
    }
    if (!grid_sums<4>(v, partials, ticket, sum) || threadIdx.x != 0) return;
    host[0] = sqrt(sum[2]);
    host[1] = sc[11].x;
    sc[0] = make_double2(sum[0], sum[1]);
    bicg_stage(0, sc);
}

template <typename CY>
__global__ void k_axpy_mixed(size_t n, const double2 *__restrict__ a, const CY *__restrict__ x, double2 *__restrict__ y) {
    pdl_enter();
    const double2 av = a[0];
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT)
        y[q] = cfma(av, to_c(x[q], 0.0), y[q]);
}

// y = W x or W^{-1} x, W_p = prod_axes w_axis[a][i_a] on interior nodes (boundary left).
// y = w x (inverse: x / w) on interior nodes, w the product of the axes' dual volumes;
// conj_x: x is conjugated first.
__global__ void k_weight(int nx, int ny, int nz, int dim, const double2 *__restrict__ wx,
                         const double2 *__restrict__ wy, const double2 *__restrict__ wz, int inverse, int conj_x,
                         const double2 *__restrict__ x, double2 *__restrict__ y) {
    pdl_enter();
    const size_t n = (size_t)nx * ny * nz;
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const int i = (int)(q % nx), j = (int)((q / nx) % ny), k = (int)(q / ((size_t)nx * ny));
        if (i < 1 || i > nx - 2 || j < 1 || j > ny - 2 || (dim == 3 && (k < 1 || k > nz - 2))) continue;
        double2 w = cmul(wx[i], wy[j]);
        if (dim == 3) w = cmul(w, wz[k]);
        if (inverse) w = cinv(w);
        double2 v = x[q];
        if (conj_x) v.y = -v.y;
        y[q] = cmul(w, v);
    }
}

// Gradients of a real loss after the adjoint solve: lambda = w y (w as in k_weight) at interior
// nodes; grad_k2 = Re(lambda u) (null: skipped) and grad_f = conj(lambda) (null: skipped),
// both 0 on the boundary.
__global__ void k_adjoint_grads(int nx, int ny, int nz, int dim, const double2 *__restrict__ wx,
                                const double2 *__restrict__ wy, const double2 *__restrict__ wz,
                                const double2 *__restrict__ y, const double2 *__restrict__ u,
                                double *__restrict__ grad_k2, double2 *__restrict__ grad_f) {
    pdl_enter();
    const size_t n = (size_t)nx * ny * nz;
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const int i = (int)(q % nx), j = (int)((q / nx) % ny), k = (int)(q / ((size_t)nx * ny));
        const bool in = !(i < 1 || i > nx - 2 || j < 1 || j > ny - 2 || (dim == 3 && (k < 1 || k > nz - 2)));
        double2 lam = make_double2(0.0, 0.0);
        if (in) {
            double2 w = cmul(wx[i], wy[j]);
            if (dim == 3) w = cmul(w, wz[k]);
            lam = cmul(w, y[q]);
        }
        if (grad_k2) {
            const double2 b = u[q];
            grad_k2[q] = in ? (lam.x * b.x - lam.y * b.y) : 0.0;
        }
        if (grad_f) grad_f[q] = make_double2(lam.x, -lam.y);
    }
}

__global__ void k_grad_k2(int nx, int ny, int nz, int dim, const double2 *__restrict__ lam,
                          const double2 *__restrict__ u, double *__restrict__ grad) {
    pdl_enter();
    const size_t n = (size_t)nx * ny * nz;
    for (size_t q = blockIdx.x * (size_t)NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const int i = (int)(q % nx), j = (int)((q / nx) % ny), k = (int)(q / ((size_t)nx * ny));
        const bool in = !(i < 1 || i > nx - 2 || j < 1 || j > ny - 2 || (dim == 3 && (k < 1 || k > nz - 2)));
        const double2 a = lam[q], b = u[q];
        grad[q] = in ? (a.x * b.x - a.y * b.y) : 0.0;
    }
}

unsigned stream_grid(size_t n) { return (unsigned)std::min<size_t>(cdiv(n, NT), (size_t)152 * 8); }

}  // namespace

int blas_nblocks(size_t n) { return (int)std::min<size_t>(cdiv(n, NT), (size_t)MAXBLK); }

// Two blocks per SM over all block rows.
int mdot_nblocks(size_t n, int nv) {
    if (nv <= 0) return blas_nblocks(n);
    return (int)std::min<size_t>(cdiv(n, NT), (size_t)std::max(1, 2 * 152 / ((nv + 7) / 8)));
}

cudaError_t launch_mdot_norm(size_t n, const double2 *V, size_t ldv, int nv, const double2 *w, double2 *partials,
                             const int *gate, cudaStream_t s) {
    if (nv < 0 || nv > 64 || (nv == 0 && gate)) return cudaErrorInvalidValue;
    const int G = mdot_nblocks(n, nv);
    if (nv == 0) {  // the norm alone
        launch_pdl(k_norm2, G, NT, 0, s, n, w, partials);
        return cudaGetLastError();
    }
    const int chunks = (nv + 7) / 8, most = (nv + chunks - 1) / chunks;
    const dim3 g(G, chunks);
    if (most <= 2) launch_pdl(k_mdot_norm<2>, g, NT, 0, s, n, V, ldv, nv, w, partials, gate);
    else if (most <= 4) launch_pdl(k_mdot_norm<4>, g, NT, 0, s, n, V, ldv, nv, w, partials, gate);
    else launch_pdl(k_mdot_norm<8>, g, NT, 0, s, n, V, ldv, nv, w, partials, gate);
    return cudaGetLastError();
}

cudaError_t launch_update_norm(size_t n, const double2 *V, size_t ldv, int nv, const double2 *h, double2 *w,
                               double2 *partials, const int *gate, const double2 *wnorm, cudaStream_t s) {
    if (nv < 0 || nv > 64) return cudaErrorInvalidValue;
    launch_pdl(k_update_norm, blas_nblocks(n), NT, 0, s, n, V, ldv, nv, h, w, partials, gate, wnorm);
    return cudaGetLastError();
}

cudaError_t launch_reduce(const double2 *partials, int nblk, int nv, double2 *out, int mode, const int *gate,
                          cudaStream_t s, double *host_out, double2 *out2) {
    launch_pdl(k_reduce, nv, NT, 0, s, partials, nblk, out, mode, gate, host_out, out2);
    return cudaGetLastError();
}

cudaError_t launch_reduce_decide(const double2 *partials, int nblk, double2 *hnorm, int *flag, int *count, double eta,
                                 double2 *norm, cudaStream_t s) {
    launch_pdl(k_reduce_decide, 1, NT, 0, s, partials, nblk, hnorm, flag, count, eta, norm);
    return cudaGetLastError();
}

cudaError_t launch_scale_inv(size_t n, const double2 *x, const double2 *scale, double2 *y, float2 *b_out,
                             cudaStream_t s) {
    launch_pdl(k_scale_inv, stream_grid(n), NT, 0, s, n, x, scale, y, b_out);
    return cudaGetLastError();
}

template <typename CZ>
cudaError_t launch_combine(size_t n, const CZ *Z, size_t ldz, int nz, const double2 *y, const double2 *alpha,
                           double2 *x, cudaStream_t s) {
    if (nz > 64) return cudaErrorInvalidValue;
    if constexpr (sizeof(CZ) == sizeof(float2)) {
        launch_pdl(k_combine_df, stream_grid(n), NT, 0, s, n, (const float2 *)Z, ldz, nz, y, alpha, x);
    } else {
        if (alpha) return cudaErrorInvalidValue;
        launch_pdl(k_combine<CZ>, stream_grid(n), NT, 0, s, n, Z, ldz, nz, y, x);
    }
    return cudaGetLastError();
}
template cudaError_t launch_combine<float2>(size_t, const float2 *, size_t, int, const double2 *, const double2 *,
                                            double2 *, cudaStream_t);
template cudaError_t launch_combine<double2>(size_t, const double2 *, size_t, int, const double2 *, const double2 *,
                                             double2 *, cudaStream_t);

cudaError_t launch_givens(double2 *H, int ldh, int j, double *cs, double2 *sn, double2 *g, const double2 *fnorm,
                          double *est, double *est_host, const double *tol, int *stop, cudaStream_t s) {
    if (stop && !tol) return cudaErrorInvalidValue;
    k_givens<<<1, 32, 0, s>>>(H, ldh, j, cs, sn, g, fnorm, est, est_host, tol, stop);
    return cudaGetLastError();
}

cudaError_t launch_cycle_start(double2 *g, int len, const double2 *beta, int *stop, double *tol_dev, double tol,
                               cudaStream_t s) {
    if (len < 1) return cudaErrorInvalidValue;
    launch_pdl(k_cycle_start, 1, NT, 0, s, g, len, beta, stop, tol_dev, tol);
    return cudaGetLastError();
}

cudaError_t launch_reduce_dcgs2(const double2 *partials, int nblk, double2 *hv, unsigned *ticket, int j,
                                const double2 *alpha2, double2 *H, int ldh, double2 *coef, int has_w,
                                cudaStream_t s) {
    if (j < 0 || j > 64 || has_w < 0 || has_w > 2) return cudaErrorInvalidValue;
    launch_pdl(k_reduce_dcgs2, 2 * (j + 1), NT, 0, s, partials, nblk, hv, ticket, j, alpha2, H, ldh, coef, has_w);
    return cudaGetLastError();
}

cudaError_t launch_reduce_dcgs2_batch(int count, const BVec *tab, const unsigned *first, int groups, int j,
                                      int has_w, cudaStream_t s) {
    if (count < 1 || count > 65535 || j < 0 || j > 64 || groups < 1 || has_w < 0 || has_w > 2)
        return cudaErrorInvalidValue;
    launch_pdl(k_reduce_dcgs2_b, dim3(2 * (j + 1), 1, count), NT, 0, s, tab, first, groups, j, has_w);
    return cudaGetLastError();
}

cudaError_t launch_givens_batch(int count, const BVec *tab, int j, double *est_out, const double *tol, cudaStream_t s) {
    if (count < 1 || count > 65535 || j < 0 || j > 63) return cudaErrorInvalidValue;
    launch_pdl(k_givens_b, dim3(1, 1, count), 32, 0, s, tab, j, est_out, tol);
    return cudaGetLastError();
}

cudaError_t launch_backsolve(const double2 *H, int ldh, int k, const double2 *g, double2 *y, cudaStream_t s) {
    if (k < 1 || k > 64 || ldh < k) return cudaErrorInvalidValue;
    static bool attr = false;
    if (!attr) {
        const cudaError_t e = cudaFuncSetAttribute(k_backsolve, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)((64 * 64 + 64) * sizeof(double2)));
        if (e != cudaSuccess) return e;
        attr = true;
    }
    launch_pdl(k_backsolve, 1, NT, (size_t)(k * k + k) * sizeof(double2), s, H, ldh, k, g, y);
    return cudaGetLastError();
}

cudaError_t launch_bicg_scalars(int stage, double2 *sc, cudaStream_t s) {
    launch_pdl(k_bicg_scalars, 1, 32, 0, s, stage, sc);
    return cudaGetLastError();
}

cudaError_t launch_bicg_p(size_t n, const double2 *r, const double2 *v, const double2 *sc, double2 *p, float2 *b_out,
                          cudaStream_t s) {
    launch_pdl(k_bicg_p, stream_grid(n), NT, 0, s, n, r, v, sc, p, b_out);
    return cudaGetLastError();
}

cudaError_t launch_bicg_dots(int stage, size_t n, const double2 *a, const double2 *b, double2 *sc, double2 *partials,
                             unsigned *ticket, cudaStream_t s) {
    double *pd = (double *)partials;
    if (stage == 1) launch_pdl(k_bicg_dots<1>, blas_nblocks(n), NT, 0, s, n, a, b, sc, pd, ticket);
    else launch_pdl(k_bicg_dots<2>, blas_nblocks(n), NT, 0, s, n, a, b, sc, pd, ticket);
    return cudaGetLastError();
}

cudaError_t launch_bicg_s(size_t n, const double2 *r, const double2 *v, double2 *sc, double2 *so, float2 *b_out,
                          double2 *partials, unsigned *ticket, double *host, cudaStream_t s) {
    launch_pdl(k_bicg_s, blas_nblocks(n), NT, 0, s, n, r, v, sc, so, b_out, (double *)partials, ticket, host);
    return cudaGetLastError();
}

template <typename CY>
cudaError_t launch_bicg_xr(size_t n, const CY *y, const CY *z, const double2 *so, const double2 *t, const double2 *rh,
                           double2 *sc, double2 *x, double2 *r, double2 *partials, unsigned *ticket, double *host,
                           cudaStream_t s) {
    launch_pdl(k_bicg_xr<CY>, blas_nblocks(n), NT, 0, s, n, y, z, so, t, rh, sc, x, r, (double *)partials, ticket, host);
    return cudaGetLastError();
}
template cudaError_t launch_bicg_xr<float2>(size_t, const float2 *, const float2 *, const double2 *, const double2 *,
                                            const double2 *, double2 *, double2 *, double2 *, double2 *, unsigned *,
                                            double *, cudaStream_t);
template cudaError_t launch_bicg_xr<double2>(size_t, const double2 *, const double2 *, const double2 *, const double2 *,
                                             const double2 *, double2 *, double2 *, double2 *, double2 *, unsigned *,
                                             double *, cudaStream_t);

template <typename CY>
cudaError_t launch_axpy_mixed(size_t n, const double2 *a, const CY *x, double2 *y, cudaStream_t s) {
    launch_pdl(k_axpy_mixed<CY>, stream_grid(n), NT, 0, s, n, a, x, y);
    return cudaGetLastError();
}
template cudaError_t launch_axpy_mixed<float2>(size_t, const double2 *, const float2 *, double2 *, cudaStream_t);
template cudaError_t launch_axpy_mixed<double2>(size_t, const double2 *, const double2 *, double2 *, cudaStream_t);

cudaError_t launch_weight(size_t n, const int nodes[3], int dim, const double2 *w_axis[3], int inverse,
                          const double2 *x, double2 *y, cudaStream_t s, int conj_x) {
    launch_pdl(k_weight, stream_grid(n), NT, 0, s, nodes[0], nodes[1], dim == 3 ? nodes[2] : 1, dim, w_axis[0], w_axis[1],
                                           w_axis[2], inverse, conj_x, x, y);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_grads(size_t n, const int nodes[3], int dim, const double2 *w_axis[3], const double2 *y,
                                 const double2 *u, double *grad_k2, double2 *grad_f, cudaStream_t s) {
    launch_pdl(k_adjoint_grads, stream_grid(n), NT, 0, s, nodes[0], nodes[1], dim == 3 ? nodes[2] : 1, dim, w_axis[0],
               w_axis[1], w_axis[2], y, u, grad_k2, grad_f);
    return cudaGetLastError();
}

cudaError_t launch_grad_k2(size_t n, const int nodes[3], int dim, const double2 *lam, const double2 *u,
                           double *grad, cudaStream_t s) {
    launch_pdl(k_grad_k2, stream_grid(n), NT, 0, s, nodes[0], nodes[1], dim == 3 ? nodes[2] : 1, dim, lam, u, grad);
    return cudaGetLastError();
}
