// Helmholtz (complex) parts of libibem.  Fundamental solution
// u*(x, y) = exp(i kappa |x - y|) / (4 pi |x - y|) (Eq. fundament2); the bilinear
// form has no conjugation, so every block is complex-symmetric.
//
// Layout: the public complex arrays are interleaved (re, im).  Inside an
// application they are split into 2R real right-hand sides (index 2r for the
// real part, 2r + 1 for the imaginary part), so every step whose coefficients
// are real (T^T, moments, M2M, L2L, back-projection, T) runs the real kernels
// unchanged; only the near product and the coupling mix real and imaginary
// parts.
//
// Near blocks: [n_near][nb][nb] double2 (re, im).  Coupling matrices of the
// FP64 operator: one of two mirrored blocks stored as double-float complex (re_hi,
// re_lo, im_hi, im_lo), layout [n_up][kpt][4 q2] like the Laplace case
// (kernels_helm_df.cu), or - when they would not fit in the memory budget -
// generated on the fly.
#include <algorithm>

#include "fp64_eval.cuh"
#include "ibem_internal.cuh"

namespace ibem {

static inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// exp(i kappa r) / (4 pi r) * w
__device__ inline void helm_kernel64(double kappa, double r, double w, double* re, double* im) {
    double s, c;
    sincos(kappa * r, &s, &c);
    double f = w / (4.0 * IBEM_PI * r);
    *re = f * c;
    *im = f * s;
}

// ---- near field: FP32 copy and diagonal --------------------------------------------
__global__ void helm_to_float_kernel(const double2* __restrict__ in, float2* __restrict__ out, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = make_float2((float)in[i].x, (float)in[i].y);
}

// Jacobi diagonal (complex) of T A_near T^T
__global__ void helm_near_diag_kernel(int64_t N, int p, int ne1, const int64_t* __restrict__ nptr,
                                      const int32_t* __restrict__ nsrc, const double2* __restrict__ blocks,
                                      const double* __restrict__ ext, double2* __restrict__ diag) {
    int64_t dof = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (dof >= N) return;
    int pp = p + 1, nb = pp * pp, n1 = ne1 + p;
    int patch = (int)(dof / ((int64_t)n1 * n1));
    int rem = (int)(dof % ((int64_t)n1 * n1));
    int jv = rem / n1, ju = rem % n1;
    int64_t per = (int64_t)ne1 * ne1;
    double accr = 0.0, acci = 0.0;
    for (int iy = jv - p; iy <= jv; ++iy)
        for (int ix = ju - p; ix <= ju; ++ix) {
            if (ix < 0 || iy < 0 || ix >= ne1 || iy >= ne1) continue;
            int64_t e = patch * per + morton2(ix, iy);
            const double* cu = ext + ((int64_t)ix * pp + (ju - ix)) * pp;
            const double* cv = ext + ((int64_t)iy * pp + (jv - iy)) * pp;
            for (int iy2 = jv - p; iy2 <= jv; ++iy2)
                for (int ix2 = ju - p; ix2 <= ju; ++ix2) {
                    if (ix2 < 0 || iy2 < 0 || ix2 >= ne1 || iy2 >= ne1) continue;
                    int64_t e2 = patch * per + morton2(ix2, iy2);
                    int64_t lo = nptr[e], hi = nptr[e + 1];
                    while (lo < hi) {
                        int64_t mid = (lo + hi) >> 1;
                        if (nsrc[mid] < e2) lo = mid + 1; else hi = mid;
                    }
                    if (lo >= nptr[e + 1] || nsrc[lo] != e2) continue;
                    const double2* B = blocks + lo * nb * nb;
                    const double* du = ext + ((int64_t)ix2 * pp + (ju - ix2)) * pp;
                    const double* dv = ext + ((int64_t)iy2 * pp + (jv - iy2)) * pp;
                    for (int i = 0; i < nb; ++i) {
                        double ti = cu[i % pp] * cv[i / pp];
                        double rr = 0.0, ri = 0.0;
                        for (int j = 0; j < nb; ++j) {
                            double tj = du[j % pp] * dv[j / pp];
                            rr += B[i * nb + j].x * tj;
                            ri += B[i * nb + j].y * tj;
                        }
                        accr += ti * rr;
                        acci += ti * ri;
                    }
                }
        }
    diag[dof] = make_double2(accr, acci);
}

// ---- coupling matrices (stored, double-float complex) ------------------------------
__global__ void helm_far_assemble_kernel(int64_t n_far, const int32_t* __restrict__ ftgt,
                                         const int32_t* __restrict__ fsrc, const double* __restrict__ igeo, int q2,
                                         int kpt, double kappa, const double2* __restrict__ trig,
                                         float4* __restrict__ K) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t per = (int64_t)kpt * 4 * q2;
    if (idx >= n_far * per) return;
    int64_t blk = idx / per;
    int r = (int)(idx % per);
    int kk = r / (4 * q2), t = r % (4 * q2);
    int a = t >> 2, s = t & 3, b = s + 4 * kk;
    double vr = 0.0, vi = 0.0;
    if (b < q2) {
        const double* A = igeo + 4 * ((int64_t)ftgt[blk] * q2 + a);
        const double* B = igeo + 4 * ((int64_t)fsrc[blk] * q2 + b);
        double d0 = A[0] - B[0], d1 = A[1] - B[1], d2 = A[2] - B[2];
        green64<true>(d0 * d0 + d1 * d1 + d2 * d2, kappa, A[3] * B[3] * (1.0 / (4.0 * IBEM_PI)), trig, &vr, &vi);
    }
    float rh = (float)vr, ih = (float)vi;
    K[idx] = make_float4(rh, (float)(vr - (double)rh), ih, (float)(vi - (double)ih));
}

// Complex coupling generated on the fly in FP64 (when the stored matrices would
// not fit): thread (g, a) handles target point a against blocks g, g + G, ...
__global__ void helm_coupling64_otf_kernel(const int32_t* __restrict__ rows, const int64_t* __restrict__ fptr,
                                           const int32_t* __restrict__ fsrc, const double* __restrict__ igeo, int q2,
                                           int G, int R, int64_t C, double kappa, const double* __restrict__ xh,
                                           double* __restrict__ yh) {
    extern __shared__ double red[];
    const int sigma = rows[blockIdx.x];
    const int64_t r = blockIdx.y;
    const int t = threadIdx.x, g = t / q2, a = t % q2;
    double accr = 0.0, acci = 0.0;
    if (g < G) {
        const double* X = igeo + 4 * ((int64_t)sigma * q2 + a);
        const double* xre = xh + (2 * r) * C * q2;
        const double* xim = xh + (2 * r + 1) * C * q2;
        for (int64_t blk = fptr[sigma] + g; blk < fptr[sigma + 1]; blk += G) {
            int64_t tau = fsrc[blk];
            for (int b = 0; b < q2; ++b) {
                const double* Y = igeo + 4 * (tau * q2 + b);
                double d0 = X[0] - Y[0], d1 = X[1] - Y[1], d2 = X[2] - Y[2];
                double kr, ki;
                helm_kernel64(kappa, sqrt(d0 * d0 + d1 * d1 + d2 * d2), X[3] * Y[3], &kr, &ki);
                double vr = xre[tau * q2 + b], vi = xim[tau * q2 + b];
                accr += kr * vr - ki * vi;
                acci += kr * vi + ki * vr;
            }
        }
    }
    red[2 * t] = accr;
    red[2 * t + 1] = acci;
    __syncthreads();
    if (t < q2) {
        double vr = 0.0, vi = 0.0;
        for (int k = 0; k < G; ++k) {
            vr += red[2 * (k * q2 + t)];
            vi += red[2 * (k * q2 + t) + 1];
        }
        yh[((2 * r) * C + sigma) * q2 + t] = vr;
        yh[((2 * r + 1) * C + sigma) * q2 + t] = vi;
    }
}

// Complex coupling generated on the fly in FP32: phase kappa r reduced to
// [-pi, pi] in FP32 before the hardware sine / cosine; the per-block sums are
// accumulated in double.  src32c[t][b] = (x, y, z, k_b / (4 pi)), the moments are
// read as (re, im) floats.
__global__ void helm_coupling32_kernel(const int32_t* __restrict__ rows, const int64_t* __restrict__ fptr,
                                       const int32_t* __restrict__ fsrc, const float* __restrict__ igeo32, int q2,
                                       int G, int64_t C, float kappa, const float2* __restrict__ xh32,
                                       double* __restrict__ yh_re, double* __restrict__ yh_im) {
    extern __shared__ double red[];
    const int sigma = rows[blockIdx.x];
    const int t = threadIdx.x, g = t / q2, a = t % q2;
    double accr = 0.0, acci = 0.0;
    const float inv2pi = 0.15915494309189535f, twopi = 6.283185307179586f;
    if (g < G) {
        const float* X = igeo32 + 4 * ((int64_t)sigma * q2 + a);
        const float x0 = X[0], x1 = X[1], x2 = X[2];
        for (int64_t blk = fptr[sigma] + g; blk < fptr[sigma + 1]; blk += G) {
            const int64_t tau = fsrc[blk];
            const float4* Y = reinterpret_cast<const float4*>(igeo32) + tau * q2;
            const float2* V = xh32 + tau * q2;
            float fr = 0.f, fi = 0.f;
            for (int b = 0; b < q2; ++b) {
                float4 y = Y[b];
                float2 v = V[b];
                float d0 = x0 - y.x, d1 = x1 - y.y, d2 = x2 - y.z;
                float r2 = d0 * d0 + d1 * d1 + d2 * d2;
                float rinv = rsqrtf(r2);
                float ph = kappa * (r2 * rinv);
                ph = fmaf(-twopi, rintf(ph * inv2pi), ph);
                float sn, cs;
                __sincosf(ph, &sn, &cs);
                float w = y.w * rinv;
                float kr = w * cs, ki = w * sn;
                fr = fmaf(kr, v.x, fmaf(-ki, v.y, fr));
                fi = fmaf(kr, v.y, fmaf(ki, v.x, fi));
            }
            accr += (double)fr;
            acci += (double)fi;
        }
    }
    red[2 * t] = accr;
    red[2 * t + 1] = acci;
    __syncthreads();
    if (t < q2) {
        double vr = 0.0, vi = 0.0;
        for (int k = 0; k < G; ++k) {
            vr += red[2 * (k * q2 + t)];
            vi += red[2 * (k * q2 + t) + 1];
        }
        double ka = (double)igeo32[4 * ((int64_t)sigma * q2 + t) + 3] / (4.0 * IBEM_PI);
        yh_re[(int64_t)sigma * q2 + t] = vr * ka;
        yh_im[(int64_t)sigma * q2 + t] = vi * ka;
    }
}

__global__ void helm_src32_kernel(int64_t n, const double* __restrict__ xre, const double* __restrict__ xim,
                                  float2* __restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = make_float2((float)xre[i], (float)xim[i]);
}

// ---- near product (complex) -------------------------------------------------------
// y*_e += sum B x*_s over the row; x*, y* in the split layout (2R real vectors).
template <typename T2, typename T>
__global__ void helm_near_apply_kernel(const int64_t* __restrict__ nptr, const int32_t* __restrict__ nsrc,
                                       const T2* __restrict__ blocks, int nb, int64_t E, const T* __restrict__ xs,
                                       double* __restrict__ ys) {
    extern __shared__ double red[];
    const int64_t e = blockIdx.x, r = blockIdx.y;
    const int t = threadIdx.x, nbb = nb * nb;
    double accr = 0.0, acci = 0.0;
    if (t < nbb) {
        int j = t % nb;
        const T* xre = xs + (2 * r) * E * nb;
        const T* xim = xs + (2 * r + 1) * E * nb;
        T pr = (T)0, pi = (T)0;
        for (int64_t k = nptr[e]; k < nptr[e + 1]; ++k) {
            T2 b = blocks[k * nbb + t];
            int64_t o = (int64_t)nsrc[k] * nb + j;
            T vr = xre[o], vi = xim[o];
            pr += b.x * vr - b.y * vi;
            pi += b.x * vi + b.y * vr;
        }
        accr = (double)pr;
        acci = (double)pi;
    }
    red[2 * t] = accr;
    red[2 * t + 1] = acci;
    __syncthreads();
    if (t < nb) {
        double vr = 0.0, vi = 0.0;
        for (int j = 0; j < nb; ++j) {
            vr += red[2 * (t * nb + j)];
            vi += red[2 * (t * nb + j) + 1];
        }
        ys[((2 * r) * E + e) * nb + t] += vr;
        ys[((2 * r + 1) * E + e) * nb + t] += vi;
    }
}

// FP64-accurate near product for several right-hand sides in double-float on
// the FP32 pipe: one CTA per target element; per near block of its row the
// block (FP64, split into hi + lo pairs) and the source element's lifted
// coefficients of every right-hand side are staged in shared memory, and thread
// (row i, right-hand side r) accumulates sum_j B[i][j] x*_s[j][r] with exact
// products and TwoSum accumulation (as the coupling's double-float arithmetic);
// each block is read once for all right-hand sides.  Adds to ys (split layout).
// The coefficients are split once per application (helm_split_lift_kernel): splitting
// them again for each of some 50 near blocks kept the FP64 pipe busier than the
// products the FP32 pipe.  The sums are those of S slices, every S-th block each, added in
// FP64 in order.  S depends on the degree only, so a column's bits do not depend on
// how many are applied with it: two slices where two blocks fit a CTA's registers
// (p <= 3), else one.  The slices are groups of threads that take S blocks at a time, or,
// where a slice's (row, right-hand side) pairs would exceed its threads eightfold, sets of
// sums that all threads fill in turn.  Stages are double buffered (one barrier per
// stage).  Bound: FP32 issue beside the FP64 splits of the blocks; with few columns
// latency (level 3, 8 columns: both pipes 40% busy).  p = 2, with the split: level 5, 64
// columns 4.0 ms (6.18 with the coefficients split per block); level 3, 8 columns 0.10 ms
// (0.20).
constexpr int HN_T = 256;

__device__ __forceinline__ void hn_split(double v, float& h, float& l) {
    h = (float)v;
    l = (float)(v - (double)h);
}
__device__ __forceinline__ void hn_mac(float ah, float al, float bh, float bl, float& hi, float& lo) {
    const float p = ah * bh;
    float e = fmaf(ah, bh, -p);
    e = fmaf(ah, bl, fmaf(al, bh, e));
    const float t = hi + p;
    const float z = t - hi;
    const float err = (hi - (t - z)) + (p - z);
    hi = t;
    lo += err + e;
}

// lifted coefficients of the split layout [2R][E nb] -> (re_h, re_l, im_h, im_l) [E nb][R]
__global__ void helm_split_lift_kernel(int R, int64_t n, const double* __restrict__ xs, float4* __restrict__ out) {
    __shared__ double2 tile[32][33];
    const int64_t k0 = (int64_t)blockIdx.x * 32;
    const int r0 = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int r = ty; r < 32; r += 8)
        if (r0 + r < R && k0 + tx < n)
            tile[r][tx] = make_double2(xs[(int64_t)(2 * (r0 + r)) * n + k0 + tx],
                                       xs[(int64_t)(2 * (r0 + r) + 1) * n + k0 + tx]);
    __syncthreads();
    for (int k = ty; k < 32; k += 8)
        if (r0 + tx < R && k0 + k < n) {
            const double2 v = tile[tx][k];
            float4 o;
            hn_split(v.x, o.x, o.y);
            hn_split(v.y, o.z, o.w);
            out[(k0 + k) * R + r0 + tx] = o;
        }
}

// S slices, P of them side by side (P = S or 1); MAXP pairs (row, right-hand side) per
// thread: nb R <= MAXP HN_T / P.  Dynamic shared memory 2 P (nb^2 + nb R) float4.
template <int S, int P, int MAXP>
__global__ void __launch_bounds__(HN_T) helm_near_df_kernel(const int64_t* __restrict__ nptr,
                                                            const int32_t* __restrict__ nsrc,
                                                            const double2* __restrict__ blocks, int nb, int R, int64_t E,
                                                            const float4* __restrict__ xl, double* __restrict__ ys) {
    extern __shared__ float4 hn_sm[];
    constexpr int SETS = S / P, NTH = HN_T / P;
    constexpr int MAXB = 3;          // block entries per thread: P nb^2 <= 3 HN_T
    const int64_t e = blockIdx.x;
    const int t = threadIdx.x, nbb = nb * nb, np = nb * R, sl = t / NTH, ts = t - sl * NTH;
    const int per = P * (nbb + np);  // float4 per stage: P blocks, then P coefficient sets
    float acc[SETS][MAXP][4];
#pragma unroll
    for (int q = 0; q < SETS; ++q)
#pragma unroll
        for (int k = 0; k < MAXP; ++k) acc[q][k][0] = acc[q][k][1] = acc[q][k][2] = acc[q][k][3] = 0.0f;
    const int64_t k0 = nptr[e];
    const int n = (int)(nptr[e + 1] - k0);
    double2 bn[MAXB];
    auto fetch = [&](int c) {        // blocks c .. c + P - 1: entries into registers, coefficients into the stage
        const int live = n - c < P ? n - c : P;
#pragma unroll
        for (int m = 0; m < MAXB; ++m) {
            const int q = t + HN_T * m;
            if (q < live * nbb) bn[m] = blocks[(k0 + c) * nbb + q];
        }
        float4* X = hn_sm + ((c / P) & 1) * per + P * nbb;
        for (int q = t; q < live * np; q += HN_T) {
            const int b = q / np, o = q - b * np;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             (unsigned)__cvta_generic_to_shared(X + q)),
                         "l"(xl + (int64_t)nsrc[k0 + c + b] * np + o)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (n > 0) fetch(0);
    for (int c0 = 0; c0 < n; c0 += S) {
#pragma unroll
        for (int set = 0; set < SETS; ++set) {
            const int c = c0 + set * P;
            if (c >= n) break;
            const int live = n - c < P ? n - c : P;
            float4* Bs = hn_sm + ((c / P) & 1) * per;
#pragma unroll
            for (int m = 0; m < MAXB; ++m) {
                const int q = t + HN_T * m;
                if (q < live * nbb) {
                    float4 v;
                    hn_split(bn[m].x, v.x, v.y);
                    hn_split(bn[m].y, v.z, v.w);
                    Bs[q] = v;
                }
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();         // the stage is complete; the other one is used
            if (c + P < n) fetch(c + P);
            if (sl < live) {
                const float4* B = Bs + sl * nbb;
                const float4* X = Bs + P * nbb + sl * np;
#pragma unroll
                for (int m = 0; m < MAXP; ++m) {
                    const int p = ts + NTH * m;
                    if (p < np) {
                        const int i = p / R, r = p - i * R;
                        float(&a)[4] = acc[set][m];
                        for (int j = 0; j < nb; ++j) {
                            const float4 b = B[i * nb + j], x = X[j * R + r];
                            // (Br + i Bi)(xr + i xi) = (Br xr - Bi xi) + i (Br xi + Bi xr)
                            hn_mac(b.x, b.y, x.x, x.y, a[0], a[1]);
                            hn_mac(-b.z, -b.w, x.z, x.w, a[0], a[1]);
                            hn_mac(b.x, b.y, x.z, x.w, a[2], a[3]);
                            hn_mac(b.z, b.w, x.x, x.y, a[2], a[3]);
                        }
                    }
                }
            }
        }
    }
    if (P > 1) {                     // the later slices' sums through shared memory
        __syncthreads();
#pragma unroll
        for (int m = 0; m < MAXP; ++m) {
            const int p = ts + NTH * m;
            if (sl > 0 && p < np)
                hn_sm[(sl - 1) * np + p] = make_float4(acc[0][m][0], acc[0][m][1], acc[0][m][2], acc[0][m][3]);
        }
        __syncthreads();
        if (sl > 0) return;
    }
#pragma unroll
    for (int m = 0; m < MAXP; ++m) {
        const int p = ts + NTH * m;
        if (p < np) {
            const int i = p / R, r = p - i * R;
            double vr = (double)acc[0][m][0] + (double)acc[0][m][1], vi = (double)acc[0][m][2] + (double)acc[0][m][3];
#pragma unroll
            for (int q = 1; q < S; ++q) {
                float4 v;
                if constexpr (P > 1) v = hn_sm[(q - 1) * np + p];
                else v = make_float4(acc[q % SETS][m][0], acc[q % SETS][m][1], acc[q % SETS][m][2], acc[q % SETS][m][3]);
                vr += (double)v.x + (double)v.y;
                vi += (double)v.z + (double)v.w;
            }
            ys[((int64_t)(2 * r) * E + e) * nb + i] += vr;
            ys[((int64_t)(2 * r + 1) * E + e) * nb + i] += vi;
        }
    }
}

// near product of R >= 4 columns, nb R <= 8 HN_T
static cudaError_t launch_helm_near_df(ibem_handle* h, int R) {
    const Plan& P = h->P;
    const int np = P.nb * R;
    auto go = [&](auto kern, int side) -> cudaError_t {
        const size_t sm = (size_t)2 * side * (P.nb * P.nb + np) * sizeof(float4);
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e) return e;
        kern<<<(unsigned)P.E, HN_T, sm, h->stream>>>(h->d_near_ptr, h->d_near_src,
                                                     reinterpret_cast<const double2*>(h->d_near), P.nb, R, P.E,
                                                     h->d_xsdf, h->d_ys);
        h->launches++;
        return cudaGetLastError();
    };
    if (P.nb <= 16) {
        const int per = (np + HN_T / 2 - 1) / (HN_T / 2);
        if (per <= 1) return go(helm_near_df_kernel<2, 2, 1>, 2);
        if (per <= 2) return go(helm_near_df_kernel<2, 2, 2>, 2);
        if (per <= 4) return go(helm_near_df_kernel<2, 2, 4>, 2);
        if (per <= 8) return go(helm_near_df_kernel<2, 2, 8>, 2);
        return go(helm_near_df_kernel<2, 1, 8>, 1);
    }
    const int per = (np + HN_T - 1) / HN_T;
    if (per <= 1) return go(helm_near_df_kernel<1, 1, 1>, 1);
    if (per <= 2) return go(helm_near_df_kernel<1, 1, 2>, 1);
    if (per <= 4) return go(helm_near_df_kernel<1, 1, 4>, 1);
    return go(helm_near_df_kernel<1, 1, 8>, 1);
}

// ---- layout conversion ---------------------------------------------------------------
// interleaved [R][n][2] <-> split [2R][n]
__global__ void helm_split_vec_kernel(int R, int64_t n, const double* __restrict__ in, double* __restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)R * n) return;
    int64_t r = i / n, k = i % n;
    out[(2 * r) * n + k] = in[2 * i];
    out[(2 * r + 1) * n + k] = in[2 * i + 1];
}

__global__ void helm_join_vec_kernel(int R, int64_t n, const double* __restrict__ in, double* __restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)R * n) return;
    int64_t r = i / n, k = i % n;
    out[2 * i] = in[(2 * r) * n + k];
    out[2 * i + 1] = in[(2 * r + 1) * n + k];
}

// ---- host launchers ----------------------------------------------------------------------
cudaError_t helm_launch_near_assembly(ibem_handle* h) {
    Plan& P = h->P;
    const int nb = P.nb;
    const double kappa = P.prm.kappa;
    cudaError_t e;
    double2* blocks = reinterpret_cast<double2*>(h->d_near);
    for (int cls : {CLS_REGULAR, CLS_SUBDIV}) {
        if (h->n_list[cls] > 0 && near_streamed(P.Q, nb, true, cls == CLS_SUBDIV) &&
            (e = launch_near_stream(h, cls, true, kappa, h->d_near)))
            return e;
    }
    if ((e = launch_near_graded(h, true, kappa, h->d_near))) return e;
    if ((e = launch_near_blocks(h, true, kappa, h->d_near))) return e;
    if ((e = cudaGetLastError())) return e;
    int64_t nn = P.n_near * nb * nb;
    helm_to_float_kernel<<<nblk(nn, 256), 256, 0, h->stream>>>(blocks, reinterpret_cast<float2*>(h->d_near32), nn);
    helm_near_diag_kernel<<<nblk(P.N, 128), 128, 0, h->stream>>>(P.N, P.p, P.ne1, h->d_near_ptr, h->d_near_src, blocks,
                                                                 h->d_ext, reinterpret_cast<double2*>(h->d_diag));
    return cudaGetLastError();
}

cudaError_t helm_launch_far_assembly(ibem_handle* h) {
    Plan& P = h->P;
    if (P.n_far == 0 || !h->d_Kc) return cudaSuccess;
    int64_t total = h->n_up * (int64_t)h->kpt * 4 * P.q2;   // one of two mirrored blocks
    if (total == 0) return cudaSuccess;
    helm_far_assemble_kernel<<<nblk(total, 256), 256, 0, h->stream>>>(h->n_up, h->d_up_tgt, h->d_up_src, h->d_igeo,
                                                                      P.q2, h->kpt, P.prm.kappa, h->d_trig64, h->d_Kc);
    return cudaGetLastError();
}

// y = T A T^T x for the complex operator; x, y interleaved [R][N][2].
cudaError_t helm_apply_operator(ibem_handle* h, const double* x, double* y, int nrhs, int precision,
                                double* xsplit, double* ysplit) {
    Plan& P = h->P;
    cudaStream_t st = h->stream;
    const int R = nrhs, R2 = 2 * nrhs;
    const int T = 256;
    cudaError_t e;
    {
        PhaseTimer pt(h, 0);
        helm_split_vec_kernel<<<nblk((int64_t)R * P.N, T), T, 0, st>>>(R, P.N, x, xsplit);
        lift_kernel<<<nblk(R2 * P.E * P.nb, T), T, 0, st>>>(R2, P.E, P.p, P.ne1, h->d_ext, xsplit, P.N, h->d_xs);
        h->launches += 2;
    }
    if (P.q > 0) {
        const int q2 = P.q2;
        const int64_t leaf_off = P.level_off[P.m];
        PhaseTimer pt1(h, 1);
        leaf_moment_kernel<<<nblk(R2 * P.E * q2, T), T, 0, st>>>(R2, P.E, P.pp, P.q, h->d_M, h->d_xs, leaf_off, P.C,
                                                                  h->d_xh);
        h->launches++;
        if ((e = launch_m2m(h, R2, h->d_xh))) return e;
        if ((e = cudaMemsetAsync(h->d_yh, 0, (size_t)R2 * P.C * q2 * sizeof(double), st))) return e;
        pt1.stop();
        unsigned nrows = (unsigned)h->far_rows.size();
        if (nrows > 0) {
            PhaseTimer pt2(h, 2);
            if (precision == IBEM_FP32) {
                int G = 256 / q2 > 0 ? 256 / q2 : 1;
                int threads = ((G * q2 + 31) / 32) * 32;
                for (int r = 0; r < R; ++r) {
                    helm_src32_kernel<<<nblk(P.C * q2, T), T, 0, st>>>(P.C * q2, h->d_xh + (size_t)(2 * r) * P.C * q2,
                                                                       h->d_xh + (size_t)(2 * r + 1) * P.C * q2,
                                                                       reinterpret_cast<float2*>(h->d_src32));
                    helm_coupling32_kernel<<<nrows, threads, (size_t)2 * threads * sizeof(double), st>>>(
                        h->d_far_rows, h->d_far_ptr, h->d_far_src, h->d_igeo32, q2, G, P.C, (float)P.prm.kappa,
                        reinterpret_cast<const float2*>(h->d_src32), h->d_yh + (size_t)(2 * r) * P.C * q2,
                        h->d_yh + (size_t)(2 * r + 1) * P.C * q2);
                    h->launches += 2;
                }
            } else if (h->d_Kc) {
                if ((e = launch_helm_coupling_df(h, R))) return e;
            } else if (P.prm.fp64_coupling == IBEM_COUPLING_SLICED && sliced_supported(h)) {
                if ((e = launch_coupling_sliced(h, R))) return e;
            } else if (P.prm.fp64_coupling != IBEM_COUPLING_NATIVE && gen_supported(h)) {
                if ((e = launch_coupling_gen(h, R))) return e;
            } else {
                int G = 256 / q2 > 0 ? 256 / q2 : 1;
                int threads = ((G * q2 + 31) / 32) * 32;
                helm_coupling64_otf_kernel<<<dim3(nrows, R), threads, (size_t)2 * threads * sizeof(double), st>>>(
                    h->d_far_rows, h->d_far_ptr, h->d_far_src, h->d_igeo, q2, G, R, P.C, P.prm.kappa, h->d_xh,
                    h->d_yh);
                h->launches++;
            }
        }
        PhaseTimer pt3(h, 3);
        if ((e = launch_l2l(h, R2, h->d_yh))) return e;
        leaf_back_kernel<<<nblk(R2 * P.E * P.nb, T), T, 0, st>>>(R2, P.E, P.pp, P.q, h->d_M, h->d_yh, leaf_off, P.C,
                                                                  h->d_ys);
        h->launches++;
    } else {
        if ((e = cudaMemsetAsync(h->d_ys, 0, (size_t)R2 * P.Nstar * sizeof(double), st))) return e;
    }
    int threads = ((P.nb * P.nb + 31) / 32) * 32;
    PhaseTimer pt4(h, 4);
    if (precision == IBEM_FP32) {
        d2f_kernel<<<nblk(R2 * P.Nstar, T), T, 0, st>>>(h->d_xs, h->d_xs32, R2 * P.Nstar);
        helm_near_apply_kernel<float2, float><<<dim3((unsigned)P.E, R), threads, 2 * threads * sizeof(double), st>>>(
            h->d_near_ptr, h->d_near_src, reinterpret_cast<const float2*>(h->d_near32), P.nb, P.E, h->d_xs32, h->d_ys);
        h->launches += 2;
    } else {
        if (R >= 4 && P.nb * R <= 8 * HN_T) {
            helm_split_lift_kernel<<<dim3((unsigned)((P.Nstar + 31) / 32), (unsigned)((R + 31) / 32)), 256, 0, st>>>(
                R, P.Nstar, h->d_xs, h->d_xsdf);
            if ((e = launch_helm_near_df(h, R))) return e;
        } else {
            helm_near_apply_kernel<double2, double><<<dim3((unsigned)P.E, R), threads, 2 * threads * sizeof(double),
                                                      st>>>(h->d_near_ptr, h->d_near_src,
                                                            reinterpret_cast<const double2*>(h->d_near), P.nb, P.E,
                                                            h->d_xs, h->d_ys);
        }
        h->launches++;
    }
    pt4.stop();
    PhaseTimer pt5(h, 5);
    launch_restrict(h, R2, h->d_ys, ysplit);
    helm_join_vec_kernel<<<nblk((int64_t)R * P.N, T), T, 0, st>>>(R, P.N, ysplit, y);
    h->launches++;
    return cudaGetLastError();
}

cudaError_t helm_launch_rhs(ibem_handle* h, const double* g, int nrhs, double* b, double* gsplit, double* bsplit) {
    Plan& P = h->P;
    const int T = 256, R2 = 2 * nrhs;
    int QQ = P.Q * P.Q;
    helm_split_vec_kernel<<<nblk((int64_t)nrhs * P.nq, T), T, 0, h->stream>>>(nrhs, P.nq, g, gsplit);
    rhs_super_kernel<<<nblk(R2 * P.E * P.nb, T), T, 0, h->stream>>>(R2, P.E, QQ, P.nb, h->d_qgeo, h->d_phi, gsplit,
                                                                     P.nq, h->d_ys);
    launch_restrict(h, R2, h->d_ys, bsplit);
    helm_join_vec_kernel<<<nblk((int64_t)nrhs * P.N, T), T, 0, h->stream>>>(nrhs, P.N, bsplit, b);
    return cudaGetLastError();
}

cudaError_t helm_launch_potential(ibem_handle* h, const double* w, int nrhs, const double* pts, int64_t npts,
                                  double* u, double* wsplit) {
    helm_split_vec_kernel<<<nblk((int64_t)nrhs * h->P.N, 256), 256, 0, h->stream>>>(nrhs, h->P.N, w, wsplit);
    return launch_potential_multi(h, wsplit, nrhs, pts, npts, u);
}

}  // namespace ibem
