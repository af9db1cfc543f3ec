// FP64-accurate Helmholtz coupling from stored double-float matrices (Sec. 4.2).
//
// Coupling matrices are complex symmetric, K_{tau sigma} = K_{sigma tau}^T (the
// kernel depends on |x - y| only and the product of the surface measures
// commutes, so both are evaluated identically); only one of the
// two is stored (half_owner), [n_up][kpt][4 q2] float4 (re_hi, re_lo, im_hi, im_lo),
// entry (a, b = s + 4 kk) at [kk][4 a + s].  The CTA of row sigma streams its blocks
// once through a ring of shared-memory stages and uses each twice, for up to
// RB right-hand sides: rows give y^_sigma = sum K x^_tau, columns the block's share
// K^T x^_sigma of y^_tau, stored per block and added by helm_column_gather_kernel in
// a fixed order (no atomics: repeated applications are bitwise identical).
//
// Bound: the FP32 pipe (96 operations per stored entry and right-hand side: two
// complex multiply-adds of exact products and TwoSum sums, 0.55 ms of FP32 issue
// at level 4, q = 6 with one right-hand side, against 0.53 ms for the 3.6 GB at
// 6.8 TB/s).  Level 4, q = 6, kappa = 4, one right-hand side: 1.01 ms with the column
// shares, against 1.32 ms when both mirrored blocks were stored and read; level 3, 8
// right-hand sides: 1.81 ms against 2.00 ms (matrix read once per right-hand
// side).  The sums over blocks are as exact as the FP64 ones of that form; as plain
// double-floats they take 1 to 5% less time (1.00 and 1.71 ms) and make the error of an
// application 1.4 times as large (6.4e-16 against 4.5e-16 at level 4, q = 8).  Two
// right-hand sides per CTA: with four the unrolled code misses the instruction cache
// (2.4 ms at level 3).  Packed two-float instructions gave nothing (1.00 ms): the pipe is
// the limit (64 to 66% active at level 3), not issue.
#include <algorithm>

#include "ibem_internal.cuh"

namespace ibem {

namespace {

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

constexpr int HS_RC = 8;     // right-hand sides per pass at least
constexpr int HS_RB = 2;     // right-hand sides per CTA at most
constexpr int64_t HS_SHARES = (int64_t)256 << 20;   // bytes of column shares beyond which a pass takes no more than HS_RC

// Most right-hand sides per pass.  A pass holds the column shares of its right-hand
// sides (q^2 float4 per stored block and right-hand side), so on large trees eight;
// on small ones, which eight do not fill (level 2, q = 4, 64 right-hand sides: 8
// passes took 435 us, one 256), all that fit.
int hs_most(const ibem_handle* h) {
    const int64_t per = (h->n_up > 0 ? h->n_up : 1) * (int64_t)h->P.q2 * (int64_t)sizeof(float4);
    return (int)std::min<int64_t>(1 << 20, std::max<int64_t>(HS_RC, HS_SHARES / per / 2 * 2));
}
// passes of equal size up to a pair
int hs_pass(const ibem_handle* h, int R) {
    const int n = (R + hs_most(h) - 1) / hs_most(h);
    return std::min(R, ((R + n - 1) / n + 1) / 2 * 2);
}

__device__ __forceinline__ void hs_add(float& hi, float& lo, float h2, float l2) {
    const float s = hi + h2;
    const float z = s - hi;
    const float err = (hi - (s - z)) + (h2 - z);
    hi = s;
    lo += l2 + err;
}
// acc += a * b: exact leading product, its error and the cross terms, TwoSum
__device__ __forceinline__ void hs_mac(float ah, float al, float bh, float bl, float& hi, float& lo) {
    const float p = ah * bh;
    float e = fmaf(ah, bh, -p);
    e = fmaf(ah, bl, e);
    e = fmaf(al, bh, e);
    hs_add(hi, lo, p, e);
}
// Sum of double-floats over many blocks, in three parts: exact but for the rounding of the
// third one (2^-72), so no less accurate than an FP64 sum, which would take conversions
// and additions on the FP64 pipe (level 4, q = 6, one right-hand side: 1.33 ms).
struct hs_sum {
    float h = 0.0f, m = 0.0f, l = 0.0f;
};
__device__ __forceinline__ float hs_two_sum(float a, float b, float& e) {
    const float s = a + b, z = s - a;
    e = (a - (s - z)) + (b - z);
    return s;
}
__device__ __forceinline__ void hs_acc(hs_sum& a, float h, float l) {
    float e, f, g;
    a.h = hs_two_sum(a.h, h, e);
    const float t = hs_two_sum(a.m, l, f);
    a.m = hs_two_sum(t, e, g);
    a.l += f + g;
}
__device__ __forceinline__ double hs_value(const hs_sum& a) { return (double)a.h + ((double)a.m + (double)a.l); }
// (re, im) += k x for complex double-floats
__device__ __forceinline__ void hs_cmac(const float4 k, const float4 x, float (&s)[4]) {
    hs_mac(k.x, k.y, x.x, x.y, s[0], s[1]);
    hs_mac(-k.z, -k.w, x.z, x.w, s[0], s[1]);
    hs_mac(k.x, k.y, x.z, x.w, s[2], s[3]);
    hs_mac(k.z, k.w, x.x, x.y, s[2], s[3]);
}

__device__ inline unsigned hs_smem(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ inline void hs_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(hs_smem(bar)), "r"(bytes) : "memory");
}
__device__ inline void hs_bulk(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     hs_smem(dst)),
                 "l"(src), "r"(bytes), "r"(hs_smem(bar))
                 : "memory");
}
__device__ inline bool hs_wait(uint64_t* bar, unsigned parity, long long limit) {
    for (long long it = 0; it < limit; ++it) {
        unsigned ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(hs_smem(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// moments of the split layout [2R][C][q2], right-hand sides r0 .. r0 + rc - 1 ->
// double-float complex [groups][C][RB][q2p] (q2p even: 32-byte rows), zero-padded
__global__ void helm_split_kernel(int r0, int rc, int RB, int ng, int64_t C, int q2, int q2p,
                                  const double* __restrict__ xh, float4* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)ng * C * RB * q2p) return;
    const int a = (int)(i % q2p);
    int64_t rem = i / q2p;
    const int rr = (int)(rem % RB);
    rem /= RB;
    const int64_t c = rem % C;
    const int r = (int)(rem / C) * RB + rr;
    double vr = 0.0, vi = 0.0;
    if (a < q2 && r < rc) {
        vr = xh[((int64_t)(2 * (r0 + r)) * C + c) * q2 + a];
        vi = xh[((int64_t)(2 * (r0 + r) + 1) * C + c) * q2 + a];
    }
    const float rh = (float)vr, ih = (float)vi;
    out[i] = make_float4(rh, (float)(vr - (double)rh), ih, (float)(vi - (double)ih));
}

// Thread t = 4 a + s: row pass, row a and columns s + 4 kk; column pass, column
// t / 4 and rows t % 4 + 4 j.  A thread's sums over a block are double-float, those over the
// blocks of a row, the threads of a column and the shares of a column
// (helm_column_gather_kernel) in three parts.  EXACT: q2 == 4 KPT (even q).
// Launch bounds: the CTAs that the stages leave room for (left to itself the compiler
// takes 32 registers at q = 6 with one right-hand side, and 125 us more at level 4).
constexpr int hs_threads(int kpt) { return (16 * kpt + 31) / 32 * 32; }
constexpr int hs_ctas(int kpt, int nst) {
    return IBEM_MAX_SMEM_BYTES / (256 * kpt * kpt * nst) < 16 ? IBEM_MAX_SMEM_BYTES / (256 * kpt * kpt * nst) : 16;
}
template <int KPT, int NST, int RB, bool EXACT>
__global__ void __launch_bounds__(hs_threads(KPT), hs_ctas(KPT, NST)) helm_coupling_sym_kernel(
    const int32_t* __restrict__ rows, const int64_t* __restrict__ uptr, const int32_t* __restrict__ usrc,
    const float4* __restrict__ K, int q2_rt, int q2p, int maxrow, int64_t C, const float4* __restrict__ xh, int r0, int rc,
    double* __restrict__ yh, float4* __restrict__ colpart, int64_t n_up, long long wait_limit,
    int* __restrict__ status) {
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    int32_t* srcs = reinterpret_cast<int32_t*>(smem + 128);
    const int q2 = EXACT ? 4 * KPT : q2_rt;
    const int stride = 4 * q2;
    const int belems = KPT * stride;
    const int selems = belems + RB * q2p;
    float4* XS = reinterpret_cast<float4*>(smem + 128 + (((size_t)maxrow * 4 + 15) / 16) * 16);   // [RB][q2p]
    float4* stage = XS + RB * q2p;
    const unsigned kbytes = (unsigned)belems * 16u, xbytes = (unsigned)(RB * q2p) * 16u;
    const int sigma = rows[blockIdx.x];
    const int t = threadIdx.x, s = t & 3, a = t >> 2;
    const bool active = t < stride;
    const int64_t b0 = uptr[sigma];
    const int n = (int)(uptr[sigma + 1] - b0);
    const float4* xg = xh + (int64_t)blockIdx.y * C * RB * q2p;
    const int rg = blockIdx.y * RB;                            // first right-hand side of the group within the pass
    for (int j = t; j < n; j += blockDim.x) srcs[j] = usrc[b0 + j];
    for (int j = t; j < RB * q2p; j += blockDim.x) XS[j] = xg[(int64_t)sigma * RB * q2p + j];
    if (t == 0) {
        for (int i = 0; i < NST; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(hs_smem(&full[i])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    auto fetch = [&](int i) {
        float4* dst = stage + (size_t)(i % NST) * selems;
        uint64_t* bar = &full[i % NST];
        hs_expect_tx(bar, kbytes + xbytes);
        hs_bulk(dst, K + (b0 + i) * (int64_t)belems, kbytes, bar);
        hs_bulk(dst + belems, xg + (int64_t)srcs[i] * RB * q2p, xbytes, bar);
    };
    if (t == 0)
        for (int i = 0; i < NST && i < n; ++i) fetch(i);
    hs_sum acc[RB][2];
    int i = 0;
    bool failed = false;
    for (; i < n; ++i) {
        const bool ok = hs_wait(&full[i % NST], (unsigned)((i / NST) & 1), wait_limit);
        float col[RB][4] = {};
        if (ok && active) {
            const float4* Kb = stage + (size_t)(i % NST) * selems;
            const float4* xt = Kb + belems;
            float row[RB][4] = {};
#pragma unroll(KPT <= 9 ? KPT : 1)
            for (int kk = 0; kk < KPT; ++kk) {
                const int b = s + 4 * kk;
                if (EXACT || b < q2) {
                    const float4 kv = Kb[kk * stride + t];
#pragma unroll
                    for (int r = 0; r < RB; ++r) hs_cmac(kv, xt[r * q2p + b], row[r]);
                }
            }
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                hs_acc(acc[r][0], row[r][0], row[r][1]);
                hs_acc(acc[r][1], row[r][2], row[r][3]);
            }
            const float4* Kc = Kb + (a >> 2) * stride + (a & 3) + 4 * s;
#pragma unroll(KPT <= 9 ? KPT : 1)
            for (int j = 0; j < KPT; ++j) {
                if (EXACT || s + 4 * j < q2) {
                    const float4 kv = Kc[16 * j];
#pragma unroll
                    for (int r = 0; r < RB; ++r) hs_cmac(kv, XS[r * q2p + s + 4 * j], col[r]);
                }
            }
        }
        // columns: combine the 4 lanes that share a column (all lanes take part); lanes
        // s = 0, 1 end with the real part, s = 2, 3 with the imaginary part
        float2 share[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const bool im = s & 2;
            const float oh = __shfl_xor_sync(0xffffffffu, im ? col[r][0] : col[r][2], 2);
            const float ol = __shfl_xor_sync(0xffffffffu, im ? col[r][1] : col[r][3], 2);
            hs_sum v;
            v.h = im ? col[r][2] : col[r][0];
            v.m = im ? col[r][3] : col[r][1];
            hs_acc(v, oh, ol);
            const float vh = __shfl_xor_sync(0xffffffffu, v.h, 1), vm = __shfl_xor_sync(0xffffffffu, v.m, 1);
            v.l += __shfl_xor_sync(0xffffffffu, v.l, 1);
            hs_acc(v, vh, vm);
            share[r].x = hs_two_sum(v.h, v.m, share[r].y);
            share[r].y += v.l;
        }
        if (__syncthreads_or(!ok)) {
            failed = true;
            break;
        }
        if (t == 0 && i + NST < n) fetch(i + NST);
        if (active && (s & 1) == 0)
#pragma unroll
            for (int r = 0; r < RB; ++r)
                if (rg + r < rc)
                    reinterpret_cast<float2*>(colpart)[2 * (((int64_t)(rg + r) * n_up + b0 + i) * q2 + a) + (s >> 1)] =
                        share[r];
    }
    if (failed) {
        if (t == 0) {
            atomicOr(status, 1);
            // every issued copy must land before the CTA's shared memory is released
            for (int j = i; j < n && j < i + NST; ++j) hs_wait(&full[j % NST], (unsigned)((j / NST) & 1), 1LL << 24);
        }
        __syncthreads();
        return;
    }
#pragma unroll
    for (int r = 0; r < RB; ++r)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            double v = hs_value(acc[r][k]);
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            if (active && s == 0 && rg + r < rc) yh[((int64_t)(2 * (r0 + rg + r) + k) * C + sigma) * q2 + a] = v;
        }
}

// y^_tau += sum over the stored blocks (sigma, tau) of their column shares.
// One CTA per (tau, right-hand side): G = blockDim / q2 slices of the transposed
// list, combined in order; a list is read by G times as many threads as with one
// thread per entry of y^_tau.
__global__ void helm_column_gather_kernel(int r0, int64_t C, int q2, int G, const int64_t* __restrict__ tptr,
                                          const int32_t* __restrict__ tblk, const float4* __restrict__ colpart,
                                          int64_t n_up, double* __restrict__ yh) {
    extern __shared__ double red[];   // [G][q2][2]
    const int64_t tau = blockIdx.x, k0 = tptr[tau], k1 = tptr[tau + 1];
    if (k0 == k1) return;
    const int r = blockIdx.y, t = threadIdx.x, g = t / q2, b = t - g * q2;
    if (g < G) {
        const float4* part = colpart + (int64_t)r * n_up * q2 + b;
        hs_sum sr, si;
#pragma unroll 4
        for (int64_t k = k0 + g; k < k1; k += G) {
            const float4 v = part[(int64_t)tblk[k] * q2];
            hs_acc(sr, v.x, v.y);
            hs_acc(si, v.z, v.w);
        }
        red[2 * t] = hs_value(sr);
        red[2 * t + 1] = hs_value(si);
    }
    __syncthreads();
    if (t < 2 * q2) {
        const int bb = t >> 1, part = t & 1;
        double v = 0.0;
        for (int k = 0; k < G; ++k) v += red[2 * (k * q2 + bb) + part];
        yh[((int64_t)(2 * (r0 + r) + part) * C + tau) * q2 + bb] += v;
    }
}

template <int KPT, int NST, int RB>
cudaError_t launch_sym(ibem_handle* h, int r0, int rc, int ng, const float4* xh, float4* col) {
    constexpr bool EXACT = KPT == 1 || KPT == 4 || KPT == 9 || KPT == 16 || KPT == 25;
    const Plan& P = h->P;
    const int q2 = P.q2, q2p = (q2 + 1) & ~1;
    const int threads = ((4 * q2 + 31) / 32) * 32;
    const size_t sbytes = ((size_t)KPT * 4 * q2 + (size_t)RB * q2p) * sizeof(float4);
    const size_t sm = 128 + (((size_t)h->max_up_row * 4 + 15) / 16) * 16 + (size_t)RB * q2p * sizeof(float4) +
                      (size_t)NST * sbytes;
    auto kern = helm_coupling_sym_kernel<KPT, NST, RB, EXACT>;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm))) return e;
    kern<<<dim3((unsigned)h->up_rows.size(), (unsigned)ng), threads, sm, h->stream>>>(
        h->d_up_rows, h->d_up_ptr, h->d_up_src, h->d_Kc, q2, q2p, h->max_up_row, P.C, xh, r0, rc, h->d_yh, col,
        h->n_up, h->wait_limit, h->d_status);
    h->launches++;
    return cudaGetLastError();
}

template <int KPT, int NST>
cudaError_t launch_sym_rb(ibem_handle* h, int r0, int rc, int RB, const float4* xh, float4* col) {
    return RB == 1 ? launch_sym<KPT, NST, 1>(h, r0, rc, rc, xh, col)
                   : launch_sym<KPT, NST, 2>(h, r0, rc, (rc + 1) / 2, xh, col);
}

// rc right-hand sides from r0 in groups of RB (the last one padded): moments to xh, row
// sums, column shares to col
cudaError_t launch_groups(ibem_handle* h, int r0, int rc, int RB, float4* xh, float4* col) {
    const Plan& P = h->P;
    const int q2p = (P.q2 + 1) & ~1, ng = (rc + RB - 1) / RB, T = 256;
    helm_split_kernel<<<nblk((int64_t)ng * P.C * RB * q2p, T), T, 0, h->stream>>>(r0, rc, RB, ng, P.C, P.q2, q2p,
                                                                                  h->d_xh, xh);
    h->launches++;
    switch (h->kpt) {
        case 1: return launch_sym_rb<1, 8>(h, r0, rc, RB, xh, col);
        case 3: return launch_sym_rb<3, 6>(h, r0, rc, RB, xh, col);
        case 4: return launch_sym_rb<4, 4>(h, r0, rc, RB, xh, col);
        case 7: return launch_sym_rb<7, 3>(h, r0, rc, RB, xh, col);
        case 9: return launch_sym_rb<9, 2>(h, r0, rc, RB, xh, col);
        case 13: return launch_sym_rb<13, 2>(h, r0, rc, RB, xh, col);
        case 16: return launch_sym_rb<16, 2>(h, r0, rc, RB, xh, col);
        case 21: return launch_sym_rb<21, 1>(h, r0, rc, RB, xh, col);
        case 25: return launch_sym_rb<25, 1>(h, r0, rc, RB, xh, col);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Work space of the stored coupling for R complex right-hand sides: moments and
// column shares of one pass.  Sized with the other work vectors (ensure_workspace), not
// in the application, which a program may record into a graph.
cudaError_t ensure_helm_df(ibem_handle* h, int R) {
    const int rc = std::min(R, hs_most(h));
    if (rc <= h->hdf_rhs) return cudaSuccess;
    const Plan& P = h->P;
    cudaFree(h->d_xh4);
    cudaFree(h->d_hcol);
    h->d_xh4 = nullptr;
    h->d_hcol = nullptr;
    h->hdf_rhs = 0;
    cudaError_t e;
    if ((e = cudaMalloc(&h->d_xh4, (size_t)(rc + 1) * P.C * ((P.q2 + 1) & ~1) * sizeof(float4)))) return e;
    if ((e = cudaMalloc(&h->d_hcol, (size_t)rc * (h->n_up > 0 ? h->n_up : 1) * P.q2 * sizeof(float4)))) return e;
    h->hdf_rhs = rc;
    return cudaSuccess;
}

cudaError_t launch_helm_coupling_df(ibem_handle* h, int R) {
    const Plan& P = h->P;
    cudaStream_t st = h->stream;
    cudaError_t e;
    const int q2 = P.q2, q2p = (q2 + 1) & ~1, pass = hs_pass(h, R);
    if (h->up_rows.empty()) return cudaSuccess;
    for (int r0 = 0; r0 < R; r0 += pass) {
        const int rc = R - r0 < pass ? R - r0 : pass;
        // pairs, and an odd one by itself (as half of a pair it takes twice the time: level 4, q = 6,
        // three right-hand sides 4.27 ms, now 3.48), unless the launch is too small to fill
        // the chip and one more costs more
        const bool tiny = (int64_t)h->up_rows.size() * ((rc + 1) / 2) <= 2 * 152;
        const int two = tiny && rc > 1 ? rc : rc / HS_RB * HS_RB;
        if (two > 0 && (e = launch_groups(h, r0, two, HS_RB, h->d_xh4, h->d_hcol))) return e;
        if (two < rc && (e = launch_groups(h, r0 + two, 1, 1, h->d_xh4 + (size_t)two * P.C * q2p,
                                           h->d_hcol + (size_t)two * h->n_up * q2)))
            return e;
        const int G = 256 / q2 > 0 ? 256 / q2 : 1;
        const int threads = ((G * q2 > 2 * q2 ? G * q2 : 2 * q2) + 31) / 32 * 32;
        helm_column_gather_kernel<<<dim3((unsigned)P.C, (unsigned)rc), threads, (size_t)2 * threads * sizeof(double), st>>>(
            r0, P.C, q2, G, h->d_tr_ptr, h->d_tr_blk, h->d_hcol, h->n_up, h->d_yh);
        h->launches++;
    }
    return cudaGetLastError();
}

}  // namespace ibem
