// Direct potentials of several densities (Eq. repform):
//     u_j(x) = sum_s u*(x, y_s) mu_j(s),  mu_j(s) = W_s w_h,j(y_s) / (4 pi),
// over all Gauss points s, u* = e^{i kappa r} / r or 1 / r.
//
// A warp owns PT_P = 8 points and a slice of the sources.  It takes the sources
// four at a time: lane (point i, k) evaluates u* at (x_i, y_{s + k}) once, the
// values reach the 4 lanes of a point by shuffles, and lane (i, k) applies all four
// to the densities j = k, k + 4, ..., whose sums it keeps in registers.  So a value
// is evaluated once for up to 64 densities; atomics combine the source slices.
// Bound: the FP64 pipe, per (point, source) pair about 40 operations for the
// value and 4 (1) per complex (real) density.  Level 5, kappa = 4, 64 densities at
// 200 points: 46.2 ms against 112.5 ms with a thread per point, 16 densities
// per evaluation and sqrt, division and sincos in the value.
#include <algorithm>

#include "fp64_eval.cuh"
#include "ibem_internal.cuh"

namespace ibem {

namespace {

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

constexpr int PT_P = 8;      // points per warp
constexpr int PT_W = 4;      // warps per CTA
constexpr int PT_R = 64;     // densities per pass at most

// mu[s][j] of rc right-hand sides from the lifted coefficients xs [rc (2 rc)][E][nb]
// (complex: real and imaginary vectors in turn); consecutive threads take the Gauss
// points of one element and density, so the coefficients are broadcast
template <bool CPLX>
__global__ void densities_kernel(int64_t E, int QQ, int nb, int rc, const double* __restrict__ qgeo,
                                 const double* __restrict__ phi, const double* __restrict__ xs,
                                 double* __restrict__ mu) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= E * QQ * rc) return;
    const int q = (int)(idx % QQ), j = (int)((idx / QQ) % rc);
    const int64_t e = idx / QQ / rc, s = e * QQ + q, o = s * rc + j;
    const double* ph = phi + (int64_t)q * nb;
    const double w = qgeo[4 * s + 3] / (4.0 * IBEM_PI);
    if constexpr (CPLX) {
        const double* cr = xs + ((int64_t)(2 * j) * E + e) * nb;
        const double* ci = cr + E * nb;
        double mr = 0.0, mi = 0.0;
        for (int i = 0; i < nb; ++i) {
            mr += ph[i] * cr[i];
            mi += ph[i] * ci[i];
        }
        reinterpret_cast<double2*>(mu)[o] = make_double2(w * mr, w * mi);
    } else {
        const double* c = xs + ((int64_t)j * E + e) * nb;
        double m = 0.0;
        for (int i = 0; i < nb; ++i) m += ph[i] * c[i];
        mu[o] = w * m;
    }
}

// NJ: densities per lane (at least ceil(rc / 4))
template <bool CPLX, int NJ>
__global__ void __launch_bounds__(32 * PT_W) potential_warp_kernel(int64_t npts, const double* __restrict__ pts,
                                                                   int64_t nsrc, const double* __restrict__ qgeo,
                                                                   const double* __restrict__ mu, int rc,
                                                                   int64_t chunk, double kappa,
                                                                   const double2* __restrict__ trig,
                                                                   double* __restrict__ u) {
    constexpr int CW = CPLX ? 2 : 1;
    const int lane = threadIdx.x & 31, k = lane & 3;
    const int64_t tile = (int64_t)blockIdx.x * PT_W + (threadIdx.x >> 5);
    if (tile * PT_P >= npts) return;
    const int64_t ip = tile * PT_P + (lane >> 2);
    const int64_t iq = ip < npts ? ip : npts - 1;
    const double x0 = pts[3 * iq], x1 = pts[3 * iq + 1], x2 = pts[3 * iq + 2];
    const int64_t s0 = blockIdx.y * chunk, s1 = s0 + chunk < nsrc ? s0 + chunk : nsrc;
    double acc[NJ][CW];
#pragma unroll
    for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int c = 0; c < CW; ++c) acc[j][c] = 0.0;
    for (int64_t s = s0; s < s1; s += 4) {
        const int64_t sk = s + k < s1 ? s + k : s1 - 1;
        const double* y = qgeo + 4 * sk;
        const double d0 = x0 - y[0], d1 = x1 - y[1], d2 = x2 - y[2];
        double gr, gi;
        green64<CPLX>(fma(d0, d0, fma(d1, d1, d2 * d2)), kappa, 1.0, trig, &gr, &gi);
        const int live = (int)(s1 - s < 4 ? s1 - s : 4);
#pragma unroll 1
        for (int q = 0; q < live; ++q) {
            const int from = (lane & ~3) | q;
            const double hr = __shfl_sync(0xffffffffu, gr, from);
            const double hi = CPLX ? __shfl_sync(0xffffffffu, gi, from) : 0.0;
            const double* m = mu + ((s + q) * rc + k) * CW;
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                if (4 * j + k < rc) {
                    if constexpr (CPLX) {
                        const double2 v = *reinterpret_cast<const double2*>(m + 8 * j);
                        acc[j][0] = fma(hr, v.x, fma(-hi, v.y, acc[j][0]));
                        acc[j][CW - 1] = fma(hr, v.y, fma(hi, v.x, acc[j][CW - 1]));
                    } else {
                        acc[j][0] = fma(hr, m[4 * j], acc[j][0]);
                    }
                }
            }
        }
    }
    if (ip < npts)
#pragma unroll
        for (int j = 0; j < NJ; ++j)
            if (4 * j + k < rc)
#pragma unroll
                for (int c = 0; c < CW; ++c) atomicAdd(u + ((4 * j + k) * npts + ip) * CW + c, acc[j][c]);
}

template <bool CPLX>
cudaError_t launch_warp(ibem_handle* h, int rc, int64_t npts, const double* pts, const double* mu, double* u) {
    const Plan& P = h->P;
    const int64_t nsrc = P.E * P.Q * P.Q;
    const int64_t tiles = (npts + PT_P - 1) / PT_P;
    // slices of at least 64 sources, about 32 warps for every SM of the chip in all
    int64_t nsplit = (152 * 32 + tiles - 1) / tiles;
    nsplit = std::min<int64_t>(std::min<int64_t>(nsplit, (nsrc + 63) / 64), 65535);
    int64_t chunk = ((nsrc + nsplit - 1) / nsplit + 3) / 4 * 4;
    nsplit = (nsrc + chunk - 1) / chunk;
    const dim3 grid((unsigned)((tiles + PT_W - 1) / PT_W), (unsigned)nsplit);
    auto go = [&](auto kern) {
        kern<<<grid, 32 * PT_W, 0, h->stream>>>(npts, pts, nsrc, h->d_qgeo, mu, rc, chunk, P.prm.kappa, h->d_trig64, u);
        h->launches++;
        return cudaGetLastError();
    };
    const int nj = (rc + 3) / 4;
    return nj <= 1   ? go(potential_warp_kernel<CPLX, 1>)
           : nj <= 2 ? go(potential_warp_kernel<CPLX, 2>)
           : nj <= 4 ? go(potential_warp_kernel<CPLX, 4>)
           : nj <= 8 ? go(potential_warp_kernel<CPLX, 8>)
                     : go(potential_warp_kernel<CPLX, 16>);
}

}  // namespace

// Direct potential of nrhs densities; w is [R][N] real vectors, for a complex handle
// [2R][N] (real and imaginary part in turn).  The temporary data (densities at
// the Gauss points, up to PT_R of them) is released on the stream.
cudaError_t launch_potential_multi(ibem_handle* h, const double* w, int nrhs, const double* pts, int64_t npts,
                                   double* u) {
    const Plan& P = h->P;
    cudaStream_t st = h->stream;
    cudaError_t e;
    const int T = 256, QQ = P.Q * P.Q, CW = h->helm ? 2 : 1;
    const int64_t nsrc = P.E * QQ;
    if ((e = cudaMemsetAsync(u, 0, (size_t)CW * nrhs * npts * sizeof(double), st))) return e;
    if (npts <= 0) return cudaSuccess;
    // densities per pass: all of them up to PT_R, fewer where the table would exceed
    // 1 GiB (but at least 16 complex or 4 real ones)
    const int64_t fit = (int64_t)(1 << 30) / (nsrc * CW * 8);
    const int pass = (int)std::min<int64_t>(nrhs, std::min<int64_t>(PT_R, std::max<int64_t>(fit, h->helm ? 16 : 4)));
    double *mu = nullptr, *xs = nullptr;
    if ((e = cudaMallocAsync((void**)&mu, (size_t)nsrc * pass * CW * sizeof(double), st))) return e;
    if ((e = cudaMallocAsync((void**)&xs, (size_t)CW * pass * P.Nstar * sizeof(double), st))) {
        cudaFreeAsync(mu, st);
        return e;
    }
    for (int r0 = 0; r0 < nrhs && !e; r0 += pass) {
        const int rc = nrhs - r0 < pass ? nrhs - r0 : pass;
        lift_kernel<<<nblk((int64_t)CW * rc * P.E * P.nb, T), T, 0, st>>>(CW * rc, P.E, P.p, P.ne1, h->d_ext,
                                                                         w + (int64_t)CW * r0 * P.N, P.N, xs);
        if (h->helm)
            densities_kernel<true><<<nblk(nsrc * rc, T), T, 0, st>>>(P.E, QQ, P.nb, rc, h->d_qgeo, h->d_phi, xs, mu);
        else
            densities_kernel<false><<<nblk(nsrc * rc, T), T, 0, st>>>(P.E, QQ, P.nb, rc, h->d_qgeo, h->d_phi, xs, mu);
        h->launches += 2;
        double* ur = u + (int64_t)CW * r0 * npts;
        e = h->helm ? launch_warp<true>(h, rc, npts, pts, mu, ur) : launch_warp<false>(h, rc, npts, pts, mu, ur);
    }
    cudaFreeAsync(mu, st);
    cudaFreeAsync(xs, st);
    return e;
}

}  // namespace ibem
