// Near-field assembly (FP64): Galerkin blocks of element pairs in the Bernstein
// superspace (Sec. 3.2, Sec. 4.3, Sec. 4 item 4),
//     B[i][j] = int_t int_s k(x) k(y) u*(F(x), F(y)) B_i(x) B_j(y) dy dx,
// Laplace and Helmholtz, for regular and subdivided pairs (product Gauss rules)
// and for touching pairs (Duffy-type rules).
//
// Everything here is bound by the FP64 pipe (2 operations per clock and SM; the
// forms before this one ran it at 88-92%), so the work is in the operation count:
//  - u* and the rules are symmetric, so the block of (s, t) is the transpose of that
//    of (t, s): each unordered pair is formed once and written twice, and an
//    identical pair takes half of its pieces (B = S + S^T);
//  - a kernel value takes a reciprocal square root and a table-based e^{i theta}
//    (fp64_eval.cuh) instead of square root, division and sincos;
//  - a sphere face gives point and surface measure from one reciprocal square root;
//  - sums against B_i(x) B_j(y) are factorised over the directions in which the rule
//    is a product.
// Operations per point and complex value (p = 2): touching pairs about 150 instead
// of 820, product rules 45 instead of 107.
// Sphere, p = 2, level 3, kappa = 4: touching 11.8 ms instead of 96.8, subdivided and
// regular 12.9 ms instead of 42.2; whole assembly at level 5 (kappa = 4) 0.34 s
// instead of 1.89 s, Laplace p = 3 level 5 0.32 s instead of 1.93 s.
#include "fp64_eval.cuh"
#include "ibem_internal.cuh"

namespace ibem {

namespace {

constexpr int NT = 128;      // threads per CTA

__device__ inline void element_at(int64_t e, int ne1, int* patch, int* ix, int* iy) {
    const int64_t per = (int64_t)ne1 * ne1;
    *patch = (int)(e / per);
    uint32_t x, y;
    morton2_inv((uint32_t)(e % per), &x, &y);
    *ix = (int)x;
    *iy = (int)y;
}

__device__ __noinline__ void general_point(GeomView g, int patch, double u, double v, double* F, double* k) {
    double Fu[3], Fv[3];
    eval_patch(g, patch, u, v, F, Fu, Fv);
    *k = surface_measure(Fu, Fv);
}

// F(u, v) and the surface measure.  Sphere face: c = n + a t1 + b t2 with the
// orthonormal frame (n, t1, t2), F = c0 + R c / |c|, measure 4 R^2 / |c|^3 (central
// projection of a plane at distance 1, parameters scaled by 2).
__device__ __forceinline__ void point_at(const GeomView& g, int patch, double u, double v, double* F, double* k) {
    const PatchDesc& P = g.patches[patch];
    if (P.kind != IBEM_PATCH_SPHERE_FACE) {
        general_point(g, patch, u, v, F, k);
        return;
    }
    double du = 1.0, dv = 1.0;
    if (P.perturbed) {
        u = perturbation_f(u, &du);
        v = perturbation_f(v, &dv);
    }
    const double a = fma(2.0, u, -1.0), b = fma(2.0, v, -1.0);
    double c[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) c[i] = fma(b, P.t2[i], fma(a, P.t1[i], P.n[i]));
    const double inv = rsqrt(fma(c[0], c[0], fma(c[1], c[1], c[2] * c[2])));
    const double q = P.R * inv;
#pragma unroll
    for (int i = 0; i < 3; ++i) F[i] = fma(q, c[i], P.c0[i]);
    *k = 4.0 * q * q * inv;
    if (P.perturbed) *k *= du * dv;
}

// Bernstein polynomials of degree PP - 1 at t
template <int PP>
__device__ __forceinline__ void bernstein_at(double t, double (&b)[PP]) {
    const double s = 1.0 - t;
    b[0] = 1.0;
#pragma unroll
    for (int d = 1; d < PP; ++d) {
        double prev = 0.0;
#pragma unroll
        for (int i = 0; i < PP - 1; ++i)
            if (i < d) {
                const double cur = b[i];
                b[i] = fma(s, cur, prev);
                prev = t * cur;
            }
        b[d] = prev;
    }
}

// index of the pair (s, t) in the lists, -1 if it is not there (the plan refuses such lists)
__device__ inline int64_t mirror_of(int64_t t, int64_t s, const int64_t* __restrict__ nptr,
                                    const int32_t* __restrict__ nsrc) {
    int64_t lo = nptr[s], hi = nptr[s + 1];
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (nsrc[mid] < t) lo = mid + 1;
        else hi = mid;
    }
    return lo < nptr[s + 1] && nsrc[lo] == t ? lo : -1;
}

// ---- regular and subdivided pairs ------------------------------------------------
// One CTA per pair.  An element carries NQ x NQ points: the Gauss rule (NQ = Q) or,
// subdivided, the rule on both halves of either direction (NQ = 2 Q), which is the
// same sum as over the 16 sub-square pairs.  In chunks of CA target points: thread
// items (a, b_v) evaluate the NQ values over b_u and keep T[a][b_v][j_u]; then
// H[a][j] = sum_{b_v} B_{j_v}(b_v) T; then B[i][j] += sum_a B_i(a) H[a][j].
// Shared: XA, XB [NQ^2][4], b1 [NQ][PP], T [CA][NQ][PP], H [CA][nb] (complex twice).
inline __host__ __device__ int product_chunk(int NQ) { return 4 * NT / NQ < NQ * NQ ? 4 * NT / NQ : NQ * NQ; }

template <bool CPLX, int PP>
__global__ void __launch_bounds__(NT) near_product_kernel(GeomView g, const int32_t* __restrict__ list,
                                                          const int32_t* __restrict__ tgt,
                                                          const int32_t* __restrict__ src,
                                                          const int64_t* __restrict__ nptr,
                                                          const int32_t* __restrict__ nsrc,
                                                          const double* __restrict__ qgeo,
                                                          const double* __restrict__ rule, int Q, int ne1, bool subdiv,
                                                          double kappa, const double2* __restrict__ trig,
                                                          double* __restrict__ blocks) {
    constexpr int CW = CPLX ? 2 : 1, nb = PP * PP, NE = (nb * nb + NT - 1) / NT;
    extern __shared__ double sm[];
    const int NQ = subdiv ? 2 * Q : Q, NA = NQ * NQ, CA = product_chunk(NQ);
    double* XA = sm;
    double* XB = XA + 4 * NA;
    double* b1 = XB + 4 * NA;
    double* T = b1 + NQ * PP;
    double* H = T + (size_t)CA * NQ * PP * CW;
    __shared__ int64_t mirror;
    const int64_t k = list[blockIdx.x], t = tgt[k], s = src[k];
    const double h = 1.0 / ne1;
    if (threadIdx.x == 0) mirror = mirror_of(t, s, nptr, nsrc);
    for (int i = threadIdx.x; i < 2 * NA; i += NT) {
        const int which = i / NA, q = i - which * NA, qu = q % NQ, qv = q / NQ;
        double* o = (which ? XB : XA) + 4 * q;
        if (!subdiv) {
            const double* in = qgeo + 4 * (NA * (which ? s : t) + q);
            o[0] = in[0]; o[1] = in[1]; o[2] = in[2]; o[3] = in[3];
        } else {
            int patch, ix, iy;
            element_at(which ? s : t, ne1, &patch, &ix, &iy);
            const double u = 0.5 * (qu / Q) + 0.5 * rule[qu % Q], v = 0.5 * (qv / Q) + 0.5 * rule[qv % Q];
            double F[3], m;
            point_at(g, patch, (ix + u) * h, (iy + v) * h, F, &m);
            o[0] = F[0]; o[1] = F[1]; o[2] = F[2];
            o[3] = 0.25 * rule[Q + qu % Q] * rule[Q + qv % Q] * m * h * h;
        }
    }
    for (int q = threadIdx.x; q < NQ; q += NT) {
        double b[PP];
        bernstein_at<PP>(subdiv ? 0.5 * (q / Q) + 0.5 * rule[q % Q] : rule[q], b);
#pragma unroll
        for (int j = 0; j < PP; ++j) b1[q * PP + j] = b[j];
    }
    double acc[NE][CW];
#pragma unroll
    for (int i = 0; i < NE; ++i)
#pragma unroll
        for (int c = 0; c < CW; ++c) acc[i][c] = 0.0;
    const double inv4pi = 1.0 / (4.0 * IBEM_PI);
    for (int a0 = 0; a0 < NA; a0 += CA) {
        const int na = NA - a0 < CA ? NA - a0 : CA;
        __syncthreads();   // XA, XB written; T and H of the previous chunk used
        for (int it = threadIdx.x; it < na * NQ; it += NT) {
            const int a = it % na, bv = it / na;
            const double* A = XA + 4 * (a0 + a);
            const double x0 = A[0], x1 = A[1], x2 = A[2], wa = A[3] * inv4pi;
            double row[PP][CW];
#pragma unroll
            for (int j = 0; j < PP; ++j)
#pragma unroll
                for (int c = 0; c < CW; ++c) row[j][c] = 0.0;
            const double* B = XB + 4 * bv * NQ;
            for (int bu = 0; bu < NQ; ++bu) {
                const double d0 = x0 - B[4 * bu], d1 = x1 - B[4 * bu + 1], d2 = x2 - B[4 * bu + 2];
                double v[2];
                green64<CPLX>(fma(d0, d0, fma(d1, d1, d2 * d2)), kappa, wa * B[4 * bu + 3], trig, &v[0], &v[1]);
#pragma unroll
                for (int j = 0; j < PP; ++j)
#pragma unroll
                    for (int c = 0; c < CW; ++c) row[j][c] = fma(v[c], b1[bu * PP + j], row[j][c]);
            }
            double* o = T + (size_t)(a * NQ + bv) * PP * CW;
#pragma unroll
            for (int j = 0; j < PP; ++j)
#pragma unroll
                for (int c = 0; c < CW; ++c) o[j * CW + c] = row[j][c];
        }
        __syncthreads();
        for (int it = threadIdx.x; it < na * nb; it += NT) {
            const int a = it / nb, j = it - a * nb, ju = j % PP, jv = j / PP;
            double v[CW] = {};
            const double* in = T + ((size_t)a * NQ * PP + ju) * CW;
            for (int bv = 0; bv < NQ; ++bv)
#pragma unroll
                for (int c = 0; c < CW; ++c) v[c] = fma(b1[bv * PP + jv], in[bv * PP * CW + c], v[c]);
#pragma unroll
            for (int c = 0; c < CW; ++c) H[it * CW + c] = v[c];
        }
        __syncthreads();
#pragma unroll
        for (int n = 0; n < NE; ++n) {
            const int e = threadIdx.x + NT * n;
            if (e < nb * nb) {
                const int i = e / nb, j = e - i * nb;
                double v[CW] = {};
                for (int a = 0; a < na; ++a) {
                    const int q = a0 + a;
                    const double w = b1[(q % NQ) * PP + i % PP] * b1[(q / NQ) * PP + i / PP];
#pragma unroll
                    for (int c = 0; c < CW; ++c) v[c] = fma(w, H[(a * nb + j) * CW + c], v[c]);
                }
#pragma unroll
                for (int c = 0; c < CW; ++c) acc[n][c] += v[c];
            }
        }
    }
    const int64_t k2 = mirror;
#pragma unroll
    for (int n = 0; n < NE; ++n) {
        const int e = threadIdx.x + NT * n;
        if (e < nb * nb) {
            const int i = e / nb, j = e - i * nb;
#pragma unroll
            for (int c = 0; c < CW; ++c) {
                blocks[(k * nb * nb + e) * CW + c] = acc[n][c];
                if (k2 >= 0) blocks[(k2 * nb * nb + j * nb + i) * CW + c] = acc[n][c];
            }
        }
    }
}

// ---- touching pairs ---------------------------------------------------------------
// Duffy-type rules in the canonical coordinates (x1, x2, y1, y2), n Gauss points per
// variable (a, b, c, s):
//   identical (8 pieces: triangle, ordering in x1 / y1, ordering in x2 / y2; the
//     second ordering of x1 / y1 is the first with x and y exchanged and is left to
//     S + S^T), edge (6: pyramid, ordering), vertex (4: which coordinate is xi).
// For a fixed triple (a, b, c) the coordinates x1, y1 are fixed and x2, y2 are affine
// in s, so with the element coordinates u' of x1 and t' of x2 (after the pair's
// orientation) the block is
//   sum over triples of [B_i1(x1) B_j1(y1)] [sum_s v(s) B_i2(x2(s)) B_j2(y2(s))].
// A thread takes a triple, its n points and the inner sum; the outer product over
// NT triples runs through shared memory (P, W: [PP^2][NT]).
struct Triple {
    double x1, y1, x20, x2s, y20, y2s, w;   // x2 = x20 + x2s s
};

__device__ __forceinline__ Triple duffy_triple(int cls, int piece, double a, double b, double c, double w) {
    Triple r;
    if (cls == CLS_VERTEX) {
        // the largest coordinate is a; the others a b, a c, a s (the rule is symmetric in b, c, s)
        const double ab = a * b, ac = a * c;
        r.w = w * a * a * a;
        r.x20 = r.x2s = r.y20 = r.y2s = 0.0;
        if (piece == 0) { r.x1 = a; r.x20 = ab; r.y1 = ac; r.y2s = a; }
        else if (piece == 1) { r.x1 = ab; r.x20 = a; r.y1 = ac; r.y2s = a; }
        else if (piece == 2) { r.x1 = ab; r.x20 = ac; r.y1 = a; r.y2s = a; }
        else { r.x1 = ab; r.x2s = a; r.y1 = ac; r.y20 = a; }
        return r;
    }
    double z;       // |y2 - x2|
    if (cls == CLS_IDENTICAL) {
        const double ab = a * b, z1 = piece & 2 ? ab : a;
        z = piece & 2 ? a : ab;
        const double lo = (1.0 - z1) * c;
        r.x1 = lo;
        r.y1 = lo + z1;
        r.w = w * a * (1.0 - z1) * (1.0 - z);
    } else {
        const double ab = a * b, ac = a * c;
        const int pyr = piece >> 1;
        r.x1 = pyr == 0 ? a : ab;
        r.y1 = pyr == 0 ? ab : (pyr == 1 ? a : ac);
        z = pyr == 2 ? a : ac;
        r.w = w * a * a * (1.0 - z);
    }
    r.x2s = r.y2s = 1.0 - z;
    r.x20 = piece & 1 ? z : 0.0;
    r.y20 = piece & 1 ? 0.0 : z;
    return r;
}

// the symmetries of the square as x' from s or t and flips: (s', t') = (s or 1 - s,
// t or 1 - t), (x, y) = (s', t') or (t', s') (the order of dihedral())
__device__ __forceinline__ void orientation(int k, bool* swap, bool* fs, bool* ft) {
    *swap = (0x5A >> k) & 1;     // 1, 3, 4, 6
    *fs = (0x6C >> k) & 1;       // 2, 3, 5, 6
    *ft = (0xC6 >> k) & 1;       // 1, 2, 6, 7
}

template <bool CPLX, int PP>
__global__ void __launch_bounds__(NT) near_touch_kernel(GeomView g, int cls, const int32_t* __restrict__ list,
                                                        const int32_t* __restrict__ tgt,
                                                        const int32_t* __restrict__ src,
                                                        const int32_t* __restrict__ orient,
                                                        const int64_t* __restrict__ nptr,
                                                        const int32_t* __restrict__ nsrc,
                                                        const double* __restrict__ rule, int n, int ne1, double kappa,
                                                        const double2* __restrict__ trig,
                                                        double* __restrict__ blocks) {
    constexpr int CW = CPLX ? 2 : 1, nb = PP * PP, NE = (nb * nb + NT - 1) / NT;
    extern __shared__ double sm[];
    double* Ps = sm;                     // [nb][NT]
    double* Ws = Ps + nb * NT;           // [CW][nb][NT]
    __shared__ int64_t mirror;
    const int64_t k = list[blockIdx.x], t = tgt[k], s = src[k];
    if (threadIdx.x == 0) mirror = mirror_of(t, s, nptr, nsrc);
    int pa, ixa, iya, pb, ixb, iyb;
    element_at(t, ne1, &pa, &ixa, &iya);
    element_at(s, ne1, &pb, &ixb, &iyb);
    bool swA, fsA, ftA, swB, fsB, ftB;
    orientation(orient[k] >> 3, &swA, &fsA, &ftA);
    orientation(orient[k] & 7, &swB, &fsB, &ftB);
    const double h = 1.0 / ne1;
    const double scale = h * h * h * h / (4.0 * IBEM_PI);
    const int n3 = n * n * n;
    const int total = (cls == CLS_IDENTICAL ? 4 : (cls == CLS_EDGE ? 6 : 4)) * n3;
    // the entries of a thread rotate with the CTA, so that the idle warps of a small
    // block do not always share a scheduler
    const int e0 = (threadIdx.x + 32 * (blockIdx.x & 3)) % NT;
    double acc[NE][CW];
#pragma unroll
    for (int i = 0; i < NE; ++i)
#pragma unroll
        for (int c = 0; c < CW; ++c) acc[i][c] = 0.0;
    for (int base = 0; base < total; base += NT) {
        const int it = base + threadIdx.x;
        if (it < total) {
            const int piece = it / n3, r = it - piece * n3, qa = r / (n * n), qb = (r / n) % n, qc = r % n;
            Triple tr = duffy_triple(cls, piece, rule[qa], rule[qb], rule[qc],
                                     scale * rule[n + qa] * rule[n + qb] * rule[n + qc]);
            if (fsA) tr.x1 = 1.0 - tr.x1;
            if (fsB) tr.y1 = 1.0 - tr.y1;
            if (ftA) { tr.x20 = 1.0 - tr.x20; tr.x2s = -tr.x2s; }
            if (ftB) { tr.y20 = 1.0 - tr.y20; tr.y2s = -tr.y2s; }
            double W[nb][CW];
#pragma unroll
            for (int j = 0; j < nb; ++j)
#pragma unroll
                for (int c = 0; c < CW; ++c) W[j][c] = 0.0;
            double FA[3], FB[3], kA = 0.0, kB = 0.0;
            for (int q = 0; q < n; ++q) {
                const double x2 = fma(tr.x2s, rule[q], tr.x20), y2 = fma(tr.y2s, rule[q], tr.y20);
                // a vertex pair moves one of its two points only
                if (q == 0 || tr.x2s != 0.0)
                    point_at(g, pa, (ixa + (swA ? x2 : tr.x1)) * h, (iya + (swA ? tr.x1 : x2)) * h, FA, &kA);
                if (q == 0 || tr.y2s != 0.0)
                    point_at(g, pb, (ixb + (swB ? y2 : tr.y1)) * h, (iyb + (swB ? tr.y1 : y2)) * h, FB, &kB);
                const double d0 = FA[0] - FB[0], d1 = FA[1] - FB[1], d2 = FA[2] - FB[2];
                double v[2];
                green64<CPLX>(fma(d0, d0, fma(d1, d1, d2 * d2)), kappa, tr.w * rule[n + q] * kA * kB, trig, &v[0],
                              &v[1]);
                double bx[PP], by[PP];
                bernstein_at<PP>(x2, bx);
                bernstein_at<PP>(y2, by);
#pragma unroll
                for (int i = 0; i < PP; ++i)
#pragma unroll
                    for (int c = 0; c < CW; ++c) {
                        const double vb = v[c] * bx[i];
#pragma unroll
                        for (int j = 0; j < PP; ++j) W[i * PP + j][c] = fma(vb, by[j], W[i * PP + j][c]);
                    }
            }
            double bx[PP], by[PP];
            bernstein_at<PP>(tr.x1, bx);
            bernstein_at<PP>(tr.y1, by);
#pragma unroll
            for (int i = 0; i < PP; ++i)
#pragma unroll
                for (int j = 0; j < PP; ++j) {
                    Ps[(i * PP + j) * NT + threadIdx.x] = bx[i] * by[j];
#pragma unroll
                    for (int c = 0; c < CW; ++c) Ws[(c * nb + i * PP + j) * NT + threadIdx.x] = W[i * PP + j][c];
                }
        }
        __syncthreads();
        const int m = total - base < NT ? total - base : NT;
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            const int e = e0 + NT * i;
            if (e < nb * nb) {
                const double* p = Ps + (e / nb) * NT;
                const double* w = Ws + (e % nb) * NT;
                double v[CW] = {};
                for (int q = 0; q < m; ++q)
#pragma unroll
                    for (int c = 0; c < CW; ++c) v[c] = fma(p[q], w[c * nb * NT + q], v[c]);
#pragma unroll
                for (int c = 0; c < CW; ++c) acc[i][c] += v[c];
            }
        }
        __syncthreads();
    }
    // entry e = (i1 j1, i2 j2) -> block entry (i, j); identical pairs add the transpose
    double* S = sm;                      // [nb][nb] (complex twice): at most 25 x 25 x 2 <= 3 x 25 x 128
#pragma unroll
    for (int q = 0; q < NE; ++q) {
        const int e = e0 + NT * q;
        if (e < nb * nb) {
            const int i1 = e / nb / PP, j1 = e / nb % PP, i2 = e % nb / PP, j2 = e % PP;
            const int i = swA ? i1 * PP + i2 : i2 * PP + i1, j = swB ? j1 * PP + j2 : j2 * PP + j1;
#pragma unroll
            for (int c = 0; c < CW; ++c) S[(i * nb + j) * CW + c] = acc[q][c];
        }
    }
    __syncthreads();
    const int64_t k2 = mirror;
    for (int e = threadIdx.x; e < nb * nb * CW; e += NT) {
        const int c = e % CW, ij = e / CW, i = ij / nb, j = ij - i * nb;
        const double v = S[e], vt = S[(j * nb + i) * CW + c];
        if (cls == CLS_IDENTICAL) {
            blocks[k * nb * nb * CW + e] = v + vt;
        } else {
            blocks[k * nb * nb * CW + e] = v;
            if (k2 >= 0) blocks[k2 * nb * nb * CW + e] = vt;
        }
    }
}

template <bool CPLX, int PP>
cudaError_t launch_pp(ibem_handle* h, double kappa, double* blocks) {
    const Plan& P = h->P;
    constexpr int CW = CPLX ? 2 : 1, nb = PP * PP;
    const GeomView g{h->d_patches, h->d_knots, h->d_cpw};
    cudaError_t e;
    for (int cls : {CLS_REGULAR, CLS_SUBDIV}) {
        if (h->n_list[cls] == 0 || near_streamed(P.Q, nb, CPLX, cls == CLS_SUBDIV)) continue;
        const int NQ = cls == CLS_SUBDIV ? 2 * P.Q : P.Q, CA = product_chunk(NQ);
        const size_t smem = ((size_t)8 * NQ * NQ + (size_t)NQ * PP + (size_t)CA * NQ * PP * CW + (size_t)CA * nb * CW) *
                            sizeof(double);
        if ((e = cudaFuncSetAttribute(near_product_kernel<CPLX, PP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem)))
            return e;
        near_product_kernel<CPLX, PP><<<(unsigned)h->n_list[cls], NT, smem, h->stream>>>(
            g, h->d_pairs_by_cls[cls], h->d_near_tgt, h->d_near_src, h->d_near_ptr, h->d_near_src, h->d_qgeo,
            h->d_gauss, P.Q, P.ne1, cls == CLS_SUBDIV, kappa, h->d_trig64, blocks);
    }
    const size_t smem = (size_t)(1 + CW) * nb * NT * sizeof(double);
    if ((e = cudaFuncSetAttribute(near_touch_kernel<CPLX, PP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
        return e;
    for (int cls : {CLS_IDENTICAL, CLS_EDGE, CLS_VERTEX}) {
        if (h->n_list[cls] == 0) continue;
        near_touch_kernel<CPLX, PP><<<(unsigned)h->n_list[cls], NT, smem, h->stream>>>(
            g, cls, h->d_pairs_by_cls[cls], h->d_near_tgt, h->d_near_src, h->d_near_orient, h->d_near_ptr,
            h->d_near_src, h->d_gauss + 2 * P.Q, P.Qs, P.ne1, kappa, h->d_trig64, blocks);
    }
    return cudaGetLastError();
}

template <bool CPLX>
cudaError_t launch_cplx(ibem_handle* h, double kappa, double* blocks) {
    switch (h->P.pp) {
        case 1: return launch_pp<CPLX, 1>(h, kappa, blocks);
        case 2: return launch_pp<CPLX, 2>(h, kappa, blocks);
        case 3: return launch_pp<CPLX, 3>(h, kappa, blocks);
        case 4: return launch_pp<CPLX, 4>(h, kappa, blocks);
        case 5: return launch_pp<CPLX, 5>(h, kappa, blocks);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// The product rules form the regular and subdivided pairs up to the order whose
// Q^2 x Q^2 kernel matrix would fit in a CTA's shared memory (12 for Laplace, 10 for
// Helmholtz at p = 2); the streaming kernel, whose shared memory grows with Q^2 only,
// takes the higher ones.  The line is not where the two are level: assembly of the
// sphere at p = 2, level 2 takes 15.2 ms with order 12 and 48.9 with 13 for Laplace, 19.1
// with order 10, 74.7 with 12 and 97.4 with 13 for Helmholtz, and the kernel values alone
// would account for factors of 1.4 and 2.1.
bool near_streamed(int Q, int nb, bool cplx, bool subdiv) {
    const size_t QQ = (size_t)Q * Q, cw = cplx ? 2 : 1;
    return (subdiv ? 32 * QQ + cw * QQ * QQ + cw * QQ * nb + cw * nb * nb : 8 * QQ + cw * QQ * QQ + cw * QQ * nb) *
               sizeof(double) >
           IBEM_MAX_SMEM_BYTES;
}

// Near blocks of every class whose pairs are not streamed; the class lists hold one
// of every two mirrored pairs (and all identical ones).
cudaError_t launch_near_blocks(ibem_handle* h, bool cplx, double kappa, double* blocks) {
    return cplx ? launch_cplx<true>(h, kappa, blocks) : launch_cplx<false>(h, kappa, blocks);
}

}  // namespace ibem
