// Maffettone-Minale droplet model (Sec. 2, Eqs. 1, 2, 4, 5 of Milan et al.,
// arXiv:2112.09972) for many gradient histories at once: one thread per
// trajectory integrates the morphology tensor M with classical RK4 and
// records D.  The paper compares its LBM droplets with this model; batching
// it on the GPU gives the model's deformation statistics over as many tracer
// trajectories as the LBM ensemble (Sec. 6).
//
// With tau_d = eta_s R / sigma, Ca(t) = tau_d ||G(t)||_inf (Eq. 3, element-wise
// maximum) and G = A the velocity gradient in lattice units,
//   dM/dt = [ f2(chi, Ca) tau_d (S M + M S) + tau_d (W M - M W)
//             - f1(chi) (M - 3 III_M / II_M I) ] / tau_d
// in LBM time, S and W the symmetric and antisymmetric parts of A (Eq. 2),
// II_M = ((tr M)^2 - M:M) / 2, III_M = det M, f1 and f2 of Eq. 5.  A(t) is the
// table row at integer t, linear in between.  D = (L - W)/(L + W) with L, W
// the square roots of M's extreme eigenvalues (Eq. 4).

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/lbm.h"
#include "lbm_eigen.cuh"

namespace lbmgb_mm {
namespace {

// symmetric 3x3 as 6 entries: xx, xy, xz, yy, yz, zz
template <typename C>
struct Sym {
    C v[6];
};

// n / d (d > 0) to the rounding of C or one unit more: an approximate float32
// reciprocal refined in C (4 to 6 instructions instead of a divide's dozen,
// which in float64 all run on the FP64 pipe); the plain divide outside
// float32's range.
__device__ __forceinline__ float quotient(float n, float d) {
    if (!(d > 1e-30f && d < 1e30f)) return n / d;
    const float y = __fdividef(1.f, d);
    const float q = n * y;
    return fmaf(fmaf(-q, d, n), y, q);
}
__device__ __forceinline__ double quotient(double n, double d) {
    const float df = (float)d;
    if (!(df > 1e-30f && df < 1e30f)) return n / d;
    const double y = (double)__fdividef(1.f, df);
    double q = n * y;
    q = fma(fma(-q, d, n), y, q);
    return fma(fma(-q, d, n), y, q);
}

// The largest |v_j|; float64 compares the bit patterns, which order as the
// values for numbers of one sign, on the integer pipe.
__device__ __forceinline__ float largest(const float (&v)[9]) {
    float m = 0.f;
#pragma unroll
    for (int j = 0; j < 9; ++j) m = fmaxf(m, fabsf(v[j]));
    return m;
}
__device__ __forceinline__ double largest(const double (&v)[9]) {
    unsigned long long m = 0;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v[j]) & 0x7fffffffffffffffull;
        m = b > m ? b : m;
    }
    return __longlong_as_double((long long)m);
}

// The linear part of the model at one time: B = f2(Ca) S + W - k / 2 I,
// row-major, k = f1 / tau_d, so that f2 (S M + M S) + W M - M W - k M =
// B M + (B M)^T (S symmetric, W antisymmetric).
template <typename C>
struct Flow {
    C b[9];
};
template <typename C>
__device__ __forceinline__ Flow<C> flow_at(const C (&a0)[9], const C (&d)[9], C t, C tau_d, C f2_0, C k) {
    C A[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) A[j] = fma(t, d[j], a0[j]);
    const C Ca = tau_d * largest(A), c2 = Ca * Ca;
    const C f2 = f2_0 + quotient(C(3) * c2, fma(C(6), c2, C(2)));
    const C p = fma(C(0.5), f2, C(0.5)), m = fma(C(0.5), f2, C(-0.5));
    Flow<C> F;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            F.b[3 * a + b] = a == b ? fma(f2, A[4 * a], C(-0.5) * k) : fma(p, A[3 * a + b], m * A[3 * b + a]);
    return F;
}

// dM/dt = B M + (B M)^T + 3 k III / II I.
template <typename C>
__device__ __forceinline__ Sym<C> rhs(const Sym<C>& M, const Flow<C>& F, C k3) {
    const C* m = M.v;
    const C* b = F.b;
    // cofactors: II is their trace, III the expansion along the first row
    const C c0 = fma(m[3], m[5], -m[4] * m[4]), c1 = fma(m[0], m[5], -m[2] * m[2]), c2 = fma(m[0], m[3], -m[1] * m[1]);
    const C u = fma(m[1], m[5], -m[4] * m[2]), v = fma(m[1], m[4], -m[3] * m[2]);
    const C III = fma(m[0], c0, fma(m[2], v, -m[1] * u));
    const C iso = quotient(k3 * III, c0 + c1 + c2);
    Sym<C> r;
    r.v[0] = fma(C(2), fma(b[0], m[0], fma(b[1], m[1], b[2] * m[2])), iso);
    r.v[3] = fma(C(2), fma(b[3], m[1], fma(b[4], m[3], b[5] * m[4])), iso);
    r.v[5] = fma(C(2), fma(b[6], m[2], fma(b[7], m[4], b[8] * m[5])), iso);
    // (B M)_ab + (B M)_ba
    r.v[1] = fma(b[0], m[1], fma(b[1], m[3], b[2] * m[4])) + fma(b[3], m[0], fma(b[4], m[1], b[5] * m[2]));
    r.v[2] = fma(b[0], m[2], fma(b[1], m[4], b[2] * m[5])) + fma(b[6], m[0], fma(b[7], m[1], b[8] * m[2]));
    r.v[4] = fma(b[3], m[2], fma(b[4], m[4], b[5] * m[5])) + fma(b[6], m[1], fma(b[7], m[3], b[8] * m[4]));
    return r;
}

template <typename C>
__device__ __forceinline__ Sym<C> axpy(const Sym<C>& m, C h, const Sym<C>& k) {
    Sym<C> r;
#pragma unroll
    for (int e = 0; e < 6; ++e) r.v[e] = fma(h, k.v[e], m.v[e]);
    return r;
}

template <typename C>
__device__ __forceinline__ double deformation(const Sym<C>& M) {
    const double m[6] = {(double)M.v[0], (double)M.v[1], (double)M.v[2],
                         (double)M.v[3], (double)M.v[4], (double)M.v[5]};
    return lbmgb::deformation_of(m);
}

// One warp per CTA, so that few trajectories still spread over the SMs: the
// float64 form is bound by the FP64 pipe (one warp instruction per 16 cycles
// and SM), the float32 form by its dependent chain at about one warp per
// scheduler.  A stage is one B M product (27 multiply-adds), the cofactors
// and one quotient; B is formed once per time it is needed at (the middle
// serves two stages, the end is the next substep's start), and the next row
// of A is loaded a step ahead.  Measured on GB300, 16384 trajectories:
// float64, 50 steps of 4 substeps, 6912 -> 2780 us, float32, 250 steps of 10
// substeps with 31 records, 4908 -> 1520 us, against separate S M and W M
// products formed per stage and a Jacobi D; one warp's float64 chain alone
// (100 trajectories) takes 2530 us.
constexpr int kMMThreads = 32;
template <typename C>
__global__ void __launch_bounds__(kMMThreads) k_mm_rk4(const double* __restrict__ A, long long T, long long n, C tau_d,
                                                       C f2_0, C kf, int substeps, int record_every,
                                                       double* __restrict__ D, double* __restrict__ Mout) {
    const long long k = (long long)blockIdx.x * kMMThreads + threadIdx.x;
    if (k >= n) return;
    Sym<C> M;
#pragma unroll
    for (int e = 0; e < 6; ++e) M.v[e] = (e == 0 || e == 3 || e == 5) ? C(1) : C(0);
    D[k] = 0.0;  // the sphere
    const C h = C(1) / C(substeps);
    C a0[9], d[9];
    double next[9];
    const double* row = A + k * 9;
#pragma unroll
    for (int j = 0; j < 9; ++j) a0[j] = (C)row[j];
    if (T > 1)
#pragma unroll
        for (int j = 0; j < 9; ++j) next[j] = row[n * 9 + j];
#pragma unroll
    for (int j = 0; j < 9; ++j) d[j] = C(0);
    Flow<C> Fs = flow_at<C>(a0, d, C(0), tau_d, f2_0, kf);
    const C kiso = C(3) * kf;
    int until = record_every;
    long long rec = 0;
    for (long long s = 0; s + 1 < T; ++s) {
#pragma unroll
        for (int j = 0; j < 9; ++j) d[j] = (C)next[j] - a0[j];
        row += n * 9;
        C a1[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) a1[j] = (C)next[j];
        if (s + 2 < T)
#pragma unroll
            for (int j = 0; j < 9; ++j) next[j] = row[n * 9 + j];
        for (int q = 0; q < substeps; ++q) {
            // A at the middle and end of the substep (linear in t)
            const Flow<C> Fm = flow_at<C>(a0, d, (C(q) + C(0.5)) * h, tau_d, f2_0, kf);
            const Sym<C> k1 = rhs(M, Fs, kiso);
            Sym<C> sum = k1;
            const Sym<C> k2 = rhs(axpy(M, C(0.5) * h, k1), Fm, kiso);
            const Sym<C> kc = rhs(axpy(M, C(0.5) * h, k2), Fm, kiso);
#pragma unroll
            for (int e = 0; e < 6; ++e) sum.v[e] = fma(C(2), k2.v[e] + kc.v[e], sum.v[e]);
            Fs = flow_at<C>(a0, d, C(q + 1) * h, tau_d, f2_0, kf);
            const Sym<C> k4 = rhs(axpy(M, h, kc), Fs, kiso);
#pragma unroll
            for (int e = 0; e < 6; ++e) M.v[e] = fma(h / C(6), sum.v[e] + k4.v[e], M.v[e]);
        }
#pragma unroll
        for (int j = 0; j < 9; ++j) a0[j] = a1[j];
        if (--until == 0) {
            until = record_every;
            D[++rec * n + k] = deformation(M);
        }
    }
    if (Mout)
#pragma unroll
        for (int e = 0; e < 6; ++e) Mout[k * 6 + e] = (double)M.v[e];
}

}  // namespace
}  // namespace lbmgb_mm

extern "C" int lbm_mm_integrate(const double* A, int64_t T, int64_t n, double tau_d, double chi, int32_t substeps,
                                int32_t record_every, int32_t precision, double* D, double* M, void* cuda_stream) {
    if (!A || !D || T < 1 || n < 1 || !(tau_d > 0.0) || !(chi > 0.0) || substeps < 1 || record_every < 1)
        return LBM_EINVAL;
    if (precision != LBM_FP64 && precision != LBM_FP32) return LBM_EINVAL;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int threads = lbmgb_mm::kMMThreads;
    const unsigned blocks = (unsigned)((n + threads - 1) / threads);
    const double f1 = 40.0 * (chi + 1.0) / ((3.0 + 2.0 * chi) * (16.0 + 19.0 * chi)), f2_0 = 5.0 / (3.0 + 2.0 * chi);
    if (precision == LBM_FP64)
        lbmgb_mm::k_mm_rk4<double><<<blocks, threads, 0, s>>>(A, T, n, tau_d, f2_0, f1 / tau_d, substeps, record_every,
                                                              D, M);
    else
        lbmgb_mm::k_mm_rk4<float><<<blocks, threads, 0, s>>>(A, T, n, (float)tau_d, (float)f2_0, (float)(f1 / tau_d),
                                                             substeps, record_every, D, M);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ECUDA;
}
