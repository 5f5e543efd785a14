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
#include <math.h>
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

using lbmgb::rcp_seed;
// The same of a float64 between 2^-100 and 2^100 (narrow and widen of a positive number).
__device__ __forceinline__ double rcp_seed(double d) {
    const unsigned hi = (unsigned)__double2hiint(d) - (896u << 20), lo = (unsigned)__double2loint(d);
    const unsigned y = __float_as_uint(rcp_seed(__uint_as_float(__funnelshift_l(lo, hi, 3))));
    return __hiloint2double((int)((y >> 3) + (896u << 20)), (int)(y << 29));
}
__device__ __forceinline__ bool in_range(float d) { return d > 1e-30f && d < 1e30f; }
__device__ __forceinline__ bool in_range(double d) {
    return (unsigned)__double2hiint(d) - ((1023u - 100u) << 20) < (200u << 20);
}

// n / d, d > 0.  Safe: the plain divide.  Otherwise the reciprocal's seed y
// and its error e = 1 - d y: n y (1 + e) in float32, n y (1 + e + e^2) in
// float64, within a unit or two of the last place where d is in range; ok
// turns false where it is not.  Without the divide's branches a whole substep
// is one block that the compiler can interleave.
template <bool Safe, typename C>
__device__ __forceinline__ C quotient(C n, C d, bool& ok) {
    if constexpr (Safe) {
        return n / d;
    } else {
        ok = ok && in_range(d);
        const C y = rcp_seed(d), q = n * y;
        if constexpr (sizeof(C) == 4) {
            return fma(fma(-q, d, n), y, q);
        } else {
            const C e = fma(-d, y, C(1));
            return fma(q, fma(e, e, e), q);
        }
    }
}

// The largest v_j >= 0; float64 compares the bit patterns, which order as the
// values, on the integer pipe.
__device__ __forceinline__ float largest(const float (&v)[6]) {
    float m = 0.f;
#pragma unroll
    for (int j = 0; j < 6; ++j) m = fmaxf(m, v[j]);
    return m;
}
__device__ __forceinline__ double largest(const double (&v)[6]) {
    long long m = 0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const long long b = __double_as_longlong(v[j]);
        m = b > m ? b : m;
    }
    return __longlong_as_double(m);
}

// The gradient in the form the stages want it: 2 S and 2 W.  v[0..2] = 2 A_aa,
// v[3..5] = A_ab + A_ba, v[6..8] = A_ab - A_ba for ab = xy, xz, yz.
template <typename C>
__device__ __forceinline__ void split_gradient(const C (&A)[9], C (&v)[9]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) v[a] = A[4 * a] + A[4 * a];
    v[3] = A[1] + A[3], v[4] = A[2] + A[6], v[5] = A[5] + A[7];
    v[6] = A[1] - A[3], v[7] = A[2] - A[6], v[8] = A[5] - A[7];
}

// The linear part of the model at one time: 2 B = f2(Ca) 2 S + 2 W - k I,
// row-major, k = f1 / tau_d, so that f2 (S M + M S) + W M - M W - k M =
// B M + (B M)^T (S symmetric, W antisymmetric).  ||G||_inf takes the larger of
// |A_ab| and |A_ba| as |S_ab| + |W_ab|; ca is sqrt(3) tau_d / 2, so that
// u = 3 Ca^2 and f2 = f2_0 + u / (2 u + 2).
template <typename C>
struct Flow {
    C b[9];
};
template <bool Safe, typename C>
__device__ __forceinline__ Flow<C> flow_at(const C (&v0)[9], const C (&d)[9], C t, C ca, C f2_0, C k, bool& ok) {
    C v[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) v[j] = fma(t, d[j], v0[j]);
    const C g[6] = {fabs(v[0]), fabs(v[1]), fabs(v[2]), fabs(v[3]) + fabs(v[6]), fabs(v[4]) + fabs(v[7]),
                    fabs(v[5]) + fabs(v[8])};
    const C c = ca * largest(g), u = c * c;
    const C f2 = f2_0 + quotient<Safe, C>(u, fma(C(2), u, C(2)), ok);
    Flow<C> F;
#pragma unroll
    for (int a = 0; a < 3; ++a) F.b[4 * a] = fma(f2, v[a], -k);
    F.b[1] = fma(f2, v[3], v[6]), F.b[3] = fma(f2, v[3], -v[6]);
    F.b[2] = fma(f2, v[4], v[7]), F.b[6] = fma(f2, v[4], -v[7]);
    F.b[5] = fma(f2, v[5], v[8]), F.b[7] = fma(f2, v[5], -v[8]);
    return F;
}

// x y + z w + iso: float64 (bound by the number of instructions) adds iso
// inside the chain, float32 (bound by the chain's length, iso comes last) after it.
template <typename C>
__device__ __forceinline__ C diagonal(C b0, C m0, C b1, C m1, C b2, C m2, C iso) {
    if constexpr (sizeof(C) == 4) return fma(b0, m0, fma(b1, m1, b2 * m2)) + iso;
    else return fma(b0, m0, fma(b1, m1, fma(b2, m2, iso)));
}

// dM/dt = B M + (B M)^T + 3 k III / II I: the diagonal as it is, the other
// entries twice (the factors of two go into the step's coefficients).
template <bool Safe, typename C>
__device__ __forceinline__ Sym<C> rhs(const Sym<C>& M, const Flow<C>& F, C k3, bool& ok) {
    const C* m = M.v;
    const C* b = F.b;
    // cofactors of the first row: III is the expansion along it, II = c0 + m_xx (m_yy + m_zz) - m_xy^2 - m_xz^2
    const C c0 = fma(m[3], m[5], -m[4] * m[4]);
    const C II = fma(-m[2], m[2], fma(-m[1], m[1], fma(m[0], m[3] + m[5], c0)));
    const C u = fma(m[1], m[5], -m[4] * m[2]), v = fma(m[1], m[4], -m[3] * m[2]);
    const C III = fma(m[0], c0, fma(m[2], v, -m[1] * u));
    const C iso = quotient<Safe, C>(k3 * III, II, ok);
    Sym<C> r;
    r.v[0] = diagonal(b[0], m[0], b[1], m[1], b[2], m[2], iso);
    r.v[3] = diagonal(b[3], m[1], b[4], m[3], b[5], m[4], iso);
    r.v[5] = diagonal(b[6], m[2], b[7], m[4], b[8], m[5], iso);
    // 2 (B M)_ab + 2 (B M)_ba
    r.v[1] = fma(b[0], m[1], fma(b[1], m[3], fma(b[2], m[4], fma(b[3], m[0], fma(b[4], m[1], b[5] * m[2])))));
    r.v[2] = fma(b[0], m[2], fma(b[1], m[4], fma(b[2], m[5], fma(b[6], m[0], fma(b[7], m[1], b[8] * m[2])))));
    r.v[4] = fma(b[3], m[2], fma(b[4], m[4], fma(b[5], m[5], fma(b[6], m[1], fma(b[7], m[3], b[8] * m[4])))));
    return r;
}

// m + h k, with k as rhs leaves it.
template <typename C>
__device__ __forceinline__ Sym<C> axpy(const Sym<C>& m, C h, const Sym<C>& k) {
    Sym<C> r;
#pragma unroll
    for (int e = 0; e < 6; ++e) r.v[e] = fma(e == 0 || e == 3 || e == 5 ? h : C(0.5) * h, k.v[e], m.v[e]);
    return r;
}

// M between substeps: float32 keeps what the diagonal's sums round off.  The
// diagonal lies near one, where a substep's rounding is 6e-8, and D of a nearly
// spherical droplet is a small difference of its entries: hundreds of substeps
// left 1e-6 of D, twice as much by chance in one form of the arithmetic as in
// another.  (The other entries are as small as D, and so are their roundings.)
// 16384 trajectories, 250 steps of 10 substeps: D 1.3e-6 -> 2.2e-7 from the
// float64 integrator's, 653 -> 675 us.
template <typename C>
struct State {
    Sym<C> m;
    C lo[3];
    // m += h k, with k as rhs leaves it
    __device__ __forceinline__ void add(C h, const Sym<C>& k) {
        if constexpr (sizeof(C) == 4) {
            const Sym<C> p = axpy(m, h, k);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const int e = a == 0 ? 0 : 2 + a + (a == 2);  // xx, yy, zz
                const C inc = fma(h, k.v[e], lo[a]), s = m.v[e] + inc;
                lo[a] = inc - (s - m.v[e]);  // exact while |inc| <= |m|
                m.v[e] = s;
            }
            m.v[1] = p.v[1], m.v[2] = p.v[2], m.v[4] = p.v[4];
        } else {
            m = axpy(m, h, k);
        }
    }
    __device__ __forceinline__ void entries(double (&out)[6]) const {
#pragma unroll
        for (int e = 0; e < 6; ++e) out[e] = (double)m.v[e];
        if constexpr (sizeof(C) == 4)
#pragma unroll
            for (int a = 0; a < 3; ++a)
                if (isfinite(lo[a])) out[a == 0 ? 0 : 2 + a + (a == 2)] += (double)lo[a];  // (not so where m overflowed)
    }
};

// The substeps of one time step from M and the flow Fs at its start; false
// where a quotient's denominator was out of range.
template <bool Safe, typename C>
__device__ __forceinline__ bool time_step(State<C>& M, Flow<C>& Fs, const C (&v0)[9], const C (&d)[9], C ca, C f2_0, C k,
                                          C h, int substeps) {
    bool ok = true;
    const C k3 = C(3) * k;
    C q = C(0);
#pragma unroll 1
    for (int i = 0; i < substeps; ++i) {
        // A at the middle and end of the substep (linear in t)
        const Flow<C> Fm = flow_at<Safe, C>(v0, d, fma(q, h, C(0.5) * h), ca, f2_0, k, ok);
        q += C(1);
        const Sym<C> k1 = rhs<Safe>(M.m, Fs, k3, ok);
        const Sym<C> k2 = rhs<Safe>(axpy(M.m, C(0.5) * h, k1), Fm, k3, ok);
        const Sym<C> kc = rhs<Safe>(axpy(M.m, C(0.5) * h, k2), Fm, k3, ok);
        Fs = flow_at<Safe, C>(v0, d, q * h, ca, f2_0, k, ok);
        const Sym<C> k4 = rhs<Safe>(axpy(M.m, h, kc), Fs, k3, ok);
        Sym<C> sum;
#pragma unroll
        for (int e = 0; e < 6; ++e) sum.v[e] = fma(C(2), k2.v[e] + kc.v[e], k1.v[e]) + k4.v[e];
        M.add(h / C(6), sum);
    }
    return ok;
}

template <typename C>
__device__ __forceinline__ double deformation(const State<C>& M) {
    double m[6];
    M.entries(m);
    return lbmgb::deformation_of(m);
}

template <typename C>
__device__ __forceinline__ void store_entries(const State<C>& M, double* out) {
    double m[6];
    M.entries(m);
#pragma unroll
    for (int e = 0; e < 6; ++e) out[e] = m[e];
}

// The substeps from row to row of A with the rows in gradient form: v0 is the
// row before, v1 the row after.
template <typename C>
__device__ __forceinline__ void advance(State<C>& M, Flow<C>& Fs, C (&v0)[9], const C (&v1)[9], C ca, C f2_0, C kf, C h,
                                        int substeps) {
    C d[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) d[j] = v1[j] - v0[j];
    const State<C> M0 = M;
    const Flow<C> F0 = Fs;
    if (!time_step<false>(M, Fs, v0, d, ca, f2_0, kf, h, substeps)) {
        M = M0;
        Fs = F0;
        time_step<true>(M, Fs, v0, d, ca, f2_0, kf, h, substeps);
    }
#pragma unroll
    for (int j = 0; j < 9; ++j) v0[j] = v1[j];
}
template <typename C>
__device__ __forceinline__ Flow<C> first_flow(const C (&v0)[9], C ca, C f2_0, C kf) {
    C d[9] = {};
    bool ok = true;
    const Flow<C> F = flow_at<false, C>(v0, d, C(0), ca, f2_0, kf, ok);
    return ok ? F : flow_at<true, C>(v0, d, C(0), ca, f2_0, kf, ok);
}
template <typename C>
__device__ __forceinline__ State<C> sphere() {
    return {{{C(1), C(0), C(0), C(1), C(0), C(1)}}, {C(0), C(0), C(0)}};
}

// One warp per CTA, so that few trajectories still spread over the SMs: at
// 16384 trajectories there is less than one warp to a scheduler.  The float64
// form is then bound by the number of FP64 instructions (one per 64 cycles
// and scheduler), the float32 form by its dependent chain.  A stage is one
// B M product (27 multiply-adds), the invariants and one quotient; B is
// formed once per time it is needed at (the middle serves two stages, the end
// is the next substep's start), and the next row of A is loaded a step ahead.
// Measured on GB300, 16384 trajectories: float64, 50 steps of 4 substeps,
// 6912 -> 2085 us against separate S M and W M products formed per stage, the
// plain divide and a Jacobi D (FP64 pipe 93 % busy on the SMs with four
// warps); one warp's float64 chain alone (100 trajectories) takes 1980 us.
constexpr int kMMThreads = 32;
template <typename C>
__global__ void __launch_bounds__(kMMThreads) k_mm_rk4(const double* __restrict__ A, long long T, long long n, C ca,
                                                       C f2_0, C kf, int substeps, int record_every,
                                                       double* __restrict__ D, double* __restrict__ Mout) {
    const long long k = (long long)blockIdx.x * kMMThreads + threadIdx.x;
    if (k >= n) return;
    State<C> M = sphere<C>();
    D[k] = 0.0;
    const C h = C(1) / C(substeps);
    C a[9], v0[9];
    double next[9];
    const double* row = A + k * 9;
#pragma unroll
    for (int j = 0; j < 9; ++j) a[j] = (C)row[j];
    if (T > 1)
#pragma unroll
        for (int j = 0; j < 9; ++j) next[j] = row[n * 9 + j];
    split_gradient(a, v0);
    Flow<C> Fs = first_flow(v0, ca, f2_0, kf);
    int until = record_every;
    long long rec = 0;
    for (long long s = 0; s + 1 < T; ++s) {
        C v1[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) a[j] = (C)next[j];
        split_gradient(a, v1);
        row += n * 9;
        if (s + 2 < T)
#pragma unroll
            for (int j = 0; j < 9; ++j) next[j] = row[n * 9 + j];
        advance(M, Fs, v0, v1, ca, f2_0, kf, h, substeps);
        if (--until == 0) {
            until = record_every;
            D[++rec * n + k] = deformation(M);
        }
    }
    if (Mout) store_entries(M, Mout + k * 6);
}

// The float32 form for no more trajectories than the chip has schedulers for
// their warps.  One warp then has a scheduler for itself, and what it does
// besides the stages is time that nothing hides: the FP64 chain of each D (10
// thousand cycles, as much as 25 substeps) and the conversions of each row.
// So two more warps serve each integrating one through shared memory: a
// feeder that loads, converts and splits the rows of A two ahead, and a
// recorder that turns M into D.  The arithmetic is that of k_mm_rk4.
// 16384 trajectories, 250 steps of 10 substeps, 31 records: 675 us; 655 against 788
// without the serving warps (and 4908 with the stages as in the note above);
// 500 us of it are the substeps, 400 cycles each for some 300 instructions.
//
// Hand-over by named barriers of the two warps' 64 threads: the writer waits
// for "empty" (from the second time on), writes its slot and arrives at
// "full"; the reader waits for "full", copies the slot into registers and
// arrives at "empty" if the slot will be written again.  Both sides count
// rows and records alike, so every wait has its arrival.
constexpr int kMMGroup = 4;  // integrating warps of a full CTA
struct MMSlot {
    float row[9][32];
    float m[9][32];  // M, then the diagonal's low parts
};
__device__ __forceinline__ void pair_sync(int id) {
    __syncwarp();
    asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}
__device__ __forceinline__ void pair_arrive(int id) {
    __syncwarp();
    asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory");
}

__global__ void __launch_bounds__(96 * kMMGroup) k_mm_rk4_served(const double* __restrict__ A, long long T, long long n,
                                                                 float ca, float f2_0, float kf, int substeps,
                                                                 int record_every, double* __restrict__ D,
                                                                 double* __restrict__ Mout) {
    __shared__ MMSlot slots[kMMGroup];
    // warps 0 .. W-1 integrate, W .. 2W-1 feed, 2W .. 3W-1 record; with W = 4 the three of a group share a scheduler
    const int warps = blockDim.x / 32, W = warps / 3;
    const int warp = threadIdx.x / 32, role = warp / W, w = warp % W, lane = threadIdx.x % 32;
    const long long first = ((long long)blockIdx.x * W + w) * 32;
    if (first >= n) return;  // the whole group
    const bool live = first + lane < n;
    const long long k = live ? first + lane : n - 1;
    MMSlot& q = slots[w];
    const int row_full = 4 * w, row_empty = 4 * w + 1, m_full = 4 * w + 2, m_empty = 4 * w + 3;
    const long long records = (T - 1) / record_every;
    if (role == 1) {
        const double* row = A + k * 9;
        double x[9], y[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) x[j] = row[j];
        if (T > 1)
#pragma unroll
            for (int j = 0; j < 9; ++j) y[j] = row[n * 9 + j];
        for (long long s = 0; s < T; ++s) {
            float a[9], v[9];
#pragma unroll
            for (int j = 0; j < 9; ++j) a[j] = (float)x[j];
            split_gradient(a, v);
#pragma unroll
            for (int j = 0; j < 9; ++j) x[j] = y[j];
            if (s + 2 < T)
#pragma unroll
                for (int j = 0; j < 9; ++j) y[j] = row[2 * n * 9 + j];
            if (s + 8 < T) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + 8 * n * 9));
            row += n * 9;
            if (s) pair_sync(row_empty);
#pragma unroll
            for (int j = 0; j < 9; ++j) q.row[j][lane] = v[j];
            pair_arrive(row_full);
        }
    } else if (role == 2) {
        if (live) D[k] = 0.0;
        for (long long rec = 1; rec <= records; ++rec) {
            State<float> M;
            pair_sync(m_full);
#pragma unroll
            for (int e = 0; e < 6; ++e) M.m.v[e] = q.m[e][lane];
#pragma unroll
            for (int a = 0; a < 3; ++a) M.lo[a] = q.m[6 + a][lane];
            if (rec < records) pair_arrive(m_empty);
            const double def = deformation(M);
            if (live) D[rec * n + k] = def;
        }
    } else {
        State<float> M = sphere<float>();
        const float h = 1.f / (float)substeps;
        float v0[9];
        pair_sync(row_full);
#pragma unroll
        for (int j = 0; j < 9; ++j) v0[j] = q.row[j][lane];
        if (T > 1) pair_arrive(row_empty);
        Flow<float> Fs = first_flow(v0, ca, f2_0, kf);
        int until = record_every;
        long long rec = 0;
        for (long long s = 0; s + 1 < T; ++s) {
            float v1[9];
            pair_sync(row_full);
#pragma unroll
            for (int j = 0; j < 9; ++j) v1[j] = q.row[j][lane];
            if (s + 2 < T) pair_arrive(row_empty);
            advance(M, Fs, v0, v1, ca, f2_0, kf, h, substeps);
            if (--until == 0) {
                until = record_every;
                if (rec++) pair_sync(m_empty);
#pragma unroll
                for (int e = 0; e < 6; ++e) q.m[e][lane] = M.m.v[e];
#pragma unroll
                for (int a = 0; a < 3; ++a) q.m[6 + a][lane] = M.lo[a];
                pair_arrive(m_full);
            }
        }
        if (Mout && live) store_entries(M, Mout + k * 6);
    }
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
    const double ca = 0.5 * sqrt(3.0) * tau_d;
    if (precision == LBM_FP64) {
        lbmgb_mm::k_mm_rk4<double><<<blocks, threads, 0, s>>>(A, T, n, ca, f2_0, f1 / tau_d, substeps, record_every, D,
                                                              M);
    } else {
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return LBM_ECUDA;
        // up to one integrating warp per scheduler each is served; above that the warps hide one another's waits, and
        // the served form would hold fewer of them.  One group to a CTA while every group finds an SM of its own.
        const int group = blocks <= (unsigned)sms ? 1 : lbmgb_mm::kMMGroup;
        if (blocks <= (unsigned)(sms * lbmgb_mm::kMMGroup))
            lbmgb_mm::k_mm_rk4_served<<<(blocks + group - 1) / group, 96 * group, 0, s>>>(
                A, T, n, (float)ca, (float)f2_0, (float)(f1 / tau_d), substeps, record_every, D, M);
        else
            lbmgb_mm::k_mm_rk4<float><<<blocks, threads, 0, s>>>(A, T, n, (float)ca, (float)f2_0, (float)(f1 / tau_d),
                                                                 substeps, record_every, D, M);
    }
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ECUDA;
}
