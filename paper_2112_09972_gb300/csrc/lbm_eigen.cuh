// Droplet shape from its second moments: 3x3 symmetric eigen-decomposition
// and the deformation D of Sec. 2, Eq. 4.  Shared by the single-box and the
// batched reductions.  Not part of the C ABI.
#pragma once

#include <cuda_runtime.h>

namespace lbmgb {
namespace {

// Symmetric 3x3 eigen-decomposition by cyclic Jacobi rotations.  a is
// overwritten; on return lam holds the eigenvalues and v the eigenvectors
// (column k of v belongs to lam[k]).
//
// The FP64 pipe of this GPU runs at 1/64 of the float32 rate and a float64
// divide or square root is a chain of a dozen such instructions, so each
// rotation's tangent t comes from float32 (of the entries scaled by the
// trace) and its cosine from a float32 reciprocal square root carried to
// float64 by two Newton steps: c^2 (1 + t^2) = 1 and s = t c to float64
// rounding whatever t is, so every rotation is orthogonal to float64
// rounding, and a t that is off by 1e-7 only leaves 1e-7 of the off-diagonal
// entry for the next sweep.  (With float64 divides and roots the final kernel
// of lbm_deformation took 52 us, one thread's dependent chain.)
__device__ void jacobi3(double a[3][3], double lam[3], double v[3][3]) {
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) v[i][j] = (i == j) ? 1.0 : 0.0;
    for (int sweep = 0; sweep < 64; ++sweep) {
        const double off = fabs(a[0][1]) + fabs(a[0][2]) + fabs(a[1][2]);
        const double scale = fabs(a[0][0]) + fabs(a[1][1]) + fabs(a[2][2]);
        if (off <= 1e-300 || off <= 1e-17 * scale) break;
        // 1 / max(scale, off) to float32 accuracy, as a power of two (exact scaling)
        const double big = scale > off ? scale : off;
        const int ex = ((__double2hiint(big) >> 20) & 0x7ff) - 1023;
        const double unit = __hiloint2double((1023 - (ex < 1000 ? (ex > -1000 ? ex : -1000) : 1000)) << 20, 0);
#pragma unroll
        for (int pq = 0; pq < 3; ++pq) {
            const int p = pq < 2 ? 0 : 1, q = pq == 0 ? 1 : 2, r = 3 - p - q;
            const double apq = a[p][q], app = a[p][p], aqq = a[q][q];
            // tan of the angle that annihilates a[p][q]: t = sgn(d) 2 a_pq / (|d| + hypot(d, 2 a_pq)), d = a_qq - a_pp
            const float d = (float)((aqq - app) * unit), o = (float)(2.0 * apq * unit);
            const float h = fabsf(d) + sqrtf(fmaf(d, d, o * o));
            if (!(h > 0.f)) continue;  // both below float32's range of the scale: nothing to rotate
            const float tf = copysignf(1.f, d) * (o / h);
            const double t = (double)tf, n = fma(t, t, 1.0);
            double c = (double)rsqrtf(fmaf(tf, tf, 1.f));
            c *= fma(-0.5 * n * c, c, 1.5);
            c *= fma(-0.5 * n * c, c, 1.5);
            const double s = t * c;
            // A <- J^T A J
            const double x = fma(c, app, -s * apq), y = fma(c, apq, -s * aqq);
            const double z = fma(s, app, c * apq), w = fma(s, apq, c * aqq);
            a[p][p] = fma(c, x, -s * y);
            a[q][q] = fma(s, z, c * w);
            a[p][q] = a[q][p] = fma(s, x, c * y);
            const double apr = a[p][r], aqr = a[q][r];
            a[p][r] = a[r][p] = fma(c, apr, -s * aqr);
            a[q][r] = a[r][q] = fma(s, apr, c * aqr);
#pragma unroll
            for (int k = 0; k < 3; ++k) {  // V <- V J
                const double vkp = v[k][p], vkq = v[k][q];
                v[k][p] = fma(c, vkp, -s * vkq);
                v[k][q] = fma(s, vkp, c * vkq);
            }
        }
    }
    for (int k = 0; k < 3; ++k) lam[k] = a[k][k];
}

// D = (sqrt(l1) - sqrt(l3)) / (sqrt(l1) + sqrt(l3)) of the largest and
// smallest eigenvalue of the symmetric matrix m = (xx, xy, xz, yy, yz, zz),
// eigenvalues below zero taken as zero (Eq. 4).
__device__ __noinline__ double deformation_jacobi(const double (&m)[6]) {
    double a[3][3] = {{m[0], m[1], m[2]}, {m[1], m[3], m[4]}, {m[2], m[4], m[5]}};
    double lam[3], v[3][3];
    jacobi3(a, lam, v);
    const double hi = sqrt(fmax(fmax(lam[0], fmax(lam[1], lam[2])), 0.0));
    const double lo = sqrt(fmax(fmin(lam[0], fmin(lam[1], lam[2])), 0.0));
    return hi + lo > 0.0 ? (hi - lo) / (hi + lo) : 0.0;
}

// 1 / sqrt(a) and 1 / a in float64 from float32 seeds (a within float32's range).
__device__ __forceinline__ double rsqrt64(double a) {
    double y = (double)rsqrtf((float)a);
    y = fma(0.5 * y, fma(-a * y, y, 1.0), y);
    return fma(0.5 * y, fma(-a * y, y, 1.0), y);
}
__device__ __forceinline__ double rcp64(double a) {
    double y = (double)__frcp_rn((float)a);
    y = fma(y, fma(-a, y, 1.0), y);
    return fma(y, fma(-a, y, 1.0), y);
}

// The same D for the conformation tensors of the surrogate and of the
// Maffettone-Minale model, one per thread.  The FP64 pipe bounds these
// kernels, so instead of Jacobi sweeps (about 300 FP64 instructions) the two
// outer eigenvalues q + p x are the outer roots of x^3 - 3 x = 2 r (q the mean
// eigenvalue, p^2 = |m - q|^2 / 6, 2 r = det((m - q) / p)): x = 2 cos(.) in
// float32, then three Newton steps whose slope's reciprocal is float32,
// about 90 FP64 instructions.  Near a double root (|r| within 1e-4 of 1: the
// roots' error is then amplified above 1e-13), near a sphere, for eigenvalues
// that are not well above zero and outside float32's range, Jacobi decides.
__device__ __forceinline__ double deformation_of(const double (&m)[6]) {
    const double q = (m[0] + m[3] + m[5]) * (1.0 / 3.0);
    const double a = m[0] - q, b = m[3] - q, c = m[5] - q;
    const double off2 = fma(m[1], m[1], fma(m[2], m[2], m[4] * m[4]));
    const double p2 = fma(a, a, fma(b, b, fma(c, c, 2.0 * off2))) * (1.0 / 6.0);
    const float qf = (float)q, p2f = (float)p2;
    if (qf > 1e-12f && qf < 1e12f && p2f > 1e-10f * qf * qf && p2f < 0.2f * qf * qf) {
        const double ip = rsqrt64(p2);
        const double p = p2 * ip;
        // 2 r = det(m - q) / p^3
        const double det = fma(a, fma(b, c, -m[4] * m[4]),
                               fma(m[1], fma(m[4], m[2], -m[1] * c), m[2] * fma(m[1], m[4], -b * m[2])));
        const double r2 = det * ip * ip * ip;
        const float rf = 0.5f * (float)r2;
        if (fabsf(rf) < 1.f - 1e-4f) {
            const float phi = acosf(rf) * (1.f / 3.f);
            double x[2] = {(double)(2.f * cosf(phi)), (double)(2.f * cosf(phi + 2.0943951f))};
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int it = 0; it < 3; ++it) {
                    const double xx = x[e] * x[e];
                    const double f = fma(x[e], xx - 3.0, -r2);
                    const float slope = 3.f * ((float)xx - 1.f);
                    x[e] = fma(-f, (double)__frcp_rn(slope), x[e]);
                }
            const double l1 = fma(p, x[0], q), l3 = fma(p, x[1], q);
            if (l3 > 1e-3 * q) {
                const double s1 = l1 * rsqrt64(l1), s3 = l3 * rsqrt64(l3);
                return (s1 - s3) * rcp64(s1 + s3);
            }
        }
    }
    return deformation_jacobi(m);
}

// From the ten moments m: the moments, D, axes (axes[3*a + k]), eigenvalues
// and centre of mass into result[0..25] (the layout of lbm_deformation).
__device__ void deformation_from_moments(const double (&m)[10], double* __restrict__ result) {
    for (int k = 0; k < 10; ++k) result[k] = m[k];
    const double mass = m[0];
    const double c[3] = {m[1] / mass, m[2] / mass, m[3] / mass};
    double I[3][3];
    I[0][0] = m[4] / mass - c[0] * c[0];
    I[0][1] = I[1][0] = m[5] / mass - c[0] * c[1];
    I[0][2] = I[2][0] = m[6] / mass - c[0] * c[2];
    I[1][1] = m[7] / mass - c[1] * c[1];
    I[1][2] = I[2][1] = m[8] / mass - c[1] * c[2];
    I[2][2] = m[9] / mass - c[2] * c[2];
    double lam[3], v[3][3];
    jacobi3(I, lam, v);
    // order by decreasing eigenvalue
    int ord[3] = {0, 1, 2};
    for (int i = 0; i < 3; ++i)
        for (int j = i + 1; j < 3; ++j)
            if (lam[ord[j]] > lam[ord[i]]) { const int tmp = ord[i]; ord[i] = ord[j]; ord[j] = tmp; }
    for (int k = 0; k < 3; ++k) {
        const int col = ord[k];
        int big = 0;
        for (int a = 1; a < 3; ++a)
            if (fabs(v[a][col]) > fabs(v[big][col])) big = a;
        const double sgn = v[big][col] < 0.0 ? -1.0 : 1.0;
        for (int a = 0; a < 3; ++a) result[11 + 3 * a + k] = sgn * v[a][col];
        result[20 + k] = lam[col];
        result[23 + k] = c[k];
    }
    const double a1 = sqrt(fmax(lam[ord[0]], 0.0)), a3 = sqrt(fmax(lam[ord[2]], 0.0));
    result[10] = (a1 - a3) / (a1 + a3);
}

}  // namespace
}  // namespace lbmgb
