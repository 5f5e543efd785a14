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

// float64 to float32 (truncated) and back by shifts, for magnitudes between
// 2^-100 and 2^100: conversions to and from 64 bits run on the FP64 pipe, at
// its rate of one warp instruction per 16 cycles and SM.
__device__ __forceinline__ float narrow(double d) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    return __uint_as_float((hi & 0x80000000u) | __funnelshift_l(lo, (hi & 0x7fffffffu) - (896u << 20), 3));
}
__device__ __forceinline__ double widen(float f) {
    const unsigned b = __float_as_uint(f);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}
// 1 / d from the reciprocal unit, to 23 bits.
__device__ __forceinline__ float rcp_seed(float d) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(d));
    return y;
}

// 1 / sqrt(a) and 1 / a in float64 from float32 seeds (a within 2^+-100):
// with e = 1 - a y^2 or 1 - a y of the seed y (1e-7), the series of
// (1 - e)^-1/2 and (1 - e)^-1 to e^2 leaves e^3.
__device__ __forceinline__ double rsqrt64(double a) {
    const double y = widen(rsqrtf(narrow(a))), e = fma(-a * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double rcp64(double a) {
    const double y = widen(rcp_seed(narrow(a))), e = fma(-a, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// One Newton step of x^3 - 3 x = r2 near an outer root (1 < |x|) with a
// float32 slope.
__device__ __forceinline__ double root_step(double x, double r2) {
    const double xx = x * x;
    return fma(-fma(x, xx - 3.0, -r2), widen(rcp_seed(3.f * (narrow(xx) - 1.f))), x);
}

// Half the distance of the two close eigenvalues of the traceless symmetric
// N = (a, n1, n2; n1, b, n4; n2, n4, c) whose third one is mu, close to 2 or
// -2: N is projected on the plane normal to mu's eigenvector, so
// the error is that of N's entries however close the two are, where a root of
// the characteristic polynomial would lose half the digits.
__device__ __forceinline__ double half_gap(double a, double b, double c, double n1, double n2, double n4, double mu) {
    // N - mu is -+3 (1 - v v^T): the smallest diagonal entry names v's
    // largest component, which the permutation makes the third
    const double da = fabs(a - mu), db = fabs(b - mu), dc = fabs(c - mu);
    if (da < dc && da <= db) {
        double t = a; a = c; c = t;
        t = n1; n1 = n4; n4 = t;
    } else if (db < dc) {
        double t = b; b = c; c = t;
        t = n1; n1 = n2; n2 = t;
    }
    const double ea = a - mu, eb = b - mu;
    double x = fma(n1, n4, -n2 * eb), y = fma(n1, n2, -n4 * ea), z = fma(ea, eb, -n1 * n1);
    const double iv = rsqrt64(fma(x, x, fma(y, y, z * z)));
    x *= iv;
    y *= iv;
    z *= iv;  // positive: 9 v_z^2 before
    // orthonormal u, w normal to (x, y, z)
    const double g = -rcp64(1.0 + z), h = x * y * g;
    const double u0 = fma(x * x, g, 1.0), w1 = fma(y * y, g, 1.0);
    const double nu0 = fma(a, u0, fma(n1, h, -n2 * x)), nu1 = fma(n1, u0, fma(b, h, -n4 * x)),
                 nu2 = fma(n2, u0, fma(n4, h, -c * x));
    const double nw0 = fma(a, h, fma(n1, w1, -n2 * y)), nw1 = fma(n1, h, fma(b, w1, -n4 * y)),
                 nw2 = fma(n2, h, fma(n4, w1, -c * y));
    const double uu = fma(u0, nu0, fma(h, nu1, -x * nu2)), ww = fma(h, nw0, fma(w1, nw1, -y * nw2));
    const double uw = fma(h, nu0, fma(w1, nu1, -y * nu2)), d = 0.5 * (uu - ww);
    return sqrt(fma(d, d, uw * uw));
}

// The same D for the conformation tensors of the surrogate and of the
// Maffettone-Minale model, one per thread.  The FP64 pipe bounds these
// kernels, so instead of Jacobi sweeps (about 300 FP64 instructions) the two
// outer eigenvalues q + p x are the outer roots of x^3 - 3 x = 2 r (q the mean
// eigenvalue, p^2 = |m - q|^2 / 6, 2 r = det((m - q) / p)): x = 2 cos(.) in
// float32, then two Newton steps whose slope's reciprocal is float32 (1e-7 ->
// 1e-13 -> rounding); and sqrt(l1), sqrt(l3) enter as their product alone,
//   D = (l1 - l3) / (l1 + l3 + 2 sqrt(l1 l3)),
// about 60 FP64 instructions.  m - q is formed from the differences of the
// diagonal, which keeps its digits near a sphere.  Near a double root (r
// within 1e-3 of +-1) the simple root and half_gap give the eigenvalues.
// For a sphere (|m - q| below 1e-10 q), for eigenvalues that are not well
// above zero and outside float32's range Jacobi decides.
__device__ __forceinline__ double deformation_of(const double (&m)[6]) {
    const double third = 1.0 / 3.0, q = (m[0] + m[3] + m[5]) * third;
    const double d0 = m[0] - m[3], d1 = m[3] - m[5];
    const double a = fma(2.0, d0, d1) * third, b = (d1 - d0) * third, c = -a - b;
    const double off2 = fma(m[1], m[1], fma(m[2], m[2], m[4] * m[4]));
    const double p2 = fma(a, a, fma(b, b, fma(c, c, 2.0 * off2))) * (1.0 / 6.0);
    const float qf = (float)q, p2f = (float)p2;
    if (qf > 1e-12f && qf < 1e12f && p2f > 1e-30f && p2f > 1e-20f * qf * qf && p2f < 0.2f * qf * qf) {
        const double ip = rsqrt64(p2);
        const double p = p2 * ip;
        // 2 r = det(m - q) / p^3
        const double det = fma(a, fma(b, c, -m[4] * m[4]),
                               fma(m[1], fma(m[4], m[2], -m[1] * c), m[2] * fma(m[1], m[4], -b * m[2])));
        const double r2 = det * ip * ip * ip;
        // r = cos 3 phi, from its distance to the nearer end
        const float ef = fmaxf((float)fma(-0.5, fabs(r2), 1.0), 0.f);
        double l1, l3;
        if (ef > 1e-3f) {
            const float th = (2.f / 3.f) * asinf(sqrtf(0.5f * ef));
            const float phi = r2 >= 0.0 ? th : 1.04719755f - th;
            const double x1 = widen(2.f * cosf(phi)), x3 = widen(2.f * cosf(phi + 2.0943951f));
            l1 = p * root_step(root_step(x1, r2), r2);
            l3 = p * root_step(root_step(x3, r2), r2);
        } else {
            // the root near +-2, from 2 - 2 (1 - |r|) / 9
            const double x = copysign(2.0 - (2.0 / 9.0) * (double)ef, r2);
            const double xs = root_step(root_step(x, r2), r2), mu = p * xs;
            const double gap = p * half_gap(a * ip, b * ip, c * ip, m[1] * ip, m[2] * ip, m[4] * ip, xs);
            l1 = r2 >= 0.0 ? mu : fma(-0.5, mu, gap);
            l3 = r2 >= 0.0 ? fma(-0.5, mu, -gap) : mu;
        }
        const double n = l1 - l3;
        l1 += q;
        l3 += q;
        if (l3 > 1e-3 * q) {
            const double g = l1 * l3;
            return n * rcp64(fma(2.0 * g, rsqrt64(g), l1 + l3));
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
