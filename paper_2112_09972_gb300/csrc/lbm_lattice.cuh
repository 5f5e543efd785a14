// Device-side D3Q19 lattice helpers shared by the CUDA translation units of
// the library (not by the CPU oracle).
#pragma once

#include <cuda_runtime.h>

namespace lbmgb {
namespace {

// D3Q19 velocities in the order documented in lbm.h: direction 2k is the
// opposite of direction 2k-1.  Every loop over directions is unrolled, so
// these fold to immediates.
__host__ __device__ __forceinline__ constexpr int cx_(int i) {
    constexpr int t[19] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
    return t[i];
}
__host__ __device__ __forceinline__ constexpr int cy_(int i) {
    constexpr int t[19] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
    return t[i];
}
__host__ __device__ __forceinline__ constexpr int cz_(int i) {
    constexpr int t[19] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};
    return t[i];
}

template <typename C>
__host__ __device__ __forceinline__ constexpr C wgt(int i) {
    return i == 0 ? C(1) / C(3) : (i < 7 ? C(1) / C(18) : C(1) / C(36));
}

// c_i . u as at most two additions: a product with a zero component is not
// dropped by the compiler (it would not be zero for infinities), and three
// such terms per direction were a tenth of a node's instructions.
template <typename C>
__device__ __forceinline__ C dot_c(int i, C ux, C uy, C uz) {
    C v = C(0);
    bool any = false;
    if (cx_(i)) {
        v = cx_(i) > 0 ? ux : -ux;
        any = true;
    }
    if (cy_(i)) {
        v = any ? (cy_(i) > 0 ? v + uy : v - uy) : (cy_(i) > 0 ? uy : -uy);
        any = true;
    }
    if (cz_(i)) v = any ? (cz_(i) > 0 ? v + uz : v - uz) : (cz_(i) > 0 ? uz : -uz);
    return v;
}

// Eq. 8 for weight w and cu = c_i . u.
template <typename C>
__device__ __forceinline__ C feq_of(C rho, C w, C cu, C u2x) {
    return rho * w * (C(1) + C(3) * cu + C(4.5) * cu * cu - u2x);
}

// Eq. 8 with u2x = 1.5 |u|^2 precomputed.
template <typename C>
__device__ __forceinline__ C feq(int i, C rho, C ux, C uy, C uz, C u2x) {
    return feq_of<C>(rho, wgt<C>(i), dot_c<C>(i, ux, uy, uz), u2x);
}

// MRT collision: row k of the D3Q19 moment basis of d'Humieres et al. (2002)
// at direction i (density, energy, energy square, momentum and energy flux,
// stress and its partners, third-order moments), its squared norm, and the
// relaxation rate of moment k: 1/tau for density, momentum and stress (the
// velocity-shift forcing and Eq. 10), r[0..4] = s_e, s_eps, s_q, s_pi, s_m
// for the rest.
__host__ __device__ __forceinline__ constexpr int mrt_row(int k, int i) {
    const int cx = cx_(i), cy = cy_(i), cz = cz_(i);
    const int c2 = cx * cx + cy * cy + cz * cz;
    switch (k) {
        case 0: return 1;
        case 1: return 19 * c2 - 30;
        case 2: return (21 * c2 * c2 - 53 * c2 + 24) / 2;
        case 3: return cx;
        case 4: return (5 * c2 - 9) * cx;
        case 5: return cy;
        case 6: return (5 * c2 - 9) * cy;
        case 7: return cz;
        case 8: return (5 * c2 - 9) * cz;
        case 9: return 3 * cx * cx - c2;
        case 10: return (3 * c2 - 5) * (3 * cx * cx - c2);
        case 11: return cy * cy - cz * cz;
        case 12: return (3 * c2 - 5) * (cy * cy - cz * cz);
        case 13: return cx * cy;
        case 14: return cy * cz;
        case 15: return cx * cz;
        case 16: return (cy * cy - cz * cz) * cx;
        case 17: return (cz * cz - cx * cx) * cy;
        default: return (cx * cx - cy * cy) * cz;
    }
}
__host__ __device__ __forceinline__ constexpr int mrt_norm(int k) {
    int n = 0;
    for (int i = 0; i < 19; ++i) n += mrt_row(k, i) * mrt_row(k, i);
    return n;
}
// Group g[] / o[] of direction pair k = (i - 1) / 2: which accumulator of
// mrt_free the sum of the pair's deviations goes to (even: 0 the rest
// direction, 1..3 the axes x, y, z, 4..6 the edges xy, xz, yz).
__host__ __device__ __forceinline__ constexpr int mrt_group(int i) {
    return i == 0 ? 0 : (i < 7 ? 1 + (i - 1) / 2 : 4 + (i - 7) / 4);
}

// The part of M^-1 S M dev that the five free rates add to BGK at 1 / tau.
// All rows of M whose rate is 1 / tau (density, momentum, stress) act as BGK,
// so with D = diag(1 / |M_k|^2)
//   M^-1 S M dev = dev / tau + M^T D (S - 1 / tau) M dev,
// where only the ten rows with a free rate remain.  Each is even or odd in c,
// so it needs the sums or differences of opposite pairs only, and the even
// ones (energy 1, its square 2, stress partners 10 and 12) are equal within
// the axis and edge groups:
//   in   g[7]  sums of dev: rest; pairs of x, y, z; of xy, xz, yz (two pairs each)
//        o[9]  differences dev_i - dev_{i+1}: x, y, z; then the pair sums that
//              the fluxes take: xy and xz along x, xy and yz along y, xz and yz along z
//   out  ce[7] the even part for one direction of each group
//        co[9] the odd part along c: the axes x, y, z; then per unit of c_x on
//              xy and xz edges, of c_y on xy and yz, of c_z on xz and yz
// About 75 operations a component where the 19 x 19 products take over 500
// (float64: 32^3 60 us per step in two passes).
template <typename C>
__device__ __forceinline__ void mrt_free(const C (&g)[7], const C (&o)[9], C inv_tau, const C (&r)[5], C (&ce)[7],
                                         C (&co)[9]) {
    const C A = g[1] + g[2] + g[3], E = g[4] + g[5] + g[6];
    const C e = (r[0] - inv_tau) * C(1.0 / mrt_norm(1)) * (C(8) * E - C(11) * A - C(30) * g[0]);
    const C q = (r[1] - inv_tau) * C(1.0 / mrt_norm(2)) * (E - C(4) * A + C(12) * g[0]);
    const C p = (r[3] - inv_tau) * C(1.0 / mrt_norm(10)) *
                (C(2) * (g[2] + g[3]) - C(4) * g[1] + (g[4] + g[5]) - C(2) * g[6]);
    const C w = (r[3] - inv_tau) * C(1.0 / mrt_norm(12)) * (C(2) * (g[3] - g[2]) + (g[4] - g[5]));
    ce[0] = C(12) * q - C(30) * e;
    const C a = -C(11) * e - C(4) * q, b = C(8) * e + q;
    ce[1] = a - C(4) * p;
    ce[2] = a + C(2) * p - C(2) * w;
    ce[3] = a + C(2) * p + C(2) * w;
    ce[4] = b + p + w;
    ce[5] = b + p - w;
    ce[6] = b - C(2) * p;
    const C kq = (r[2] - inv_tau) * C(1.0 / mrt_norm(4)), km = (r[4] - inv_tau) * C(1.0 / mrt_norm(16));
    const C qx = kq * (o[3] + o[4] - C(4) * o[0]), mx = km * (o[3] - o[4]);
    const C qy = kq * (o[5] + o[6] - C(4) * o[1]), my = km * (o[6] - o[5]);
    const C qz = kq * (o[7] + o[8] - C(4) * o[2]), mz = km * (o[7] - o[8]);
    co[0] = -C(4) * qx;
    co[1] = -C(4) * qy;
    co[2] = -C(4) * qz;
    co[3] = qx + mx;  // c_x on xy
    co[4] = qx - mx;  // c_x on xz
    co[5] = qy - my;  // c_y on xy
    co[6] = qy + my;  // c_y on yz
    co[7] = qz + mz;  // c_z on xz
    co[8] = qz - mz;  // c_z on yz
}
// Adds direction pair (i, i + 1)'s deviations to the groups of mrt_free.
template <typename C>
__device__ __forceinline__ void mrt_gather(int i, C dp, C dm, C (&g)[7], C (&o)[9]) {
    g[mrt_group(i)] += dp + dm;
    const C d = dp - dm;
    if (i < 7) {
        o[(i - 1) / 2] += d;
        return;
    }
    if (cx_(i)) o[cy_(i) ? 3 : 4] += d;  // c_x = +1 on every edge pair's first direction that has one
    if (cy_(i)) o[cx_(i) ? 5 : 6] += cy_(i) > 0 ? d : -d;
    if (cz_(i)) o[cx_(i) ? 7 : 8] += cz_(i) > 0 ? d : -d;
}
// The odd part for direction i of a pair (the opposite direction has its negative).
template <typename C>
__device__ __forceinline__ C mrt_odd(int i, const C (&co)[9]) {
    if (i < 7) return co[(i - 1) / 2];
    C v = C(0);
    if (cx_(i)) v = co[cy_(i) ? 3 : 4];
    if (cy_(i)) {
        const C t = co[cx_(i) ? 5 : 6];
        v = cx_(i) ? (cy_(i) > 0 ? v + t : v - t) : t;
    }
    if (cz_(i)) {
        const C t = co[cx_(i) ? 7 : 8];
        v = cz_(i) > 0 ? v + t : v - t;
    }
    return v;
}

// out_i = f_i - (M^-1 S M dev)_i with dev = f - f_eq.
template <typename C>
__device__ __forceinline__ void mrt_relax(const C (&f)[19], const C (&dev)[19], C inv_tau, const C (&r)[5],
                                          C (&out)[19]) {
    C g[7] = {dev[0], C(0), C(0), C(0), C(0), C(0), C(0)};
    C o[9] = {C(0), C(0), C(0), C(0), C(0), C(0), C(0), C(0), C(0)};
#pragma unroll
    for (int i = 1; i < 19; i += 2) mrt_gather<C>(i, dev[i], dev[i + 1], g, o);
    C ce[7], co[9];
    mrt_free<C>(g, o, inv_tau, r, ce, co);
    out[0] = f[0] - inv_tau * dev[0] - ce[0];
#pragma unroll
    for (int i = 1; i < 19; i += 2) {
        const C e = ce[mrt_group(i)], d = mrt_odd<C>(i, co);
        out[i] = f[i] - inv_tau * dev[i] - (e + d);
        out[i + 1] = f[i + 1] - inv_tau * dev[i + 1] - (e - d);
    }
}

template <typename C>
__device__ __forceinline__ C mrt_rate(int k, C inv_tau, const C (&r)[5]) {
    return (k == 0 || k == 3 || k == 5 || k == 7 || k == 9 || k == 11 || k == 13 || k == 14 || k == 15)
               ? inv_tau
               : (k == 1 ? r[0] : (k == 2 ? r[1] : ((k == 4 || k == 6 || k == 8) ? r[2] : ((k == 10 || k == 12) ? r[3] : r[4]))));
}

// out_i = f_i - sum_k M_ki s_k (M dev)_k / |M_k|^2 with dev = f - f_eq, moment
// by moment.  Float32 and 16-bit storage take this order of operations: the
// other one moves their roundings, and D of a small droplet with them, by as
// much as float32 leaves of it (64 x 88 x 20, R = 3.4, 36 steps: 6e-7 from the
// 64-bit result here, 4e-6 with mrt_relax).
template <typename C>
__device__ __forceinline__ void mrt_relax_full(const C (&f)[19], const C (&dev)[19], C inv_tau, const C (&r)[5],
                                          C (&out)[19]) {
    C rel[19];
#pragma unroll
    for (int k = 0; k < 19; ++k) {
        C mk = C(0);
#pragma unroll
        for (int i = 0; i < 19; ++i)
            if (mrt_row(k, i) != 0) mk += C(mrt_row(k, i)) * dev[i];
        rel[k] = mrt_rate<C>(k, inv_tau, r) * mk / C(mrt_norm(k));
    }
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        C back = C(0);
#pragma unroll
        for (int k = 0; k < 19; ++k)
            if (mrt_row(k, i) != 0) back += C(mrt_row(k, i)) * rel[k];
        out[i] = f[i] - back;
    }
}

__device__ __forceinline__ int wrap(int a, int n) {
    a = a < 0 ? a + n : a;
    return a >= n ? a - n : a;
}

// Sum of 19 values as f0 + sum over opposite pairs.
template <typename C>
__device__ __forceinline__ C sum19(const C (&f)[19]) {
    C s = f[0];
#pragma unroll
    for (int i = 1; i < 19; i += 2) s += f[i] + f[i + 1];
    return s;
}

}  // namespace
}  // namespace lbmgb
