// Node-level device code of the float32 and 16-bit storage kernels, shared by
// the row-tiled cluster kernels (lbm_fast.cu) and the two-pass kernels
// (lbm_flat32.cu): model constants, the reads and writes of a node's
// populations, and its collision (Sec. 2, Eqs. 6-10 of Milan et al.,
// arXiv:2112.09972).  Not part of the C ABI.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>
#include <utility>

#include "lbm_dev.cuh"
#include "lbm_internal.h"
#include "lbm_lattice.cuh"

namespace lbmgb {
namespace {

struct FastModel {
    float inv_tau[2], tau[2], G, rho_b[2];
    float omit[2];  // 1 - 1/tau
    float sh[2];    // -G tau: the velocity shift tau_s F^s / rho_s per unit of the other component's force sum
    float mrt[5];   // MRT free rates (s_e, s_eps, s_q, s_pi, s_m) when the kernel relaxes moments
};

FastModel fast_model(const Model& m) {
    FastModel fm;
    for (int q = 0; q < 2; ++q) {
        fm.inv_tau[q] = (float)(1.0 / m.tau[q]);
        fm.tau[q] = (float)m.tau[q];
        fm.rho_b[q] = (float)m.rho_b[q];
        fm.omit[q] = (float)(1.0 - 1.0 / m.tau[q]);
        fm.sh[q] = (float)(-m.G * m.tau[q]);
    }
    fm.G = (float)m.G;
    for (int k = 0; k < 5; ++k) fm.mrt[k] = (float)m.mrt_rates[k];
    return fm;
}

// Compile-time loop: f(std::integral_constant<int, 0>) ... f(..., N - 1).
template <typename F, int... I>
__device__ __forceinline__ void sfor_(F& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void sfor(F&& f) {
    sfor_(f, std::make_integer_sequence<int, N>{});
}

// Pairs {A, B} of the two components in packed float32 arithmetic: one
// instruction adds or multiplies both, each half rounded as the scalar
// instruction rounds it, so the results are the scalar ones.  The 16-bit
// forms use it: their kernels issue on 58 % of the cycles, the words already
// hold both components, and the arithmetic instructions of a node update
// halve (256^3 per step: binary16 733 -> 689 us, bfloat16 768 -> 707).  Float32
// storage does not: its staged kernel carries 76 populations in registers,
// which the pairing made spill (128^3 133 -> 153 us).
__device__ __forceinline__ float2 pair(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    float2 r;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long&>(r))
        : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
    return r;
}
// c_i . u of both components (dot_c).
__device__ __forceinline__ float2 dot_c2(int i, float2 ux, float2 uy, float2 uz) {
    float2 v = both(0.f);
    bool any = false;
    if (cx_(i)) {
        v = cx_(i) > 0 ? ux : pair(-ux.x, -ux.y);
        any = true;
    }
    if (cy_(i)) {
        v = any ? (cy_(i) > 0 ? add2(v, uy) : sub2(v, uy)) : (cy_(i) > 0 ? uy : pair(-uy.x, -uy.y));
        any = true;
    }
    if (cz_(i)) v = any ? (cz_(i) > 0 ? add2(v, uz) : sub2(v, uz)) : (cz_(i) > 0 ? uz : pair(-uz.x, -uz.y));
    return v;
}

// Global loads and stores at a pointer plus an immediate byte offset.  The
// first read of a plane keeps its lines in L2 (evict_last policy) for the
// second read one plane later, which marks them last-use; the written state
// is streamed out.  The populations read are never written by the kernel, so
// the loads may be scheduled freely.
template <int OFF, bool NC = true>
__device__ __forceinline__ float ld_keep(const void* p, unsigned long long pol) {
    float v;
    if constexpr (!NC) asm("ld.global.L2::cache_hint.f32 %0, [%1+%3], %2;" : "=f"(v) : "l"(p), "l"(pol), "n"(OFF));
    else asm("ld.global.nc.L2::cache_hint.f32 %0, [%1+%3], %2;" : "=f"(v) : "l"(p), "l"(pol), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ float ld_last(const void* p) {
    float v;
    asm("ld.global.lu.f32 %0, [%1+%2];" : "=f"(v) : "l"(p), "n"(OFF));
    return v;
}
template <int OFF, bool NC = true>
__device__ __forceinline__ unsigned ld_keep_u32(const void* p, unsigned long long pol) {
    unsigned v;
    if constexpr (!NC) asm("ld.global.L2::cache_hint.b32 %0, [%1+%3], %2;" : "=r"(v) : "l"(p), "l"(pol), "n"(OFF));
    else asm("ld.global.nc.L2::cache_hint.b32 %0, [%1+%3], %2;" : "=r"(v) : "l"(p), "l"(pol), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ unsigned ld_last_u32(const void* p) {
    unsigned v;
    asm("ld.global.lu.b32 %0, [%1+%2];" : "=r"(v) : "l"(p), "n"(OFF));
    return v;
}
__device__ __forceinline__ float4 ld_keep_f4(const void* p, unsigned long long pol) {
    float4 v;
    asm("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ float4 ld_last_f4(const void* p) {
    float4 v;
    asm("ld.global.lu.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
template <int OFF>
__device__ __forceinline__ void st_cs(void* p, float v) {
    asm volatile("st.global.cs.f32 [%0+%2], %1;" ::"l"(p), "f"(v), "n"(OFF));
}
template <int OFF>
__device__ __forceinline__ void st_cs_u32(void* p, unsigned v) {
    asm volatile("st.global.cs.b32 [%0+%2], %1;" ::"l"(p), "r"(v), "n"(OFF));
}
__device__ __forceinline__ void st_cs_f4(void* p, float4 v) {
    asm volatile("st.global.cs.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
}

// Compile-time geometry of the row-interleaved layout for row width TX (the
// values make_layout computes): entries before x = 0, entries per population
// row and layout units per row block (elements of 4 bytes for float32, units
// of 2 bytes for deviations).
template <int TX, typename ST>
struct RowGeo;
template <int TX>
struct RowGeo<TX, float> {
    static constexpr int X0 = 8, PITCH = TX + 16, ROW = 38 * PITCH;
};
template <int TX, typename T>
struct RowGeo<TX, Dev<T>> {
    static constexpr int X0 = 16, PITCH = TX + 32, ROW = 44 * PITCH;
};

// Storage-specific reads and writes of the row kernels.  A node's accesses
// go through its pointer `base` (the node in plane -1) and, per plane p, the
// three pointers P3 of planes p - 1, p, p + 1.
template <int TX, typename ST>
struct RowIO;

template <int TX>
struct RowIO<TX, float> {
    using G = RowGeo<TX, float>;
    struct P3 {
        const char* m;
        const char* o;
        const char* p;
    };
    using Out = float*;  // element (s = 0, i = 0) of the node in the written plane
    // element (s = 0, i = 0) of node (x, y) in plane -1
    static __device__ __forceinline__ const char* base(const float* src, int x, int y) {
        return reinterpret_cast<const char*>(src + (long long)(y + 1) * G::ROW + G::X0 + x);
    }
    // the same node, component s (the halo threads sum one component each)
    static __device__ __forceinline__ const char* base_c(const float* src, int x, int y, int s) {
        return base(src, x, y) + 4 * s * 19 * G::PITCH;
    }
    static __device__ __forceinline__ P3 planes(const char* b, const Layout& L, int p) {
        const long long pl = 4 * L.plane;
        const char* o = b + (long long)(p + 1) * pl;
        return {o - pl, o, o + pl};
    }
    static __device__ __forceinline__ Out out(float* dst, const Layout& L, int x, int y, int z) {
        return dst + (long long)(z + 1) * L.plane + (long long)(y + 1) * G::ROW + G::X0 + x;
    }
    // byte offset of population (s, i) pulled into the node (it comes from
    // x - c_i, which lies in plane p - c_iz: the pointer src_plane picks)
    template <int S, int I>
    static constexpr int poff() {
        return 4 * ((S * 19 + I) * G::PITCH - cy_(I) * G::ROW - cx_(I));
    }
    template <int I>
    static __device__ __forceinline__ const char* src_plane(const P3& q) {
        return cz_(I) > 0 ? q.m : (cz_(I) < 0 ? q.p : q.o);
    }
    // component S's post-streaming density (first read, kept in L2)
    template <int S, bool NC = true>
    static __device__ __forceinline__ float density(const P3& q, unsigned long long pol) {
        float r = ld_keep<poff<S, 0>(), NC>(q.o, pol);
        sfor<9>([&](auto K) {
            constexpr int i = 2 * decltype(K)::value + 1;
            r += ld_keep<poff<S, i>(), NC>(src_plane<i>(q), pol) +
                 ld_keep<poff<S, i + 1>(), NC>(src_plane<i + 1>(q), pol);
        });
        return r;
    }
    // NC false: the calling warp may have written what it reads
    template <bool NC = true>
    static __device__ __forceinline__ void densities(const P3& q, unsigned long long pol, float& ra, float& rb) {
        ra = density<0, NC>(q, pol);
        rb = density<1, NC>(q, pol);
    }
    // the node's 38 pulled populations (second read, last use); rs: unused
    // in float32 (the deviation forms return the node's rho* there)
    static __device__ __forceinline__ void populations(const P3& q, float (&f)[2][19], float (&rs)[2]) {
        rs[0] = rs[1] = 0.f;
        sfor<19>([&](auto I) {
            constexpr int i = decltype(I)::value;
            f[0][i] = ld_last<poff<0, i>()>(src_plane<i>(q));
            f[1][i] = ld_last<poff<1, i>()>(src_plane<i>(q));
        });
    }
    // one read of the 38 pulled populations and the densities summed from
    // them in the order of density() (the warp-specialised kernel)
    static __device__ __forceinline__ void load_all(const P3& q, float (&f)[2][19], float (&rs)[2], float& ra,
                                                    float& rb) {
        populations(q, f, rs);
        ra = f[0][0];
        rb = f[1][0];
#pragma unroll
        for (int i = 1; i < 19; i += 2) {
            ra += f[0][i] + f[0][i + 1];
            rb += f[1][i] + f[1][i + 1];
        }
    }
    template <int S, int I>
    static __device__ __forceinline__ void store(Out o, float v) {
        st_cs<4 * (S * 19 + I) * G::PITCH>(o, v);
    }
};

// 16-bit deviation storage: per node the float4 block {rho*_A, rho*_B, f*_0A,
// f*_0B} and the 18 words of deviation pairs {A, B}.  The plane pointers
// point at the node's word slot (x0 + x) of its row block; the node's own
// block lies a per-thread constant further (12 (x0 + x) bytes), and the word
// of direction i at the immediate 4 (3 + i) pitch.
template <int TX, typename T>
struct RowIO<TX, Dev<T>> {
    using G = RowGeo<TX, Dev<T>>;
    struct P3 {
        const char* m;
        const char* o;
        const char* p;
        int blk;  // byte offset of the node's float4 block from o
    };
    struct Out {
        unsigned* w;  // word slot of the node in the written plane
        float4* b;    // the node's float4 block
    };
    static __device__ __forceinline__ const char* base(const Dev<T>* src, int x, int y) {
        return reinterpret_cast<const char*>(src) + 2LL * (long long)(y + 1) * G::ROW + 4 * (G::X0 + x);
    }
    static __device__ __forceinline__ P3 planes(const char* b, const Layout& L, int p, int x) {
        const long long pl = 2 * L.plane;
        const char* o = b + (long long)(p + 1) * pl;
        return {o - pl, o, o + pl, 12 * (G::X0 + x)};
    }
    static __device__ __forceinline__ Out out(Dev<T>* dst, const Layout& L, int x, int y, int z) {
        char* o = reinterpret_cast<char*>(dst) + 2LL * ((long long)(z + 1) * L.plane + (long long)(y + 1) * G::ROW) +
                  4 * (G::X0 + x);
        return {reinterpret_cast<unsigned*>(o), reinterpret_cast<float4*>(o + 12 * (G::X0 + x))};
    }
    template <int I>
    static constexpr int woff() {  // byte offset of the word of direction I pulled into the node
        return 4 * (3 + I) * G::PITCH - 2 * cy_(I) * G::ROW - 4 * cx_(I);
    }
    template <int I>
    static __device__ __forceinline__ const char* src_plane(const P3& q) {
        return cz_(I) > 0 ? q.m : (cz_(I) < 0 ? q.p : q.o);
    }
    // sum_i (w_i rho* + d_i) + f*_0 = f*_0 + (1 - w_0) rho* + sum_i d_i, from
    // the node's block o and its pulled words word(integral_constant<int, i>)
    template <typename W>
    static __device__ __forceinline__ void sum_words(const float4& o, W&& word, float& ra, float& rb) {
        float da = 0.f, db = 0.f;
        sfor<9>([&](auto K) {
            constexpr int i = 2 * decltype(K)::value + 1;
            const float2 u = dev_unpack2<T>(word(std::integral_constant<int, i>{}));
            const float2 v = dev_unpack2<T>(word(std::integral_constant<int, i + 1>{}));
            da += u.x + v.x;
            db += u.y + v.y;
        });
        ra = o.z + (1.f - wgt<float>(0)) * o.x + da;
        rb = o.w + (1.f - wgt<float>(0)) * o.y + db;
    }
    template <bool NC = true>
    static __device__ __forceinline__ void densities(const P3& q, unsigned long long pol, float& ra, float& rb) {
        const float4 o = ld_keep_f4(q.o + q.blk, pol);
        sum_words(
            o,
            [&](auto I) {
                constexpr int i = decltype(I)::value;
                return ld_keep_u32<woff<i>(), NC>(src_plane<i>(q), pol);
            },
            ra, rb);
    }
    // The collision's input in deviation form: f[s][0] the rest population,
    // f[s][i >= 1] the pulled deviation d_i (the population is
    // w_i rho*_s + d_i; collide_node folds w_i rho*_s into its constants),
    // rs the node's rho* of both components.
    static __device__ __forceinline__ void populations(const P3& q, float (&f)[2][19], float (&rs)[2]) {
        const float4 o = ld_last_f4(q.o + q.blk);
        f[0][0] = o.z;
        f[1][0] = o.w;
        rs[0] = o.x;
        rs[1] = o.y;
        sfor<18>([&](auto K) {
            constexpr int i = decltype(K)::value + 1;
            const float2 v = dev_unpack2<T>(ld_last_u32<woff<i>()>(src_plane<i>(q)));
            f[0][i] = v.x;
            f[1][i] = v.y;
        });
    }
    // one read of the block and the 18 pulled words: the input of
    // populations() and the densities of densities(), with their arithmetic
    static __device__ __forceinline__ void load_all(const P3& q, float (&f)[2][19], float (&rs)[2], float& ra,
                                                    float& rb) {
        const float4 o = ld_last_f4(q.o + q.blk);
        f[0][0] = o.z;
        f[1][0] = o.w;
        rs[0] = o.x;
        rs[1] = o.y;
        float da = 0.f, db = 0.f;
        sfor<9>([&](auto K) {
            constexpr int i = 2 * decltype(K)::value + 1;
            const float2 u = dev_unpack2<T>(ld_last_u32<woff<i>()>(src_plane<i>(q)));
            const float2 v = dev_unpack2<T>(ld_last_u32<woff<i + 1>()>(src_plane<i + 1>(q)));
            da += u.x + v.x;
            db += u.y + v.y;
            f[0][i] = u.x;
            f[1][i] = u.y;
            f[0][i + 1] = v.x;
            f[1][i + 1] = v.y;
        });
        ra = o.z + (1.f - wgt<float>(0)) * o.x + da;
        rb = o.w + (1.f - wgt<float>(0)) * o.y + db;
    }
    template <int I>
    static __device__ __forceinline__ void store_word(Out o, unsigned v) {
        st_cs_u32<4 * (3 + I) * G::PITCH>(o.w, v);
    }
};

// Collision of one node from its 38 pulled populations f, its densities rho2
// and its neighbours' (nb(dx, dy, dz) -> {A, B}): momentum (Eq. 6), Shan-Chen
// force (Eq. 7), common velocity with the force shift, BGK relaxation to the
// equilibrium of Eq. 8 (Eqs. 9, 10) -- or, with MRT (float32 storage), the
// moment relaxation of the generic kernel -- and the store of the
// post-collision state (float32 populations with the rest population closing
// the mass balance, or 16-bit deviations).  Also accumulates the
// centre-of-mass partials of the droplet phase and flags non-finite
// densities.  Shared by the row kernels and the two-pass kernels of their
// widths so that every variant computes bit-identical states.
template <typename IO, typename ST, bool MRT, typename NB>
__device__ __forceinline__ void collide_core(NB&& nb, const float2 rho2, const float (&f)[2][19],
                                             const float (&rs)[2], const FastModel& m, typename IO::Out out,
                                             float (&cm)[4], int& bad, float px, float py, float pz) {
    const float rho[2] = {rho2.x, rho2.y};
    float j[2][3], acc[2][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
    if constexpr (is_dev_t<ST>::value) {
        // momentum (Eq. 6) of both components, opposite pairs differenced first
        float2 j2[3];
        bool jset[3] = {false, false, false};
        auto gather = [](float2& a, bool& set, int c, float2 d) {  // a += c d
            if (c == 0) return;
            a = set ? (c > 0 ? add2(a, d) : sub2(a, d)) : d;  // (the first direction of each sum has c = 1)
            set = true;
        };
#pragma unroll
        for (int i = 1; i < 19; i += 2) {
            const float2 d = sub2(pair(f[0][i], f[1][i]), pair(f[0][i + 1], f[1][i + 1]));
            gather(j2[0], jset[0], cx_(i), d);
            gather(j2[1], jset[1], cy_(i), d);
            gather(j2[2], jset[2], cz_(i), d);
        }
        // Shan-Chen force (Eq. 7) sums sum_i w_i rho_s(x + c_i) c_i, neighbour
        // pairs differenced first; the weight folds into the multiplier
        float2 acc2[3];
        bool aset[3] = {false, false, false};
        auto weigh = [](float2& a, bool& set, float c, float2 d) {  // a += c d
            if (c == 0.f) return;
            a = set ? fma2(both(c), d, a) : mul2(both(c), d);
            set = true;
        };
#pragma unroll
        for (int i = 1; i < 19; i += 2) {
            const float2 d = sub2(nb(cx_(i), cy_(i), cz_(i)), nb(-cx_(i), -cy_(i), -cz_(i)));
            weigh(acc2[0], aset[0], wgt<float>(i) * cx_(i), d);
            weigh(acc2[1], aset[1], wgt<float>(i) * cy_(i), d);
            weigh(acc2[2], aset[2], wgt<float>(i) * cz_(i), d);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            j[0][a] = j2[a].x;
            j[1][a] = j2[a].y;
            acc[0][a] = acc2[a].x;
            acc[1][a] = acc2[a].y;
        }
    } else {
        // momentum (Eq. 6), opposite pairs differenced first
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            float jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
            for (int i = 1; i < 19; i += 2) {
                const float d = f[s][i] - f[s][i + 1];
                if (cx_(i)) jx += (float)cx_(i) * d;
                if (cy_(i)) jy += (float)cy_(i) * d;
                if (cz_(i)) jz += (float)cz_(i) * d;
            }
            j[s][0] = jx; j[s][1] = jy; j[s][2] = jz;
        }
        // Shan-Chen force (Eq. 7) sums sum_i w_i rho_s(x + c_i) c_i, neighbour
        // pairs differenced first; the weight folds into the multiplier
#pragma unroll
        for (int i = 1; i < 19; i += 2) {
            const float2 np = nb(cx_(i), cy_(i), cz_(i)), nm = nb(-cx_(i), -cy_(i), -cz_(i));
            const float dA = np.x - nm.x, dB = np.y - nm.y;
            if (cx_(i)) { acc[0][0] += (wgt<float>(i) * cx_(i)) * dA; acc[1][0] += (wgt<float>(i) * cx_(i)) * dB; }
            if (cy_(i)) { acc[0][1] += (wgt<float>(i) * cy_(i)) * dA; acc[1][1] += (wgt<float>(i) * cy_(i)) * dB; }
            if (cz_(i)) { acc[0][2] += (wgt<float>(i) * cz_(i)) * dA; acc[1][2] += (wgt<float>(i) * cz_(i)) * dB; }
        }
    }
    const float den = rho[0] * m.inv_tau[0] + rho[1] * m.inv_tau[1];
    const float rden = __frcp_rn(den);
    float up[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) up[a] = (j[0][a] * m.inv_tau[0] + j[1][a] * m.inv_tau[1]) * rden;
    if (!(isfinite(rho[0]) && isfinite(rho[1]))) bad |= 1;
    {
        const float phi = __fdividef(rho[0] - rho[1], rho[0] + rho[1]);
        const float w = fmaxf(phi, 0.f);
        cm[0] += w;
        cm[1] = fmaf(w, px, cm[1]);
        cm[2] = fmaf(w, py, cm[2]);
        cm[3] = fmaf(w, pz, cm[3]);
    }
    if constexpr (is_dev_t<ST>::value) {
        // 16-bit deviations from w_i times the density of the node each
        // population streams to (this CTA's density planes), the pair of
        // components of one direction in one word
        // f holds the pulled deviations (f_i = w_i rho*_s + d_i, rs = rho*):
        // (1 - 1/tau) f_i = (1 - 1/tau) d_i + (1 - 1/tau) w_i rho*_s, whose
        // second term joins the equilibrium's constant (W1 / W2 below), and
        // the momentum's opposite-pair differences are those of the d_i
        using T = decltype(dev_tag(ST{}));
        float ux[2], uy[2], uz[2], base[2], e1[2], e2[2], W1[2], W2[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            ux[s] = fmaf(m.sh[s], acc[1 - s][0], up[0]);
            uy[s] = fmaf(m.sh[s], acc[1 - s][1], up[1]);
            uz[s] = fmaf(m.sh[s], acc[1 - s][2], up[2]);
            base[s] = 1.f - 1.5f * (ux[s] * ux[s] + uy[s] * uy[s] + uz[s] * uz[s]);
            const float ir = m.inv_tau[s] * rho[s];
            e1[s] = ir * wgt<float>(1);  // axis directions
            e2[s] = ir * wgt<float>(7);  // edge directions
            const float orr = m.omit[s] * rs[s];
            W1[s] = orr * wgt<float>(1);
            W2[s] = orr * wgt<float>(7);
        }
        float2 others = both(0.f);
        const float2 ux2 = pair(ux[0], ux[1]), uy2 = pair(uy[0], uy[1]), uz2 = pair(uz[0], uz[1]);
        const float2 base2 = pair(base[0], base[1]), om2 = pair(m.omit[0], m.omit[1]);
        const float2 eA = pair(e1[0], e1[1]), eE = pair(e2[0], e2[1]);
        const float2 WA = pair(W1[0], W1[1]), WE = pair(W2[0], W2[1]);
        const float2 oA = mul2(both(3.f), eA), oE = mul2(both(3.f), eE);
        sfor<9>([&](auto K) {
            constexpr int i = 2 * decltype(K)::value + 1;
            // densities of the destinations x + c_i and x - c_i (read again
            // from shared memory rather than held since the force)
            const float2 np = nb(cx_(i), cy_(i), cz_(i)), nm = nb(-cx_(i), -cy_(i), -cz_(i));
            const float2 cu = dot_c2(i, ux2, uy2, uz2);
            const float2 ev = fma2(i < 7 ? eA : eE, fma2(mul2(both(4.5f), cu), cu, base2), i < 7 ? WA : WE);
            const float2 od = mul2(i < 7 ? oA : oE, cu);
            // deviations from w_i times the destinations' densities
            const float2 da = fma2(both(-wgt<float>(i)), np, fma2(om2, pair(f[0][i], f[1][i]), add2(ev, od)));
            const float2 db = fma2(both(-wgt<float>(i)), nm, fma2(om2, pair(f[0][i + 1], f[1][i + 1]), sub2(ev, od)));
            const unsigned wa = dev_pack2<T>(da.x, da.y), wb = dev_pack2<T>(db.x, db.y);
            IO::template store_word<i>(out, wa);
            IO::template store_word<i + 1>(out, wb);
            // the values the readers will rebuild, for the mass balance
            others = add2(others, add2(fma2(both(wgt<float>(i)), np, dev_unpack2<T>(wa)),
                                       fma2(both(wgt<float>(i)), nm, dev_unpack2<T>(wb))));
        });
        st_cs_f4(out.b, make_float4(rho[0], rho[1], rho[0] - others.x, rho[1] - others.y));
    } else {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const float ux = fmaf(m.sh[s], acc[1 - s][0], up[0]);
            const float uy = fmaf(m.sh[s], acc[1 - s][1], up[1]);
            const float uz = fmaf(m.sh[s], acc[1 - s][2], up[2]);
            const float r = rho[s];
            // moving populations; the rest population then closes the mass
            // balance exactly (sum of outputs = rho), which keeps fp32
            // rounding from drifting the interface
            float others = 0.f;
            if constexpr (MRT) {
                // MRT: relax the moments of the deviation from equilibrium
                // (d'Humieres basis; momentum and stress at 1/tau)
                const float u2x = 1.5f * (ux * ux + uy * uy + uz * uz);
                float dv[19], o[19];
#pragma unroll
                for (int i = 0; i < 19; ++i) dv[i] = f[s][i] - feq<float>(i, r, ux, uy, uz, u2x);
                mrt_relax_full<float>(f[s], dv, m.inv_tau[s], m.mrt, o);
                sfor<9>([&](auto K) {
                    constexpr int i = 2 * decltype(K)::value + 1;
                    if (s == 0) {
                        IO::template store<0, i>(out, o[i]);
                        IO::template store<0, i + 1>(out, o[i + 1]);
                    } else {
                        IO::template store<1, i>(out, o[i]);
                        IO::template store<1, i + 1>(out, o[i + 1]);
                    }
                    others += o[i] + o[i + 1];
                });
            } else {
                const float base = 1.f - 1.5f * (ux * ux + uy * uy + uz * uz);
                const float ir = m.inv_tau[s] * r;
                const float e1 = ir * wgt<float>(1), e2 = ir * wgt<float>(7);
                const float om = m.omit[s];
                sfor<9>([&](auto K) {
                    constexpr int i = 2 * decltype(K)::value + 1;
                    const float cu = dot_c<float>(i, ux, uy, uz);
                    const float e = i < 7 ? e1 : e2;
                    const float ev = e * fmaf(4.5f * cu, cu, base);
                    const float od = (3.f * e) * cu;
                    const float oa = fmaf(om, f[s][i], ev + od);
                    const float ob = fmaf(om, f[s][i + 1], ev - od);
                    if (s == 0) {
                        IO::template store<0, i>(out, oa);
                        IO::template store<0, i + 1>(out, ob);
                    } else {
                        IO::template store<1, i>(out, oa);
                        IO::template store<1, i + 1>(out, ob);
                    }
                    others += oa + ob;
                });
            }
            if (s == 0) IO::template store<0, 0>(out, r - others);
            else IO::template store<1, 0>(out, r - others);
        }
    }
}

}  // namespace
}  // namespace lbmgb
