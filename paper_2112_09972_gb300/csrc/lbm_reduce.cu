// Reductions and observables over the population field:
//
//   k_moments / k_moments_final -- the droplet's ten float64 moments of
//       w = max(phi, 0), phi = (rho_A - rho_B)/(rho_A + rho_B), reduced with
//       warp shuffles, then the central second-moment tensor, its eigenvalues
//       and eigenvectors (cyclic Jacobi, float64) and the deformation
//       D = (L - W)/(L + W) of Sec. 2, Eq. 4 with L, W proportional to
//       sqrt(lambda_max), sqrt(lambda_min) (a uniform ellipsoid has principal
//       second moments a_k^2 / 5);
//   k_fields    -- rho_A, rho_B and u of the stored populations (Eq. 6);
//   k_checksums -- float64 mass of each component and total momentum;
//   k_pack / k_unpack -- float64 host layout <-> padded device layout.
// Each reads float64, float32 or 16-bit deviation storage (lbm_dev.cuh); the
// latter rebuilds the populations it needs from rho* and the deviations.
//
// Reductions are deterministic: a fixed grid, a fixed in-block tree and a
// fixed-order final pass.

#include <cuda_runtime.h>

#include <type_traits>

#include "lbm_dev.cuh"
#include "lbm_eigen.cuh"
#include "lbm_internal.h"
#include "lbm_lattice.cuh"

namespace lbmgb {
namespace {

__host__ __device__ __forceinline__ constexpr int qx(int i) {
    constexpr int t[19] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
    return t[i];
}
__host__ __device__ __forceinline__ constexpr int qy(int i) {
    constexpr int t[19] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
    return t[i];
}
__host__ __device__ __forceinline__ constexpr int qz(int i) {
    constexpr int t[19] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};
    return t[i];
}

constexpr int kRedThreads = 256;

// What 16-bit deviation storage needs to rebuild populations that leave the box.
struct DevRef {
    float rho_b[2];
    int periodic;
};

DevRef dev_ref(const Model& m) {
    DevRef r;
    r.rho_b[0] = (float)m.rho_b[0];
    r.rho_b[1] = (float)m.rho_b[1];
    r.periodic = m.periodic;
    return r;
}

// Post-collision population (s, i) of fluid node (x, y, z).  Deviation
// storage: i = 0 is the stored rest population, i >= 1 is rebuilt as
// w_i rho*(x + c_i) + d_i in float32, the arithmetic of the stream-collide
// kernels (rho_b where x + c_i lies outside the box).
template <typename S>
__device__ __forceinline__ double population(const S* __restrict__ f, const Layout& L, const DevRef& r, int s, int i,
                                             int x, int y, int z) {
    if constexpr (is_dev_t<S>::value) {
        using T = decltype(dev_tag(S{}));
        const float4* nb = reinterpret_cast<const float4*>(f);
        if (i == 0) {
            const float4 o = nb[L.dev_node(x, y, z)];
            return (double)(s ? o.w : o.z);
        }
        int xd = x + qx(i), yd = y + qy(i), zd = z + qz(i);
        float rd = r.rho_b[s];
        if (r.periodic) {
            xd = (xd + L.Lx) % L.Lx; yd = (yd + L.Ly) % L.Ly; zd = (zd + L.Lz) % L.Lz;
        }
        if (xd >= 0 && xd < L.Lx && yd >= 0 && yd < L.Ly && zd >= 0 && zd < L.Lz) {
            const float4 o = nb[L.dev_node(xd, yd, zd)];
            rd = s ? o.y : o.x;
        }
        const unsigned short b = reinterpret_cast<const unsigned short*>(f)[L.dev_at(s, i, x, y, z)];
        return (double)(wgt<float>(i) * rd + dev_to_f<T>(b));
    } else {
        (void)r;
        return (double)f[L.at(s, i, x, y, z)];
    }
}

// hi + lo += v, exactly up to the rounding of lo: TwoSum (Knuth) gives the
// rounding error of hi + v, which lo gathers.
__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float v) {
    const float s = hi + v;
    const float vv = s - hi;
    const float e = (hi - (s - vv)) + (v - vv);
    hi = s;
    lo += e;
}

// Component densities of fluid node (x, y, z) as unevaluated pairs hi + lo:
// the sum of its populations, or rho* of deviation storage (the same value up
// to float32 rounding).  Float32 storage sums in float32 (Knuth's TwoSum per
// addition, its rounding errors gathered in lo), so that the 36 additions run
// on the float32 pipe (this GPU's FP64 pipe runs at 1/64 of its rate); hi +
// lo agrees with a float64 sum to about 1e-14 relative.
template <typename S>
struct RhoPair {
    using T = typename std::conditional<std::is_same<S, double>::value, double, float>::type;
    T ah, al, bh, bl;
    __device__ __forceinline__ double a() const {
        if constexpr (std::is_same<S, float>::value) return (double)ah + (double)al;
        else return ah;
    }
    __device__ __forceinline__ double b() const {
        if constexpr (std::is_same<S, float>::value) return (double)bh + (double)bl;
        else return bh;
    }
    // false only when phi = (a - b) / (a + b) is certainly not above zero:
    // a - b below and a + b above what their evaluation here can be off by
    __device__ __forceinline__ bool droplet() const {
        if constexpr (std::is_same<S, double>::value)  // the signs, read on the integer pipe
            return (__double2hiint(ah - bh) ^ __double2hiint(ah + bh)) >= 0;
        const T d = (ah - bh) + (al - bl), t = (ah + bh) + (al + bl);
        const T m = T(1e-6) * ((fabs(ah) + fabs(bh)) + (fabs(al) + fabs(bl)));
        return !(d < -m && t > m);
    }
};
template <typename S>
__device__ __forceinline__ RhoPair<S> node_rho_pair(const S* __restrict__ f, const Layout& L, int x, int y, int z) {
    RhoPair<S> r;
    r.al = r.bl = 0;
    if constexpr (is_dev_t<S>::value) {
        const float4 o = reinterpret_cast<const float4*>(f)[L.dev_node(x, y, z)];
        r.ah = o.x;
        r.bh = o.y;
    } else {
        const long long b = L.at(0, 0, x, y, z);
        r.ah = f[b];
        r.bh = f[b + 19LL * L.pitch];
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            const S va = f[b + (long long)i * L.pitch], vb = f[b + (long long)(19 + i) * L.pitch];
            if constexpr (std::is_same<S, float>::value) {
                two_sum_acc(r.ah, r.al, va);
                two_sum_acc(r.bh, r.bl, vb);
            } else {
                r.ah += va;
                r.bh += vb;
            }
        }
    }
    return r;
}
template <typename S>
__device__ __forceinline__ void node_rho(const S* __restrict__ f, const Layout& L, int x, int y, int z, double& ra,
                                         double& rb) {
    const RhoPair<S> r = node_rho_pair(f, L, x, y, z);
    ra = r.a();
    rb = r.b();
}

// n / d to float64 rounding or one unit more: a float32 quotient carried to
// float64 by two Newton steps (4 FP64 instructions instead of a divide's
// dozen); the plain divide outside float32's range.
__device__ __forceinline__ double div64(double n, double d) {
    const float df = (float)d;
    if (!(fabsf(df) > 1e-30f && fabsf(df) < 1e30f)) return n / d;
    const double y = (double)__frcp_rn(df);
    double q = n * y;
    q = fma(fma(-q, d, n), y, q);
    return fma(fma(-q, d, n), y, q);
}

// Block-wide sum of K doubles per thread; thread 0 writes them to out[0..K).
template <int K>
__device__ void block_sum(double (&v)[K], double* out) {
    __shared__ double part[kRedThreads / 32][K];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        double a = v[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        v[k] = a;
    }
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) part[warp][k] = v[k];
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            double a = lane < kRedThreads / 32 ? part[lane][k] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
            if (lane == 0) out[k] = a;
        }
    }
}

// Ten moments of w = max(phi, 0).  Few nodes have phi > 0 (a droplet of R =
// L / 8 fills 0.8 % of its box), so only those run FP64 instructions, and
// warps and CTAs without one skip the FP64 reductions.  The CTAs walk the box
// together in node order: DRAM then serves neighbouring rows at the same time
// (a march of each warp along z read as many bytes at 45 % of its peak).
// 128^3 float32 on GB300: 180 us with ten FP64 sums per node and the
// reductions in every warp, bound by the FP64 pipe; 102 us marching; 67 us now
// (0.70 of the measured copy rate, waiting for its loads).
template <typename S>
__global__ void __launch_bounds__(kRedThreads, 4) k_moments(const S* __restrict__ f, Layout L,
                                                            double* __restrict__ partials) {
    __shared__ double part[kRedThreads / 32][10];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double m[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) m[k] = 0.0;
    bool drop = false;
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (long long)gridDim.x * blockDim.x) {
        const int row = (int)(n / L.Lx), y = row % L.Ly, z = row / L.Ly, x = (int)(n - (long long)row * L.Lx);
        const RhoPair<S> r = node_rho_pair(f, L, x, y, z);
        if (!r.droplet()) continue;
        const double ra = r.a(), rb = r.b();
        const double w = (ra - rb) / (ra + rb);
        if (w > 0.0) {
            const double px = x - 0.5 * (L.Lx - 1), py = y - 0.5 * (L.Ly - 1), pz = z - 0.5 * (L.Lz - 1);
            const double wx = w * px, wy = w * py, wz = w * pz;
            m[0] += w;
            m[1] += wx; m[2] += wy; m[3] += wz;
            m[4] = fma(wx, px, m[4]); m[5] = fma(wx, py, m[5]); m[6] = fma(wx, pz, m[6]);
            m[7] = fma(wy, py, m[7]); m[8] = fma(wy, pz, m[8]); m[9] = fma(wz, pz, m[9]);
            drop = true;
        }
    }
    const bool some = __any_sync(0xffffffffu, drop);
    if (some) {
#pragma unroll
        for (int k = 0; k < 10; ++k) {
            double a = m[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
            if (lane == 0) part[warp][k] = a;
        }
    } else if (lane < 10) {
        part[warp][lane] = 0.0;
    }
    const int any = __syncthreads_or(some);
    if (threadIdx.x < 10) {
        double a = part[0][threadIdx.x];
        if (any)
            for (int w = 1; w < kRedThreads / 32; ++w) a += part[w][threadIdx.x];
        partials[10LL * blockIdx.x + threadIdx.x] = a;
    }
}

// Sum the per-block partials in a fixed order (warp k sums moment k), then
// derive D and the axes (one thread).
constexpr int kMomentsFinalThreads = 320;
__global__ void __launch_bounds__(kMomentsFinalThreads) k_moments_final(const double* __restrict__ partials,
                                                                        int nblocks, double* __restrict__ result) {
    __shared__ double sum[10];
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
    double a = 0.0;
    for (int b0 = lane; b0 < nblocks; b0 += 256) {  // eight loads in flight
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = b0 + 32 * u < nblocks ? partials[10LL * (b0 + 32 * u) + k] : 0.0;
#pragma unroll
        for (int u = 0; u < 8; ++u) a += v[u];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if (lane == 0) sum[k] = a;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double m[10];
#pragma unroll
    for (int q = 0; q < 10; ++q) m[q] = sum[q];
    deformation_from_moments(m, result);
}

template <typename S>
__global__ void k_fields(const S* __restrict__ f, Layout L, DevRef dr, double* __restrict__ ra_out,
                         double* __restrict__ rb_out, double* __restrict__ u_out) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const int x = (int)(n % L.Lx), y = (int)((n / L.Lx) % L.Ly), z = (int)(n / ((long long)L.Lx * L.Ly));
    double r[2] = {0.0, 0.0}, j[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            const double v = population(f, L, dr, s, i, x, y, z);
            r[s] += v;
            if (qx(i)) j[0] += qx(i) * v;
            if (qy(i)) j[1] += qy(i) * v;
            if (qz(i)) j[2] += qz(i) * v;
        }
    if (ra_out) ra_out[n] = r[0];
    if (rb_out) rb_out[n] = r[1];
    if (u_out) {
        const double tot = r[0] + r[1];
        u_out[3 * n + 0] = j[0] / tot;
        u_out[3 * n + 1] = j[1] / tot;
        u_out[3 * n + 2] = j[2] / tot;
    }
}

template <typename S>
__global__ void __launch_bounds__(kRedThreads) k_checksums(const S* __restrict__ f, Layout L, DevRef dr,
                                                           double* __restrict__ partials) {
    double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(n % L.Lx), y = (int)((n / L.Lx) % L.Ly), z = (int)(n / ((long long)L.Lx * L.Ly));
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int i = 0; i < 19; ++i) {
                const double q = population(f, L, dr, s, i, x, y, z);
                v[s] += q;
                if (qx(i)) v[2] += qx(i) * q;
                if (qy(i)) v[3] += qy(i) * q;
                if (qz(i)) v[4] += qz(i) * q;
            }
    }
    block_sum<5>(v, partials + 5LL * blockIdx.x);
}

__global__ void k_checksums_final(const double* __restrict__ partials, int nblocks, double* __restrict__ out) {
    const int lane = threadIdx.x;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        double a = 0.0;
        for (int b = lane; b < nblocks; b += 32) a += partials[5LL * b + k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        if (lane == 0) out[k] = a;
    }
}

template <typename S>
__global__ void k_pack(const S* __restrict__ f, Layout L, DevRef dr, double* __restrict__ out) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= 38 * N) return;
    const int si = (int)(e / N);
    const long long n = e - si * N;
    const int x = (int)(n % L.Lx), y = (int)((n / L.Lx) % L.Ly), z = (int)(n / ((long long)L.Lx * L.Ly));
    out[e] = population(f, L, dr, si / 19, si % 19, x, y, z);
}

// Deviation storage upload, pass 1: rho*_s = float32 of the float64 sum of
// node n's populations, into rho[s * N + n].
__global__ void k_unpack_dev_rho(Layout L, const double* __restrict__ in, float* __restrict__ rho) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        double a = 0.0;
#pragma unroll
        for (int i = 0; i < 19; ++i) a += in[(long long)(s * 19 + i) * N + n];
        rho[s * N + n] = (float)a;
    }
}

// Pass 2: deviations from w_i rho*(x + c_i), node block with the rest
// population closing the node's mass (the arithmetic of the kernels).
template <typename T>
__global__ void k_unpack_dev(Dev<T>* __restrict__ f, Layout L, DevRef dr, const double* __restrict__ in,
                             const float* __restrict__ rho) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const int x = (int)(n % L.Lx), y = (int)((n / L.Lx) % L.Ly), z = (int)(n / ((long long)L.Lx * L.Ly));
    unsigned short* d = reinterpret_cast<unsigned short*>(f);
    float rest[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        float others = 0.f;
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            int xd = x + qx(i), yd = y + qy(i), zd = z + qz(i);
            if (dr.periodic) {
                xd = (xd + L.Lx) % L.Lx; yd = (yd + L.Ly) % L.Ly; zd = (zd + L.Lz) % L.Lz;
            }
            float rd = dr.rho_b[s];
            if (xd >= 0 && xd < L.Lx && yd >= 0 && yd < L.Ly && zd >= 0 && zd < L.Lz)
                rd = rho[s * N + ((long long)zd * L.Ly + yd) * L.Lx + xd];
            const float ref = wgt<float>(i) * rd;
            const unsigned short b = dev_from_f<T>((float)(in[(long long)(s * 19 + i) * N + n] - (double)ref));
            d[L.dev_at(s, i, x, y, z)] = b;
            others += ref + dev_to_f<T>(b);
        }
        rest[s] = rho[s * N + n] - others;
    }
    reinterpret_cast<float4*>(f)[L.dev_node(x, y, z)] = make_float4(rho[n], rho[N + n], rest[0], rest[1]);
}

template <typename S>
__global__ void k_unpack(S* __restrict__ f, Layout L, const double* __restrict__ in) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= 38 * N) return;
    const int si = (int)(e / N);
    const long long n = e - si * N;
    const int x = (int)(n % L.Lx), y = (int)((n / L.Lx) % L.Ly), z = (int)(n / ((long long)L.Lx * L.Ly));
    f[L.at(si / 19, si % 19, x, y, z)] = (S)in[e];
}

// ---- connected components of the droplet phase (breakup detection) ----

// The labels are a union-find forest in memory: label[n] <= n is the parent
// of node n (itself for a root), -1 outside the phase, and roots end as the
// smallest node index of their component.  Three launches, whatever the
// components' shapes, and no host round trip between them; the sweeps of
// minimum-label propagation that this replaced were launched four at a time
// with a read-back after each four.

// label[n] = the start of the run of phase nodes along x that n belongs to
// (within the 32 nodes of its warp), -1 where phi <= threshold; n = (z Ly + y)
// Lx + x.  Also zeroes the sizes and the root counter.
template <typename S>
__global__ void k_cc_init(const S* __restrict__ f, Layout L, double threshold, int* __restrict__ label,
                          int* __restrict__ size, int* __restrict__ flags) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n < 2) flags[n] = 0;
    bool in = false;
    int x = 0;
    if (n < N) {
        const int row = (int)n / L.Lx, y = row % L.Ly, z = row / L.Ly;
        x = (int)n - row * L.Lx;
        const RhoPair<S> r = node_rho_pair(f, L, x, y, z);
        // phi > threshold >= 0 needs phi > 0: no FP64 outside the droplet
        if (threshold < 0.0 || r.droplet()) {
            const double ra = r.a(), rb = r.b();
            in = (ra - rb) / (ra + rb) > threshold;
        }
    }
    const int lane = threadIdx.x & 31;
    const unsigned ins = __ballot_sync(0xffffffffu, in);
    const bool first = in && (lane == 0 || x == 0 || !((ins >> (lane - 1)) & 1u));
    const unsigned starts = __ballot_sync(0xffffffffu, first);
    if (n >= N) return;
    const int start = 31 - __clz((int)(starts & (0xffffffffu >> (31 - lane))));
    label[n] = in ? (int)n - (lane - start) : -1;
    size[n] = 0;
}

// Root of node a's tree.  Parents are smaller than their children, so the
// walk ends; `steps` bounds it all the same.
__device__ __forceinline__ int cc_find(const int* label, int a, long long& steps) {
    int p = __ldcg(label + a);
    while (p != a && --steps > 0) {
        a = p;
        p = __ldcg(label + a);
    }
    return a;
}

// Join the trees of nodes a and b: the larger root's parent becomes the
// smaller root.  A root that another thread has attached meanwhile yields its
// new parent, which is joined instead (parents only decrease).
__device__ __forceinline__ void cc_join(int* label, int a, int b, long long& steps) {
    while (steps > 0) {
        a = cc_find(label, a, steps);
        b = cc_find(label, b, steps);
        if (a == b) return;
        const int hi = a > b ? a : b, lo = a > b ? b : a;
        const int old = atomicMin(label + hi, lo);
        if (old == hi) return;
        a = old;
        b = lo;
        --steps;
    }
}

// Joins every phase node with its phase neighbours at x + 1 (where the runs
// of k_cc_init end), y + 1 and z + 1, wrapping in the periodic mode.  A y or z
// edge is left out where the nodes at x - 1 have one too (both pairs are
// joined along x).  flags[0] is set if a walk exceeded its bound.
__global__ void k_cc_join(Layout L, int periodic, int* __restrict__ label, int* __restrict__ flags) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N || __ldcg(label + n) < 0) return;
    const int row = (int)n / L.Lx, y = row % L.Ly, z = row / L.Ly, x = (int)n - row * L.Lx;
    long long steps = 64 * (N + 8);
    const bool left = x > 0 && __ldcg(label + n - 1) >= 0;
    auto edge = [&](long long nb, bool skippable) {
        if (__ldcg(label + nb) < 0) return;
        if (skippable && left && __ldcg(label + nb - 1) >= 0) return;
        cc_join(label, (int)n, (int)nb, steps);
    };
    const long long sy = L.Lx, sz = (long long)L.Lx * L.Ly;
    if (x + 1 < L.Lx) {
        if ((n & 31) == 31) edge(n + 1, false);
    } else if (periodic) {
        edge(n - x, false);
    }
    if (y + 1 < L.Ly) edge(n + sy, true);
    else if (periodic) edge(n - (long long)y * sy, true);
    if (z + 1 < L.Lz) edge(n + sz, true);
    else if (periodic) edge(n - (long long)z * sz, true);
    if (steps <= 0) flags[0] = 1;
}

// Component sizes: size[root] += 1 for every phase node, one atomic per
// distinct root of a warp.
__global__ void k_cc_sizes(Layout L, const int* __restrict__ label, int* __restrict__ size, int* __restrict__ flags) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = n < N && label[n] >= 0;
    const unsigned mask = __ballot_sync(0xffffffffu, in);
    if (!in) return;
    long long steps = N + 8;
    const int root = cc_find(label, (int)n, steps);
    if (steps <= 0) flags[0] = 1;
    const unsigned same = __match_any_sync(mask, root);
    if ((int)(threadIdx.x & 31) == __ffs((int)same) - 1) atomicAdd(size + root, __popc(same));
}

// The roots' sizes, in no particular order; flags[1] counts them.
__global__ void k_cc_roots(Layout L, const int* __restrict__ label, const int* __restrict__ size,
                           int* __restrict__ flags, long long* __restrict__ out, int cap) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    if (label[n] != (int)n) return;
    const int k = atomicAdd(flags + 1, 1);
    if (k < cap) out[k] = size[n];
}

// ---- surface-area deformation (Eq. 17) and mass reinjection ----

// phi = (a - b) / (a + b) of a node, kept for the gradient pass: a double for
// float64 storage; for the float32 and 16-bit forms an unevaluated float32
// pair hi + lo good to 2^-44, a thousandth of what the stored populations'
// own rounding leaves, so that phi, its sum and its gradient stay off the
// FP64 pipe (which bounded both passes: 96 and 88 us at 128^3 float32; 67 and
// 16 us now).
struct Pair {
    float h, l;
};
__device__ __forceinline__ Pair two_sum(float a, float b) {  // Knuth: a + b = h + l exactly
    const float h = a + b, bb = h - a;
    return {h, (a - (h - bb)) + (b - bb)};
}
__device__ __forceinline__ Pair renorm(float h, float l) {  // |h| >= |l|
    const float s = h + l;
    return {s, l - (s - h)};
}
__device__ __forceinline__ double phi_value(double p) { return p; }
__device__ __forceinline__ double phi_value(Pair p) { return (double)p.h + (double)p.l; }
__device__ __forceinline__ bool phi_number(double p) { return p == p; }
__device__ __forceinline__ bool phi_number(Pair p) { return p.h == p.h; }
__device__ __forceinline__ bool phi_less(double a, double b) { return a < b; }
__device__ __forceinline__ bool phi_less(Pair a, Pair b) { return a.h < b.h || (a.h == b.h && a.l < b.l); }

template <typename S>
struct PhiOf {
    using T = typename std::conditional<std::is_same<S, double>::value, double, Pair>::type;
};
__device__ __forceinline__ double node_phi(const RhoPair<double>& r) { return div64(r.ah - r.bh, r.ah + r.bh); }
template <typename S>
__device__ __forceinline__ Pair node_phi(const RhoPair<S>& r) {
    Pair d = two_sum(r.ah, -r.bh), t = two_sum(r.ah, r.bh);
    d.l += r.al - r.bl;
    t.l += r.al + r.bl;
    if (!(fabsf(t.h) > 1e-25f && fabsf(t.h) < 1e25f && fabsf(d.h) < 1e25f)) {
        const double p = (r.a() - r.b()) / (r.a() + r.b());
        return {(float)p, isfinite(p) ? (float)(p - (double)(float)p) : 0.f};
    }
    const float y = __frcp_rn(t.h), q = d.h * y;
    const float e = fmaf(-q, t.h, d.h) + fmaf(-q, t.l, d.l);
    return renorm(q, e * y);
}

// Sums of phi and of |grad phi|.  (The low parts in one float: gathered in a
// pair the sums of a 256 x 200 x 200 state changed by 1e-16 and the call took
// 374 us instead of 357.)
struct Acc64 {
    double s = 0.0;
    __device__ __forceinline__ void add(double v) { s += v; }
    __device__ __forceinline__ double value() const { return s; }
};
struct AccPair {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void add(Pair v) {
        two_sum_acc(h, l, v.h);
        l += v.l;
    }
    __device__ __forceinline__ double value() const { return isfinite(h) ? (double)h + (double)l : (double)h; }
};
template <typename T>
using Acc = typename std::conditional<std::is_same<T, double>::value, Acc64, AccPair>::type;

// phi of every fluid node into phi[n] (n = (z Ly + y) Lx + x) and per-block
// {sum phi, min phi, max phi}.
template <typename S>
__global__ void __launch_bounds__(kRedThreads) k_phi(const S* __restrict__ f, Layout L,
                                                     typename PhiOf<S>::T* __restrict__ phi,
                                                     double* __restrict__ partials) {
    using T = typename PhiOf<S>::T;
    __shared__ double red[3][kRedThreads / 32];
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    Acc<T> acc;
    T tlo, thi;
    bool seen = false;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (long long)gridDim.x * blockDim.x) {
        const int row = (int)(n / L.Lx), y = row % L.Ly, z = row / L.Ly, x = (int)(n - (long long)row * L.Lx);
        const T p = node_phi(node_rho_pair(f, L, x, y, z));
        phi[n] = p;
        acc.add(p);
        if (!phi_number(p)) continue;  // as fmin and fmax, the extremes pass over NaN
        if (!seen || phi_less(p, tlo)) tlo = p;
        if (!seen || phi_less(thi, p)) thi = p;
        seen = true;
    }
    double sum = acc.value(), lo = seen ? phi_value(tlo) : 1e300, hi = seen ? phi_value(thi) : -1e300;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_down_sync(0xffffffffu, sum, o);
        lo = fmin(lo, __shfl_down_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_down_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) { red[0][warp] = sum; red[1][warp] = lo; red[2][warp] = hi; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kRedThreads / 32; ++w) {
            red[0][0] += red[0][w];
            red[1][0] = fmin(red[1][0], red[1][w]);
            red[2][0] = fmax(red[2][0], red[2][w]);
        }
        double* out = partials + 4LL * blockIdx.x;
        out[0] = red[0][0]; out[1] = red[1][0]; out[2] = red[2][0];
    }
}

// sqrt(s) to float64 rounding or one unit more, from a float32 reciprocal
// square root (6 FP64 instructions instead of about 20).
__device__ __forceinline__ double sqrt64(double s) {
    const float sf = (float)s;
    if (!(sf > 1e-30f && sf < 1e30f)) return sqrt(s);
    const float yf = rsqrtf(sf);
    const double h = (double)(0.5f * yf);
    double r = s * (double)yf;
    r = fma(fma(-r, r, s), h, r);
    return fma(fma(-r, r, s), h, r);
}
// |g| from the differences of phi across a node.
__device__ __forceinline__ double magnitude(double x1, double x0, double y1, double y0, double z1, double z0) {
    const double gx = x1 - x0, gy = y1 - y0, gz = z1 - z0;
    return sqrt64(fma(gx, gx, fma(gy, gy, gz * gz)));
}
__device__ __forceinline__ Pair magnitude(Pair x1, Pair x0, Pair y1, Pair y0, Pair z1, Pair z0) {
    auto square = [](Pair a, Pair b) -> Pair {  // (a - b)^2
        // neighbours far from the interface agree in the high part: the difference is then the low one's
        const Pair t = two_sum(a.h, -b.h), d = two_sum(t.h, t.l + (a.l - b.l));
        const float p = d.h * d.h;
        return {p, fmaf(2.f * d.h, d.l, fmaf(d.h, d.h, -p))};
    };
    const Pair a = square(x1, x0), b = square(y1, y0), c = square(z1, z0);
    const Pair ab = two_sum(a.h, b.h), s = two_sum(ab.h, c.h);
    const float lo = s.l + ab.l + (a.l + b.l + c.l);
    // outside, |g| < 1e-15 or above any physical phi; infinities and NaN pass through
    if (!(s.h > 1e-30f && s.h < 1e30f)) return {sqrtf(s.h), 0.f};
    const float y = rsqrtf(s.h), r = s.h * y;
    return renorm(r, 0.5f * y * (fmaf(-r, r, s.h) + lo));
}

// How k_grad_phi walks the box: a warp takes 32 consecutive
// nodes of an x-y plane (flattened, so that no width leaves lanes idle) and
// marches one of `zparts` parts of the z extent; units of work are numbered
// segment first.
struct Columns {
    int segs, zparts, zlen;
};
Columns columns(const Layout& L, long long warps) {
    Columns c;
    c.segs = (int)(((long long)L.Lx * L.Ly + 31) / 32);
    long long zp = warps / c.segs;
    zp = zp < 1 ? 1 : (zp > L.Lz ? L.Lz : zp);
    c.zlen = (int)((L.Lz + zp - 1) / zp);
    c.zparts = (L.Lz + c.zlen - 1) / c.zlen;
    return c;
}

// Per-block sum of |grad phi| (central differences) over interior nodes into
// partials[4 b + 3]; a lane marches in z (Columns) and keeps the two planes
// beside it in registers.
template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_grad_phi(Layout L, Columns c, const T* __restrict__ phi,
                                                          double* __restrict__ partials) {
    Acc<T> acc;
    const long long sy = L.Lx, sz = (long long)L.Lx * L.Ly;
    const long long units = (long long)c.segs * c.zparts;
    const long long stride = (long long)gridDim.x * (kRedThreads / 32);
    for (long long u = (long long)blockIdx.x * (kRedThreads / 32) + (threadIdx.x >> 5); u < units; u += stride) {
        const int zp = (int)(u / c.segs), p = (int)(u - (long long)zp * c.segs) * 32 + (threadIdx.x & 31);
        const int y = p / L.Lx, x = p - y * L.Lx;
        if (x < 1 || x > L.Lx - 2 || y < 1 || y > L.Ly - 2) continue;
        const int z0 = max(zp * c.zlen, 1), z1 = min((zp + 1) * c.zlen, L.Lz - 1);
        if (z0 >= z1) continue;
        const T* q = phi + (long long)z0 * sz + p;
        T below = q[-sz], here = q[0];
        for (int z = z0; z < z1; ++z, q += sz) {
            const T above = q[sz];
            acc.add(magnitude(q[1], q[-1], q[sy], q[-sy], above, below));
            below = here;
            here = above;
        }
    }
    double v[1] = {0.5 * acc.value()};
    double out[1];
    block_sum<1>(v, out);
    if (threadIdx.x == 0) partials[4LL * blockIdx.x + 3] = out[0];
}

// Reduction of the partials in a fixed order: {sum phi, min, max, sum |grad phi|}.
__global__ void __launch_bounds__(kRedThreads) k_phi_final(const double* __restrict__ partials, int nblocks,
                                                           double* __restrict__ out) {
    __shared__ double red[4][kRedThreads];
    double sum = 0.0, lo = 1e300, hi = -1e300, g = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kRedThreads) {
        const double* p = partials + 4LL * b;
        sum += p[0];
        lo = fmin(lo, p[1]);
        hi = fmax(hi, p[2]);
        g += p[3];
    }
    const int t = threadIdx.x;
    red[0][t] = sum; red[1][t] = lo; red[2][t] = hi; red[3][t] = g;
    for (int h = kRedThreads / 2; h > 0; h >>= 1) {
        __syncthreads();
        if (t < h) {
            red[0][t] += red[0][t + h];
            red[1][t] = fmin(red[1][t], red[1][t + h]);
            red[2][t] = fmax(red[2][t], red[2][t + h]);
            red[3][t] += red[3][t + h];
        }
    }
    if (t == 0)
        for (int q = 0; q < 4; ++q) out[q] = red[q][0];
}

// Per-block {mass of A where phi > 0, mass of A elsewhere}.
template <typename S>
__global__ void __launch_bounds__(kRedThreads) k_mass_split(const S* __restrict__ f, Layout L,
                                                            double* __restrict__ partials) {
    double v[2] = {0.0, 0.0};
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(n % L.Lx), y = (int)((n / L.Lx) % L.Ly), z = (int)(n / ((long long)L.Lx * L.Ly));
        double ra, rb;
        node_rho(f, L, x, y, z, ra, rb);
        v[(ra - rb) / (ra + rb) > 0.0 ? 0 : 1] += ra;
    }
    block_sum<2>(v, partials + 2LL * blockIdx.x);
}

__global__ void __launch_bounds__(kRedThreads) k_mass_final(const double* __restrict__ partials, int nblocks,
                                                            double* __restrict__ out) {
    double v[2] = {0.0, 0.0};
    for (int k = threadIdx.x; k < nblocks; k += kRedThreads) {
        v[0] += partials[2LL * k];
        v[1] += partials[2LL * k + 1];
    }
    block_sum<2>(v, out);
}

// f_A,i *= k at the nodes where phi > 0 (phi of the populations before scaling).
template <typename S>
__global__ void k_reinject(S* __restrict__ f, Layout L, double k) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const int x = (int)(n % L.Lx), y = (int)((n / L.Lx) % L.Ly), z = (int)(n / ((long long)L.Lx * L.Ly));
    double ra, rb;
    node_rho(f, L, x, y, z, ra, rb);
    if (!((ra - rb) / (ra + rb) > 0.0)) return;
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        S* q = f + L.at(0, i, x, y, z);
        *q = (S)((double)*q * k);
    }
}

}  // namespace

int moments_blocks(const Layout& L, int num_sms) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    long long b = (N + kRedThreads - 1) / kRedThreads;
    const long long cap = 4LL * (num_sms > 0 ? num_sms : 152);
    return (int)(b < cap ? b : cap);
}

cudaError_t launch_moments(int prec, const void* f, const Layout& L, double* partials, int nblocks, double* result,
                           cudaStream_t s) {
    if (prec == kFP64) k_moments<double><<<nblocks, kRedThreads, 0, s>>>((const double*)f, L, partials);
    else if (prec == kFP32) k_moments<float><<<nblocks, kRedThreads, 0, s>>>((const float*)f, L, partials);
    else if (prec == kFP16Dev) k_moments<Dev<__half>><<<nblocks, kRedThreads, 0, s>>>((const Dev<__half>*)f, L, partials);
    else k_moments<Dev<__nv_bfloat16>><<<nblocks, kRedThreads, 0, s>>>((const Dev<__nv_bfloat16>*)f, L, partials);
    k_moments_final<<<1, kMomentsFinalThreads, 0, s>>>(partials, nblocks, result);
    return cudaGetLastError();
}

cudaError_t launch_fields(int prec, const void* f, const Layout& L, const Model& m, double* ra, double* rb, double* u,
                          cudaStream_t s) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const unsigned blocks = (unsigned)((N + 255) / 256);
    const DevRef dr = dev_ref(m);
    if (prec == kFP64) k_fields<double><<<blocks, 256, 0, s>>>((const double*)f, L, dr, ra, rb, u);
    else if (prec == kFP32) k_fields<float><<<blocks, 256, 0, s>>>((const float*)f, L, dr, ra, rb, u);
    else if (prec == kFP16Dev) k_fields<Dev<__half>><<<blocks, 256, 0, s>>>((const Dev<__half>*)f, L, dr, ra, rb, u);
    else k_fields<Dev<__nv_bfloat16>><<<blocks, 256, 0, s>>>((const Dev<__nv_bfloat16>*)f, L, dr, ra, rb, u);
    return cudaGetLastError();
}

cudaError_t launch_checksums(int prec, const void* f, const Layout& L, const Model& m, double* partials, int nblocks,
                             double* result5, cudaStream_t s) {
    const DevRef dr = dev_ref(m);
    if (prec == kFP64) k_checksums<double><<<nblocks, kRedThreads, 0, s>>>((const double*)f, L, dr, partials);
    else if (prec == kFP32) k_checksums<float><<<nblocks, kRedThreads, 0, s>>>((const float*)f, L, dr, partials);
    else if (prec == kFP16Dev)
        k_checksums<Dev<__half>><<<nblocks, kRedThreads, 0, s>>>((const Dev<__half>*)f, L, dr, partials);
    else k_checksums<Dev<__nv_bfloat16>><<<nblocks, kRedThreads, 0, s>>>((const Dev<__nv_bfloat16>*)f, L, dr, partials);
    k_checksums_final<<<1, 32, 0, s>>>(partials, nblocks, result5);
    return cudaGetLastError();
}

cudaError_t launch_pack(int prec, const void* f, const Layout& L, const Model& m, double* out, cudaStream_t s) {
    const long long E = 38LL * L.Lx * L.Ly * L.Lz;
    const unsigned blocks = (unsigned)((E + 255) / 256);
    const DevRef dr = dev_ref(m);
    if (prec == kFP64) k_pack<double><<<blocks, 256, 0, s>>>((const double*)f, L, dr, out);
    else if (prec == kFP32) k_pack<float><<<blocks, 256, 0, s>>>((const float*)f, L, dr, out);
    else if (prec == kFP16Dev) k_pack<Dev<__half>><<<blocks, 256, 0, s>>>((const Dev<__half>*)f, L, dr, out);
    else k_pack<Dev<__nv_bfloat16>><<<blocks, 256, 0, s>>>((const Dev<__nv_bfloat16>*)f, L, dr, out);
    return cudaGetLastError();
}

cudaError_t launch_unpack(int prec, void* f, const Layout& L, const Model& m, const double* in, float* scratch,
                          cudaStream_t s) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    if (is_dev(prec)) {
        if (!scratch) return cudaErrorInvalidValue;
        const unsigned blocks = (unsigned)((N + 255) / 256);
        const DevRef dr = dev_ref(m);
        k_unpack_dev_rho<<<blocks, 256, 0, s>>>(L, in, scratch);
        if (prec == kFP16Dev) k_unpack_dev<__half><<<blocks, 256, 0, s>>>((Dev<__half>*)f, L, dr, in, scratch);
        else k_unpack_dev<__nv_bfloat16><<<blocks, 256, 0, s>>>((Dev<__nv_bfloat16>*)f, L, dr, in, scratch);
        return cudaGetLastError();
    }
    const long long E = 38LL * N;
    const unsigned blocks = (unsigned)((E + 255) / 256);
    if (prec == kFP64) k_unpack<double><<<blocks, 256, 0, s>>>((double*)f, L, in);
    else k_unpack<float><<<blocks, 256, 0, s>>>((float*)f, L, in);
    return cudaGetLastError();
}

}  // namespace lbmgb

namespace lbmgb {

cudaError_t launch_cc(int prec, const void* f, const Layout& L, int periodic, double threshold, int* label, int* size,
                      int* flags, long long* out, int cap, cudaStream_t s) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const unsigned blocks = (unsigned)((N + 255) / 256);
    if (prec == kFP64) k_cc_init<double><<<blocks, 256, 0, s>>>((const double*)f, L, threshold, label, size, flags);
    else if (prec == kFP32) k_cc_init<float><<<blocks, 256, 0, s>>>((const float*)f, L, threshold, label, size, flags);
    else if (prec == kFP16Dev)
        k_cc_init<Dev<__half>><<<blocks, 256, 0, s>>>((const Dev<__half>*)f, L, threshold, label, size, flags);
    else
        k_cc_init<Dev<__nv_bfloat16>>
            <<<blocks, 256, 0, s>>>((const Dev<__nv_bfloat16>*)f, L, threshold, label, size, flags);
    k_cc_join<<<blocks, 256, 0, s>>>(L, periodic, label, flags);
    k_cc_sizes<<<blocks, 256, 0, s>>>(L, label, size, flags);
    k_cc_roots<<<blocks, 256, 0, s>>>(L, label, size, flags, out, cap);
    return cudaGetLastError();
}

}  // namespace lbmgb

namespace lbmgb {

// out[0..3] = {sum phi, min phi, max phi, sum |grad phi| over interior nodes};
// scratch: N doubles (phi) and 4 nblocks doubles.
template <typename S>
void surface_stats_t(const S* f, const Layout& L, void* scratch, double* partials, int nblocks, cudaStream_t s) {
    using T = typename PhiOf<S>::T;
    const Columns c = columns(L, (long long)nblocks * (kRedThreads / 32));
    k_phi<S><<<nblocks, kRedThreads, 0, s>>>(f, L, (T*)scratch, partials);
    k_grad_phi<T><<<nblocks, kRedThreads, 0, s>>>(L, c, (const T*)scratch, partials);
}
cudaError_t launch_surface_stats(int prec, const void* f, const Layout& L, double* phi, double* partials, int nblocks,
                                 double* out, cudaStream_t s) {
    if (prec == kFP64) surface_stats_t((const double*)f, L, phi, partials, nblocks, s);
    else if (prec == kFP32) surface_stats_t((const float*)f, L, phi, partials, nblocks, s);
    else if (prec == kFP16Dev) surface_stats_t((const Dev<__half>*)f, L, phi, partials, nblocks, s);
    else surface_stats_t((const Dev<__nv_bfloat16>*)f, L, phi, partials, nblocks, s);
    k_phi_final<<<1, kRedThreads, 0, s>>>(partials, nblocks, out);
    return cudaGetLastError();
}

// out[0..1] = {mass of A where phi > 0, elsewhere}; partials: 2 nblocks doubles.
cudaError_t launch_mass_split(int prec, const void* f, const Layout& L, double* partials, int nblocks, double* out,
                              cudaStream_t s) {
    if (prec == kFP64) k_mass_split<double><<<nblocks, kRedThreads, 0, s>>>((const double*)f, L, partials);
    else if (prec == kFP32) k_mass_split<float><<<nblocks, kRedThreads, 0, s>>>((const float*)f, L, partials);
    else return cudaErrorInvalidValue;
    k_mass_final<<<1, kRedThreads, 0, s>>>(partials, nblocks, out);
    return cudaGetLastError();
}

cudaError_t launch_reinject(int prec, void* f, const Layout& L, double k, cudaStream_t s) {
    const long long N = (long long)L.Lx * L.Ly * L.Lz;
    const unsigned blocks = (unsigned)((N + 255) / 256);
    if (prec == kFP64) k_reinject<double><<<blocks, 256, 0, s>>>((double*)f, L, k);
    else if (prec == kFP32) k_reinject<float><<<blocks, 256, 0, s>>>((float*)f, L, k);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

}  // namespace lbmgb
