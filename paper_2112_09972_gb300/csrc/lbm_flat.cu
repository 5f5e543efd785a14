// Two-pass stream-collide step for float64 storage: a density pass and a
// collision pass, each with one thread per node and no march (Sec. 2, Eqs.
// 6-10 of Milan et al., arXiv:2112.09972).
//
//   k_flat_rho     -- post-streaming densities of every node (Eq. 6) into a
//                     padded array [Lz + 2][Ly + 2][Lx + 2] of {rho_A, rho_B};
//                     its halo holds the ghost densities (ghost boundary,
//                     written once) or the periodic images
//   k_flat_collide -- pulls the populations, reads the node's and its
//                     neighbours' densities, Shan-Chen force (Eq. 7),
//                     velocity shift, BGK or MRT collision, store, and the
//                     droplet's centre of mass
//
// What bounds it.  This GPU's FP64 pipe issues one warp instruction per 16
// cycles and SM, so a float64 node update is bound by its FP64 instructions,
// not by memory: the 608 bytes of 512 nodes take 46 ns at the measured copy
// bandwidth, their 340 FP64 instructions a node 290 ns (128^3: 379 ns
// measured).  The marched tile kernel sums every density about twice (the tile's halo, and the planes
// before and after each z chunk) and evaluates each equilibrium on its own,
// 560 instructions per node.  Here each density is summed once (the second
// read of the populations costs bandwidth that is idle), opposite
// directions share their equilibria, and the launch covers the chip for any
// box: one node per thread instead of a z march per tile.  Measured per step
// against the tile kernel: 32^3 34 us (178), 64^3 191 us (365), 128^3 1551 us
// (3174), 37 x 29 x 23 29 us (160); float64 storage therefore takes these
// kernels at every size.
#include <cuda_runtime.h>

#include <algorithm>

#include "lbm_eigen.cuh"
#include "lbm_internal.h"
#include "lbm_lattice.cuh"
#include "lbm_pdl.cuh"
#include "lbm_tile.cuh"

namespace lbmgb {
namespace {

constexpr int kFlatPerSM = 6;     // resident CTAs of the collision pass
constexpr int kFlatThreads = 64;  // two warps: CTAs spread evenly over the SMs, whose FP64 pipes are the bound

// The padded density array: node (x, y, z) at ((z + 1) ny + y + 1) nx + x + 1.
struct RhoGeo {
    int nx, ny;
    __host__ __device__ long long at(int x, int y, int z) const {
        return ((long long)(z + 1) * ny + y + 1) * nx + x + 1;
    }
};
RhoGeo rho_geo(const Layout& L) { return {L.Lx + 2, L.Ly + 2}; }

struct FlatModel {
    double inv_tau[2], omit[2];  // 1 / tau, 1 - 1 / tau
    double sh[2];                // -G tau / 36: the velocity shift per unit of the other component's force sum
    double mrt[5];
};

FlatModel flat_model(const Model& m) {
    FlatModel r;
    for (int s = 0; s < 2; ++s) {
        r.inv_tau[s] = 1.0 / m.tau[s];
        r.omit[s] = 1.0 - 1.0 / m.tau[s];
        r.sh[s] = -m.G * m.tau[s] / 36.0;
    }
    for (int k = 0; k < 5; ++k) r.mrt[k] = m.mrt_rates[k];
    return r;
}

__global__ void k_flat_fill(double2* __restrict__ rho, long long n, double a, double b) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) rho[k] = make_double2(a, b);
}

template <bool PER>
__global__ void __launch_bounds__(kFlatThreads) k_flat_rho(const double* __restrict__ src, Layout L,
                                                           double2* __restrict__ rho, RhoGeo g, int zchunk) {
    pdl_wait();
    pdl_trigger();
    const int p = blockIdx.x * kFlatThreads + threadIdx.x;
    if (p >= L.Lx * L.Ly) return;
    const int y = p / L.Lx, x = p - y * L.Lx;
    const Puller<double, double, PER> P{src, L};
    const int z1 = min(((int)blockIdx.y + 1) * zchunk, L.Lz);
    for (int z = blockIdx.y * zchunk; z < z1; ++z) {
        double f[2][19];
        P.pull(x, y, z, f);
        const double2 r = make_double2(sum19<double>(f[0]), sum19<double>(f[1]));
        rho[g.at(x, y, z)] = r;
        if (PER) {  // the images in the halo (the force reads no corner)
            const int ix = x == 0 ? L.Lx : (x == L.Lx - 1 ? -1 : x);
            const int iy = y == 0 ? L.Ly : (y == L.Ly - 1 ? -1 : y);
            const int iz = z == 0 ? L.Lz : (z == L.Lz - 1 ? -1 : z);
            if (ix != x) rho[g.at(ix, y, z)] = r;
            if (iy != y) rho[g.at(x, iy, z)] = r;
            if (iz != z) rho[g.at(x, y, iz)] = r;
            if (ix != x && iy != y) rho[g.at(ix, iy, z)] = r;
            if (ix != x && iz != z) rho[g.at(ix, y, iz)] = r;
            if (iy != y && iz != z) rho[g.at(x, iy, iz)] = r;
        }
    }
}

__device__ __forceinline__ bool finite64(double v) {  // on the integer pipe
    return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
}

// Collision of one node from its pulled populations f and the density array
// (r: the node's entry; rows sy, planes sz apart), stored to dst.
template <bool MRT>
__device__ __forceinline__ void flat_node(const double2* __restrict__ r, int sy, int sz, const FlatModel& m,
                                          const double (&f)[2][19], double* __restrict__ o, long long pitch,
                                          double2& rho) {
    // momentum (Eq. 6) of both components, opposite pairs differenced first,
    // combined with the weights of the common velocity
    double j[2][3];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        double v[3];
        bool set[3] = {false, false, false};
        auto gather = [&](int a, int c, double d) {  // v[a] += c d
            if (c == 0) return;
            v[a] = set[a] ? (c > 0 ? v[a] + d : v[a] - d) : d;  // (the first direction of each sum has c = 1)
            set[a] = true;
        };
#pragma unroll
        for (int i = 1; i < 19; i += 2) {
            const double d = f[s][i] - f[s][i + 1];
            gather(0, cx_(i), d);
            gather(1, cy_(i), d);
            gather(2, cz_(i), d);
        }
        j[s][0] = v[0]; j[s][1] = v[1]; j[s][2] = v[2];
    }
    // Shan-Chen force sums (Eq. 7) in units of the edge weight 1/36
    double acc[2][3];
#pragma unroll
    for (int i = 1; i < 19; i += 2) {
        const int off = cz_(i) * sz + cy_(i) * sy + cx_(i);
        const double2 a = r[off], b = r[-off];
        const double dA = a.x - b.x, dB = a.y - b.y;
        if (i < 7) {  // axis directions come first, one per sum, with weight 2
            acc[0][i / 2] = dA + dA;
            acc[1][i / 2] = dB + dB;
            continue;
        }
        if (cx_(i)) { acc[0][0] += cx_(i) > 0 ? dA : -dA; acc[1][0] += cx_(i) > 0 ? dB : -dB; }
        if (cy_(i)) { acc[0][1] += cy_(i) > 0 ? dA : -dA; acc[1][1] += cy_(i) > 0 ? dB : -dB; }
        if (cz_(i)) { acc[0][2] += cz_(i) > 0 ? dA : -dA; acc[1][2] += cz_(i) > 0 ? dB : -dB; }
    }
    rho = *r;
    const double den = rho.x * m.inv_tau[0] + rho.y * m.inv_tau[1];
    // (rcp64 between 2^-100 and 2^100)
    const double rden =
        (unsigned)__double2hiint(den) - (923u << 20) < (200u << 20) ? rcp64(den) : 1.0 / den;
    double up[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) up[a] = (j[0][a] * m.inv_tau[0] + j[1][a] * m.inv_tau[1]) * rden;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const double rs = s ? rho.y : rho.x;
        const double ux = fma(m.sh[s], acc[1 - s][0], up[0]);
        const double uy = fma(m.sh[s], acc[1 - s][1], up[1]);
        const double uz = fma(m.sh[s], acc[1 - s][2], up[2]);
        double* os = o + (long long)(19 * s) * pitch;
        double others = 0.0;
        if constexpr (MRT) {
            const double u2x = 1.5 * (ux * ux + uy * uy + uz * uz);
            double dv[19], out[19];
#pragma unroll
            for (int i = 0; i < 19; ++i) dv[i] = f[s][i] - feq<double>(i, rs, ux, uy, uz, u2x);
            mrt_relax<double>(f[s], dv, m.inv_tau[s], m.mrt, out);
#pragma unroll
            for (int i = 1; i < 19; i += 2) {
                os[i * pitch] = out[i];
                os[(i + 1) * pitch] = out[i + 1];
                others += out[i] + out[i + 1];
            }
        } else {
            // with v = 1.5 u and c = c_i . v, the even and odd parts of
            // f_eq / tau of a pair are e base + c (2 e c) and 2 e c
            const double base = fma(-1.5, ux * ux + uy * uy + uz * uz, 1.0);
            const double ir = m.inv_tau[s] * rs;
            const double vx = 1.5 * ux, vy = 1.5 * uy, vz = 1.5 * uz;
            const double e2A = ir * (1.0 / 9.0), e2E = ir * (1.0 / 18.0);  // 2 e of axis and edge directions
            const double ib = ir * base;
            const double ebA = ib * (1.0 / 18.0), ebE = ib * (1.0 / 36.0);
            const double om = m.omit[s];
#pragma unroll
            for (int i = 1; i < 19; i += 2) {
                const double c = dot_c<double>(i, vx, vy, vz);
                const double od = (i < 7 ? e2A : e2E) * c;
                const double ev = fma(c, od, i < 7 ? ebA : ebE);
                const double oa = fma(om, f[s][i], ev + od), ob = fma(om, f[s][i + 1], ev - od);
                os[i * pitch] = oa;
                os[(i + 1) * pitch] = ob;
                others += oa + ob;
            }
        }
        // the rest population closes the mass balance exactly (sum of outputs
        // = rho), as the tile kernel's does: the sum's 36 additions a node
        // took 64^3 from 174 to 191 us per step
        os[0] = rs - others;
    }
}

// The centre sums of a z chunk's share of rows, lanes over x.  w = max(phi, 0):
// the division and the sums only in warps where a phi is not negative.
constexpr int kFlatShares = 8;  // a warp each, at most one per CTA of a chunk
__device__ __forceinline__ void flat_unit(const double2* __restrict__ rho, const RhoGeo& g, const Layout& L, int u,
                                          int shares, int zchunk, double (&cm)[4]) {
    const int lane = threadIdx.x % 32, chunk = u / shares, share = u - chunk * shares;
    const int z1 = min((chunk + 1) * zchunk, L.Lz);
    bool any = false;
    for (int z = chunk * zchunk; z < z1; ++z)
        for (int y = share; y < L.Ly; y += shares)
            for (int x = lane; x < L.Lx; x += 32) {
                const double2 r = __ldg(rho + g.at(x, y, z));
                const double d = r.x - r.y, t = r.x + r.y;
                if ((__double2hiint(d) ^ __double2hiint(t)) >= 0) {
                    const double w = fmax(d / t, 0.0);
                    cm[0] += w;
                    cm[1] = fma(w, x - 0.5 * (L.Lx - 1), cm[1]);
                    cm[2] = fma(w, y - 0.5 * (L.Ly - 1), cm[2]);
                    cm[3] = fma(w, z - 0.5 * (L.Lz - 1), cm[3]);
                    any = true;
                }
            }
    if (!__any_sync(0xffffffffu, any)) return;
#pragma unroll
    for (int q = 0; q < 4; ++q) cm[q] = warp_total(cm[q]);
}

// `centres` CTAs from `centre0` on sum the centre of mass from the density
// array (against sums at the end of every colliding CTA, per step and before
// the rest population closed the mass: 32^3 41.9 -> 31.9 us, 37 x 29 x 23 36.1 ->
// 26.9, 64^3 195 -> 174, 128^3 1433 -> 1408).
template <bool PER, bool MRT>
__global__ void __launch_bounds__(kFlatThreads, kFlatPerSM)
    k_flat_collide(const double* __restrict__ src, double* __restrict__ dst, Layout L, FlatModel m,
                   const double2* __restrict__ rho, RhoGeo g, int per_plane, int zchunk, int units, int centre0, int centres,
                   CentreParts cp, int* __restrict__ d_err) {
    pdl_wait();
    const int own = (int)blockIdx.x - centre0;
    if (own >= 0 && own < centres) {
        pdl_trigger();
        const int shares = min(kFlatShares, per_plane);
        centre_units<double>([&](int u, double (&cm)[4]) { flat_unit(rho, g, L, u, shares, zchunk, cm); }, units,
                             own, centres, cp);
        return;
    }
    const int cta = own < 0 ? (int)blockIdx.x : (int)blockIdx.x - centres, chunk = cta / per_plane;
    const int p = (cta - chunk * per_plane) * kFlatThreads + threadIdx.x;
    const int y = p / L.Lx, x = p - y * L.Lx;
    const Puller<double, double, PER> P{src, L};
    bool bad = false;
    if (p < L.Lx * L.Ly) {
        const int z1 = min((chunk + 1) * zchunk, L.Lz);
        for (int z = chunk * zchunk; z < z1; ++z) {
            double f[2][19];
            P.pull(x, y, z, f);
            double2 r;
            flat_node<MRT>(rho + g.at(x, y, z), g.nx, g.nx * g.ny, m, f, dst + L.at(0, 0, x, y, z), L.pitch, r);
            bad |= !(finite64(r.x) && finite64(r.y));
        }
    }
    pdl_trigger();
    if (bad) atomicOr(d_err, 1);
}

}  // namespace

long long flat_rho_bytes(const Layout& L) {
    return (long long)sizeof(double2) * (L.Lx + 2) * (L.Ly + 2) * (L.Lz + 2);
}

// One node per thread; the z extent is cut so that the launch has at most
// about 16 CTAs per SM, which bounds the centre-of-mass partials (small boxes:
// one plane per CTA).
Shape flat_shape(const Layout& L, int num_sms) {
    Shape sh = {};
    const long long per_plane = ((long long)L.Lx * L.Ly + kFlatThreads - 1) / kFlatThreads;
    const long long want = 16LL * (num_sms > 0 ? num_sms : 152);
    long long zc = (per_plane * L.Lz + want - 1) / want;
    if (zc < 1) zc = 1;
    while ((L.Lz + zc - 1) / zc > 65535) ++zc;
    sh.flat = kFlat64;
    // last where the colliders all run at once, so that the sums land on the SMs with one collider less (first, they
    // pushed a fifth one on some: 32^3 39.5 us against 31.5); first where they do not, so that no long sum is left over
    // (last: 128^3 1905 us against 1411)
    sh.centre_first = per_plane * ((L.Lz + zc - 1) / zc) > kFlatPerSM * (num_sms > 0 ? num_sms : 152);
    sh.tx = L.Lx;
    sh.ty = L.Lx >= kFlatThreads ? 1 : kFlatThreads / L.Lx;
    sh.zchunk = (int)zc;
    sh.grid = dim3((unsigned)per_plane, (unsigned)((L.Lz + zc - 1) / zc), 1);
    sh.threads = kFlatThreads;
    return sh;
}

cudaError_t launch_flat_fill(void* rho, const Layout& L, const Model& m, cudaStream_t s) {
    const long long n = flat_rho_bytes(L) / (long long)sizeof(double2);
    k_flat_fill<<<(unsigned)((n + 255) / 256), 256, 0, s>>>((double2*)rho, n, m.rho_b[0], m.rho_b[1]);
    return cudaGetLastError();
}

cudaError_t launch_flat(const void* src, void* dst, void* rho, const Layout& L, const Model& m, const Shape& sh,
                        CentreParts cp, int* d_err, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = sh.grid;
    cfg.blockDim = dim3(kFlatThreads, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1] = {pdl_attribute()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const RhoGeo g = rho_geo(L);
    const FlatModel fm = flat_model(m);
    const double* f = (const double*)src;
    double2* r = (double2*)rho;
    cudaError_t e = cudaLaunchKernelEx(&cfg, m.periodic ? k_flat_rho<true> : k_flat_rho<false>, f, L, r, g, sh.zchunk);
    if (e != cudaSuccess) return e;
    auto k = m.periodic ? (m.mrt ? k_flat_collide<true, true> : k_flat_collide<true, false>)
                        : (m.mrt ? k_flat_collide<false, true> : k_flat_collide<false, false>);
    const int per_plane = (int)sh.grid.x, units = std::min(kFlatShares, per_plane) * (int)sh.grid.y;
    const int colliders = (int)(sh.grid.x * sh.grid.y);
    const int centres = std::min((units + kFlatThreads / 32 - 1) / (kFlatThreads / 32), 512);
    const int centre0 = sh.centre_first ? 0 : colliders;
    cfg.gridDim = dim3(colliders + centres, 1, 1);
    return cudaLaunchKernelEx(&cfg, k, f, (double*)dst, L, fm, (const double2*)r, g, per_plane, sh.zchunk, units,
                              centre0, centres, cp, d_err);
}

}  // namespace lbmgb
