// Two-pass stream-collide step for float32 and 16-bit deviation storage with
// the ghost boundary (Sec. 2, Eqs. 6-10 of Milan et al., arXiv:2112.09972):
// a density pass and a collision pass, one thread per node and plane, as
// lbm_flat.cu does for float64.  Two forms:
//
//   k_row_rho / k_row_collide -- the row-tiled widths (Lx = TX in {32, 64, 128,
//       256}) for small boxes; the density pass writes the ghost shell too.
//       The cluster kernels (lbm_fast.cu) march a chunk of z planes one after
//       another, about 3 us a plane whatever the box, so a box too small to
//       fill the chip waits for that chain (10 planes at 64^3).  Here all
//       planes run at once; the second read of the populations comes from
//       L2, which such a box fits.  The centre is summed from the densities
//       in the cluster kernel's order and the node arithmetic is shared
//       (collide_core), so both store bit-identical states.
//   k_any_rho / k_any_collide -- float32 boxes of any other extents, in place
//       of the tile kernel, whose tiles sum their halo's densities again
//       (about as many nodes as the tile has) and march in z.
//
// Density array: [Lz + 2][Ly + 2][Lx + 2] of {rho_A, rho_B}, its halo holding
// the ghost densities.
#include <cuda_runtime.h>

#include <algorithm>

#include "lbm_centre.cuh"
#include "lbm_internal.h"
#include "lbm_node.cuh"
#include "lbm_pdl.cuh"
#include "lbm_tile.cuh"

namespace lbmgb {
namespace {

struct RhoGeo {
    int nx, ny;
    __host__ __device__ long long at(int x, int y, int z) const {
        return ((long long)(z + 1) * ny + y + 1) * nx + x + 1;
    }
};
RhoGeo rho_geo(const Layout& L) { return {L.Lx + 2, L.Ly + 2}; }

// Neighbour densities of one node: loads beside its own entry r.
struct RhoNb {
    const float2* __restrict__ r;
    int sy, sz;
    __device__ __forceinline__ float2 operator()(int dx, int dy, int dz) const {
        return __ldg(r + (dz * sz + dy * sy + dx));
    }
};

__global__ void k_fill2(float2* __restrict__ rho, long long n, float a, float b) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) rho[k] = make_float2(a, b);
}

// ---- row widths ----

template <int TX, typename ST>
__device__ __forceinline__ typename RowIO<TX, ST>::P3 node_planes(const ST* src, const Layout& L, int x, int y,
                                                                  int z) {
    using IO = RowIO<TX, ST>;
    if constexpr (is_dev_t<ST>::value) return IO::planes(IO::base(src, x, y), L, z, x);
    else return IO::planes(IO::base(src, x, y), L, z);
}

// The ghost populations that a row's nodes pull, written to the shell by the
// warp that holds the nodes (every ghost population streams to one fluid
// node, so none is written twice).  The partition of shell_node: x faces own
// their edges, y faces theirs with z.  Arithmetic as ghost_node and
// ghost_node_dev.
template <typename ST>
struct ShellWriter {
    ST* f;
    Layout L;
    GhostParams<float> g;
    float xc, yc, zc;
    int* d_err;

    __device__ __forceinline__ ShellWriter(ST* f_, const Layout& L_, const GhostParams<float>& g_,
                                           const CentreParts& cp, int* err)
        : f(f_), L(L_), g(g_), xc(0.f), yc(0.f), zc(0.f), d_err(err) {
        if (g.frame) xc = cp.frame[0], yc = cp.frame[1], zc = cp.frame[2];
    }
    // direction i, weight w, from ghost node (x, y, z) into fluid node (xi, yi, zi); cu(u): c_i . u
    template <typename CU>
    __device__ __forceinline__ void put(int i, float w, int x, int y, int z, int xi, int yi, int zi, CU&& cu) const {
        const GhostFlow<float> u = ghost_flow<float>(g, L, xc, yc, zc, x, y, z);
        const float c = cu(u);
        const float e[2] = {feq_of<float>(g.rho_b[0], w, c, u.u2x), feq_of<float>(g.rho_b[1], w, c, u.u2x)};
        if constexpr (is_dev_t<ST>::value) {
            using T = decltype(dev_tag(ST{}));
            const float4 r = __ldg(reinterpret_cast<const float4*>(f) + L.dev_node(xi, yi, zi));
            const unsigned short a = ghost_dev<T, float>(e[0], w, r.x), b = ghost_dev<T, float>(e[1], w, r.y);
            reinterpret_cast<unsigned*>(f)[L.dev_word(i, x, y, z)] = (unsigned)a | ((unsigned)b << 16);
        } else {
            f[L.at(0, i, x, y, z)] = e[0];
            f[L.at(1, i, x, y, z)] = e[1];
        }
        if (u.usq > g.mach2) atomicOr(d_err, 2);
    }
    // The k-th of the five directions into x plane 0 (sgn 1) or Lx - 1 (sgn
    // -1) at (y, z): c = sgn (1, {0, 1, -1, 0, 0}[k], {0, 0, 0, 1, -1}[k]).
    __device__ __forceinline__ void x_face(int k, int sgn, int y, int z) const {
        const int cy = k == 1 ? sgn : (k == 2 ? -sgn : 0), cz = k == 3 ? sgn : (k == 4 ? -sgn : 0);
        const int xi = sgn > 0 ? 0 : L.Lx - 1;
        put((k == 0 ? 1 : 5 + 2 * k) + (sgn < 0), k == 0 ? wgt<float>(1) : wgt<float>(7), xi - sgn, y - cy, z - cz, xi,
            y, z, [&](const GhostFlow<float>& u) {
                const float b = k == 1 ? u.uy : (k == 2 ? -u.uy : (k == 3 ? u.uz : (k == 4 ? -u.uz : 0.f)));
                const float c = u.ux + b;
                return sgn > 0 ? c : -c;
            });
    }
    template <int FACE>
    __device__ __forceinline__ void yz_face(int x, int y, int z) const {
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            if (!face_inward<FACE>(i)) continue;
            const int xs = x - cx_(i), ys = y - cy_(i), zs = z - cz_(i);
            if (xs < 0 || xs >= L.Lx || (FACE >= 4 && (ys < 0 || ys >= L.Ly))) continue;
            put(i, wgt<float>(i), xs, ys, zs, x, y, z,
                [&](const GhostFlow<float>& u) { return dot_c<float>(i, u.ux, u.uy, u.uz); });
        }
    }
    // All that the warp's 32 nodes of row (y, z) pull; its lanes read it after this.
    __device__ __forceinline__ void row(int x, int y, int z) const {
        const int lane = threadIdx.x & 31, x0 = x - lane;
        if (lane < 5 ? x0 == 0 : (lane < 10 && x0 + 32 == L.Lx)) x_face(lane % 5, lane < 5 ? 1 : -1, y, z);
        if (y == 0) yz_face<2>(x, y, z);
        if (y == L.Ly - 1) yz_face<3>(x, y, z);
        if (z == 0) yz_face<4>(x, y, z);
        if (z == L.Lz - 1) yz_face<5>(x, y, z);
        __syncwarp();
    }
};

constexpr int kRowRhoThreads = 128;
template <int TX>
constexpr int row_rho_rows() {
    return TX >= kRowRhoThreads ? 1 : kRowRhoThreads / TX;
}
// Also writes the ghost populations that its nodes pull, which saves a launch
// of the chain that a small box's step is (32^3 fp32 10.4 -> 9.4 us per step,
// 64^3 24.9 -> 24.1, bf16 18.9 -> 17.7; the other two-pass kernels lost more registers to it than
// the launch was worth: 37 x 29 x 23 fp32 11.7 -> 10.9 us, but 130^3 222 -> 242, and
// in float64 32^3 41 -> 57).
template <int TX, typename ST>
__global__ void __launch_bounds__(TX * row_rho_rows<TX>())
    k_row_rho(ST* src, Layout L, float2* __restrict__ rho, RhoGeo g, GhostParams<float> gp, CentreParts cp,
              int* __restrict__ d_err) {
    pdl_wait();
    pdl_trigger();
    const int x = threadIdx.x % TX, y = blockIdx.x * row_rho_rows<TX>() + threadIdx.x / TX, z = blockIdx.y;
    ShellWriter<ST>(src, L, gp, cp, d_err).row(x, y, z);
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
    auto q = node_planes<TX, ST>(src, L, x, y, z);
    asm volatile("" : "+l"(q.m), "+l"(q.o), "+l"(q.p)::"memory");  // the loads stay behind the ghost stores
    float ra, rb;
    RowIO<TX, ST>::template densities<false>(q, pol, ra, rb);
    rho[g.at(x, y, z)] = make_float2(ra, rb);
}

// the droplet indicator of collide_core
__device__ __forceinline__ float indicator(float2 r) { return fmaxf(__fdividef(r.x - r.y, r.x + r.y), 0.f); }

// The sums of the cluster kernel's CTA (y, chunk), in its order: thread x over
// the planes of its march, then the warps' shuffles.
template <int TX>
__device__ __forceinline__ void row_unit(const float2* __restrict__ rho, const RhoGeo& g, const Layout& L, int y,
                                         int chunk, int zchunk, float (&cm)[4]) {
    const int lane = threadIdx.x % 32;
    const int zc0 = chunk * zchunk, zc1 = min(zc0 + zchunk, L.Lz), n = zc1 - zc0;
    const bool down = chunk & 1;  // odd chunks march down
    const float py = (float)y - 0.5f * (float)(L.Ly - 1);
    float s[TX / 32][4] = {};
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
        const int z = down ? zc1 - 1 - k : zc0 + k;
        const float pz = (float)z - 0.5f * (float)(L.Lz - 1);
#pragma unroll
        for (int h = 0; h < TX / 32; ++h) {
            const float w = indicator(__ldg(rho + g.at(32 * h + lane, y, z)));
            const float px = (float)(32 * h + lane) - 0.5f * (float)(L.Lx - 1);
            s[h][0] += w;
            s[h][1] = fmaf(w, px, s[h][1]);
            s[h][2] = fmaf(w, py, s[h][2]);
            s[h][3] = fmaf(w, pz, s[h][3]);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float a = 0.f;
#pragma unroll
        for (int h = 0; h < TX / 32; ++h) {
            const float t = __shfl_sync(0xffffffffu, warp_total(s[h][q]), 0);
            if (lane == h) a = t;
        }
        cm[q] = warp_total(a);
    }
}

// One node per thread; the last CTAs of the grid sum the centre.  Registers
// allow 512 threads to an SM, held as CTAs of 128 (256 for the widest rows),
// so that 64^3 is 3.4 rounds of small CTAs.  (With 512 threads over the planes
// of a z chunk and their sums at the end it was four waves, each as long as
// its slowest warp and the reduction: 64^3 bf16 25.3 -> 18.9 us per step, fp32
// 30.8 -> 24.9, 32^3 fp32 11.4 -> 10.4.)
template <int TX>
constexpr int row_collide_rows() {
    return TX >= 128 ? 1 : 128 / TX;
}
template <int TX, typename ST, bool MRT>
__global__ void __launch_bounds__(TX * row_collide_rows<TX>(), 512 / (TX * row_collide_rows<TX>()))
    k_row_collide(const ST* __restrict__ src, ST* __restrict__ dst, Layout L, FastModel m,
                  const float2* __restrict__ rho, RhoGeo g, int colliders, int zchunk, int units, CentreParts cp,
                  int* __restrict__ d_err) {
    using IO = RowIO<TX, ST>;
    constexpr int R = row_collide_rows<TX>();
    pdl_wait();
    if ((int)blockIdx.x >= colliders) {
        pdl_trigger();
        centre_units<float>([&](int u, float (&cm)[4]) { row_unit<TX>(rho, g, L, u % L.Ly, u / L.Ly, zchunk, cm); }, units,
                     (int)blockIdx.x - colliders, (int)gridDim.x - colliders, cp);
        return;
    }
    const int per_plane = L.Ly / R, z = blockIdx.x / per_plane;
    const int x = threadIdx.x % TX, y = (blockIdx.x - z * per_plane) * R + threadIdx.x / TX;
    int bad = 0;
    float f[2][19], rs[2], cm[4] = {0.f, 0.f, 0.f, 0.f};
    IO::populations(node_planes<TX, ST>(src, L, x, y, z), f, rs);
    const float2* r = rho + g.at(x, y, z);
    collide_core<IO, ST, MRT>(RhoNb{r, g.nx, g.nx * g.ny}, __ldg(r), f, rs, m, IO::out(dst, L, x, y, z), cm, bad, 0.f,
                              0.f, 0.f);
    pdl_trigger();
    if (bad) atomicOr(d_err, bad);
}

template <int TX, typename ST, bool MRT>
cudaError_t launch_row_t(void* src, void* dst, void* rho, const Layout& L, const Model& m, const Grad& A,
                         const Shape& sh, CentreParts cp, int* d_err, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1] = {pdl_attribute()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.stream = s;
    cfg.gridDim = dim3(L.Ly / row_rho_rows<TX>(), L.Lz, 1);
    cfg.blockDim = dim3(TX * row_rho_rows<TX>(), 1, 1);
    const RhoGeo g = rho_geo(L);
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_row_rho<TX, ST>, (ST*)src, L, (float2*)rho, g, ghost_params<float>(m, A.a),
                                       cp, d_err);
    if (e != cudaSuccess) return e;
    constexpr int threads = TX * row_collide_rows<TX>();
    const int units = (int)(sh.grid.y * sh.grid.z), colliders = L.Ly / row_collide_rows<TX>() * L.Lz;
    cfg.gridDim = dim3(colliders + (units + threads / 32 - 1) / (threads / 32), 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    return cudaLaunchKernelEx(&cfg, k_row_collide<TX, ST, MRT>, (const ST*)src, (ST*)dst, L, fast_model(m),
                              (const float2*)rho, g, colliders, sh.zchunk, units, cp, d_err);
}

template <int TX>
cudaError_t launch_row_w(int prec, void* src, void* dst, void* rho, const Layout& L, const Model& m, const Grad& A,
                         const Shape& sh, CentreParts cp, int* d_err, cudaStream_t s) {
    if (prec == kFP32)
        return m.mrt ? launch_row_t<TX, float, true>(src, dst, rho, L, m, A, sh, cp, d_err, s)
                     : launch_row_t<TX, float, false>(src, dst, rho, L, m, A, sh, cp, d_err, s);
    if (m.mrt) return cudaErrorInvalidValue;
    if (prec == kFP16Dev) return launch_row_t<TX, Dev<__half>, false>(src, dst, rho, L, m, A, sh, cp, d_err, s);
    return launch_row_t<TX, Dev<__nv_bfloat16>, false>(src, dst, rho, L, m, A, sh, cp, d_err, s);
}

// ---- any extents, float32 ----

struct AnyIO {
    struct Out {
        float* p;
        int pitch;
    };
    template <int S, int I>
    static __device__ __forceinline__ void store(Out o, float v) {
        __stcs(o.p + (S * 19 + I) * o.pitch, v);
    }
};

constexpr int kAnyThreads = 128;
constexpr int kAnyShares = 8;  // centre sums: shares of a plane's rows, a warp each, at most one per CTA of a plane
__global__ void __launch_bounds__(kAnyThreads) k_any_rho(const float* __restrict__ src, Layout L,
                                                         float2* __restrict__ rho, RhoGeo g, int per_plane) {
    pdl_wait();
    pdl_trigger();
    const int z = blockIdx.x / per_plane, p = (blockIdx.x - z * per_plane) * kAnyThreads + threadIdx.x;
    if (p >= L.Lx * L.Ly) return;
    const int y = p / L.Lx, x = p - y * L.Lx;
    const Puller<float, float, false> P{src, L};
    float f[2][19];
    P.pull(x, y, z, f);
    rho[g.at(x, y, z)] = make_float2(sum19<float>(f[0]), sum19<float>(f[1]));
}

// The sums of one plane's share of rows, lanes over x.
__device__ __forceinline__ void any_unit(const float2* __restrict__ rho, const RhoGeo& g, const Layout& L, int u,
                                         int shares, float (&cm)[4]) {
    const int lane = threadIdx.x % 32, z = u / shares, share = u - z * shares;
    const float pz = (float)z - 0.5f * (float)(L.Lz - 1);
    for (int y = share; y < L.Ly; y += shares) {
        const float py = (float)y - 0.5f * (float)(L.Ly - 1);
#pragma unroll 4
        for (int x = lane; x < L.Lx; x += 32) {
            const float w = indicator(__ldg(rho + g.at(x, y, z)));
            cm[0] += w;
            cm[1] = fmaf(w, (float)x - 0.5f * (float)(L.Lx - 1), cm[1]);
            cm[2] = fmaf(w, py, cm[2]);
            cm[3] = fmaf(w, pz, cm[3]);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) cm[q] = warp_total(cm[q]);
}

template <bool MRT>
__global__ void __launch_bounds__(kAnyThreads, 5)
    k_any_collide(const float* __restrict__ src, float* __restrict__ dst, Layout L, FastModel m,
                  const float2* __restrict__ rho, RhoGeo g, int per_plane, int colliders, CentreParts cp,
                  int* __restrict__ d_err) {
    pdl_wait();
    if ((int)blockIdx.x >= colliders) {
        pdl_trigger();
        const int shares = min(kAnyShares, per_plane);
        centre_units<float>([&](int u, float (&cm)[4]) { any_unit(rho, g, L, u, shares, cm); }, shares * L.Lz,
                     (int)blockIdx.x - colliders, (int)gridDim.x - colliders, cp);
        return;
    }
    const int z = blockIdx.x / per_plane, p = (blockIdx.x - z * per_plane) * kAnyThreads + threadIdx.x;
    const int y = p / L.Lx, x = p - y * L.Lx;
    if (p < L.Lx * L.Ly) {
        const Puller<float, float, false> P{src, L};
        int bad = 0;
        float f[2][19], cm[4] = {0.f, 0.f, 0.f, 0.f};
        const float rs[2] = {0.f, 0.f};
        P.pull(x, y, z, f);
        const float2* r = rho + g.at(x, y, z);
        collide_core<AnyIO, float, MRT>(RhoNb{r, g.nx, g.nx * g.ny}, __ldg(r), f, rs, m,
                                        AnyIO::Out{dst + L.at(0, 0, x, y, z), L.pitch}, cm, bad, 0.f, 0.f, 0.f);
        if (bad) atomicOr(d_err, bad);
    }
    pdl_trigger();
}

}  // namespace

long long flat32_rho_bytes(const Layout& L) {
    return (long long)sizeof(float2) * (L.Lx + 2) * (L.Ly + 2) * (L.Lz + 2);
}

// The two-pass launch of a row-tiled shape keeps its grid and z chunks, by
// which the centre sums are ordered.
Shape flat_rows_shape(const Shape& rows) {
    Shape sh = rows;
    sh.flat = kFlatRows;
    sh.threads = rows.tx > 128 ? rows.tx : 128;
    sh.smem = 0;
    return sh;
}

// Any float32 box: one node per thread.
Shape flat_any_shape(const Layout& L) {
    Shape sh = {};
    const long long per_plane = ((long long)L.Lx * L.Ly + kAnyThreads - 1) / kAnyThreads;
    sh.flat = kFlatAny;
    sh.tx = L.Lx;
    sh.ty = L.Lx >= kAnyThreads ? 1 : kAnyThreads / L.Lx;
    sh.zchunk = 1;
    sh.grid = dim3((unsigned)per_plane, (unsigned)L.Lz, 1);
    sh.threads = kAnyThreads;
    return sh;
}

cudaError_t launch_flat32_fill(void* rho, const Layout& L, const Model& m, cudaStream_t s) {
    const long long n = flat32_rho_bytes(L) / (long long)sizeof(float2);
    k_fill2<<<(unsigned)((n + 255) / 256), 256, 0, s>>>((float2*)rho, n, (float)m.rho_b[0], (float)m.rho_b[1]);
    return cudaGetLastError();
}

cudaError_t launch_flat_rows(int prec, void* src, void* dst, void* rho, const Layout& L, const Model& m,
                             const Grad& A, const Shape& sh, CentreParts cp, int* d_err, cudaStream_t s) {
    switch (L.Lx) {
        case 32: return launch_row_w<32>(prec, src, dst, rho, L, m, A, sh, cp, d_err, s);
        case 64: return launch_row_w<64>(prec, src, dst, rho, L, m, A, sh, cp, d_err, s);
        case 128: return launch_row_w<128>(prec, src, dst, rho, L, m, A, sh, cp, d_err, s);
        case 256: return launch_row_w<256>(prec, src, dst, rho, L, m, A, sh, cp, d_err, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_flat_any(const void* src, void* dst, void* rho, const Layout& L, const Model& m, const Shape& sh,
                            CentreParts cp, int* d_err, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    const int per_plane = (int)sh.grid.x, colliders = (int)(sh.grid.x * sh.grid.y);
    cfg.gridDim = dim3(colliders, 1, 1);
    cfg.blockDim = dim3(kAnyThreads, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1] = {pdl_attribute()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const RhoGeo g = rho_geo(L);
    const float* f = (const float*)src;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_any_rho, f, L, (float2*)rho, g, per_plane);
    if (e != cudaSuccess) return e;
    // centre sums: four units (a share of a plane's rows) to a CTA
    const int units = std::min(kAnyShares, per_plane) * L.Lz;
    cfg.gridDim = dim3(colliders + (units + kAnyThreads / 32 - 1) / (kAnyThreads / 32), 1, 1);
    return cudaLaunchKernelEx(&cfg, m.mrt ? k_any_collide<true> : k_any_collide<false>, f, (float*)dst, L,
                              fast_model(m), (const float2*)rho, g, per_plane, colliders, cp, d_err);
}

}  // namespace lbmgb
