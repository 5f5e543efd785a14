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
//       (about as many nodes as the tile has) and march in z.  The node
//       arithmetic (tile_collide) and the order of the centre's sums are the
//       tile kernel's, so both store bit-identical states here too.
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
// the launch was worth: tried in them, it took 37 x 29 x 23 fp32 from 11.7 to 10.9
// us, but 130^3 from 222 to 242, and float64 32^3 from 41 to 57).
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

constexpr int kAnyThreads = 128;
constexpr int kAnyPerSM = 5;  // resident CTAs of the collision pass
int any_per_plane(const Layout& L) { return (L.Lx * L.Ly + kAnyThreads - 1) / kAnyThreads; }
int any_colliders(const Layout& L) { return any_per_plane(L) * L.Lz; }
constexpr int kAnyTileWarps = 16;  // warps of the tile kernel's largest CTA
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

// The tile kernel's launch for this box: tiles of tx x ty nodes, z chunks.
struct AnyTiles {
    int tx, ty, zchunk, nx, ny, ctas;  // nx, ny: tiles along x and y
};

// Centre of mass from the density array: one CTA for each CTA of the tile
// kernel, its sums in that kernel's order -- thread t of the tile over the
// planes of its march, the warps' shuffles, the shuffle over warps, and the
// CTAs in order at the end (centre_reduce).  In small boxes this chain is the
// longest of the launch, and its loads are what it waits for: sixteen of a
// lane's in flight instead of one 37 x 29 x 23 13.4 -> 10.6 us per step, 60 x 50 x
// 44 16.8 -> 14.6.
__device__ void any_centre(const float2* __restrict__ rho, const RhoGeo& g, const Layout& L, const AnyTiles& a, int u,
                           const CentreParts& cp) {
    __shared__ float sums[kAnyTileWarps][4];
    __shared__ unsigned last;
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    const int chunk = u / (a.nx * a.ny), tile = u - chunk * (a.nx * a.ny);
    const int x0 = tile % a.nx * a.tx, y0 = tile / a.nx * a.ty;
    const int z0 = chunk * a.zchunk, z1 = min(z0 + a.zchunk, L.Lz);
    const int threads = a.tx * a.ty, warps = (threads + 31) / 32;
    float* parts = reinterpret_cast<float*>(cp.p);
    // warp w takes the tile's warps w, w + 4, ... side by side, so that their loads are in flight together
    constexpr int H = kAnyTileWarps / (kAnyThreads / 32);
    float cm[H][4] = {}, px[H], py[H];
    const float2* r[H];
    bool in[H];
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const int t = 32 * (warp + k * (kAnyThreads / 32)) + lane, x = x0 + t % a.tx, y = y0 + t / a.tx;
        in[k] = t < threads && x < L.Lx && y < L.Ly;
        px[k] = (float)x - 0.5f * (float)(L.Lx - 1);
        py[k] = (float)y - 0.5f * (float)(L.Ly - 1);
        r[k] = rho + (in[k] ? g.at(x, y, z0) : 0);
    }
    const int sz = g.nx * g.ny;
    constexpr int U = 4;  // planes read before the first of them is summed
    for (int zu = z0; zu < z1; zu += U) {
        float2 v[U][H];
#pragma unroll
        for (int i = 0; i < U; ++i)
#pragma unroll
            for (int k = 0; k < H; ++k) v[i][k] = __ldg(r[k] + (long long)(min(zu + i, z1 - 1) - z0) * sz);
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const float pz = (float)(zu + i) - 0.5f * (float)(L.Lz - 1);
#pragma unroll
            for (int k = 0; k < H; ++k) {
                const float rk[2] = {v[i][k].x, v[i][k].y};
                // (a droplet's nodes: elsewhere w = 0 and the sums stay as they are)
                if (in[k] && zu + i < z1 && (rk[0] > rk[1]) == (rk[0] + rk[1] > 0.f))
                    droplet_sums<float>(rk, px[k], py[k], pz, cm[k]);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < H; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float s = warp_total(cm[k][q]);
            if (lane == 0) sums[warp + k * (kAnyThreads / 32)][q] = s;
        }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float s = warp_total(lane < warps ? sums[lane][q] : 0.f);
            if (lane == 0) parts[4LL * u + q] = s;
        }
        if (lane == 0) {
            __threadfence();
            last = atomicAdd(cp.counter, 1u) == (unsigned)a.ctas - 1u ? 1u : 0u;
        }
        __syncwarp();
        if (last) centre_total<float>(parts, (unsigned)a.ctas, cp.counter, cp.sum, cp.frame);
    }
}

// a.ctas CTAs from `centre0` on sum the centre, the others take a node a thread.
template <bool MRT>
__global__ void __launch_bounds__(kAnyThreads, kAnyPerSM)
    k_any_collide(const float* __restrict__ src, float* __restrict__ dst, Layout L, ModelC<float> m,
                  const float2* __restrict__ rho, RhoGeo g, int per_plane, AnyTiles a, int centre0, CentreParts cp,
                  int* __restrict__ d_err) {
    pdl_wait();
    const int own = (int)blockIdx.x - centre0;
    if (own >= 0 && own < a.ctas) {
        pdl_trigger();
        any_centre(rho, g, L, a, own, cp);
        return;
    }
    const int cta = own < 0 ? (int)blockIdx.x : (int)blockIdx.x - a.ctas;
    const int z = cta / per_plane, p = (cta - z * per_plane) * kAnyThreads + threadIdx.x;
    const int y = p / L.Lx, x = p - y * L.Lx;
    if (p < L.Lx * L.Ly) {
        const Puller<float, float, false> P{src, L};
        float f[2][19];
        P.pull(x, y, z, f);
        const RhoNb near{rho + g.at(x, y, z), g.nx, g.nx * g.ny};
        const float2 own2 = near(0, 0, 0);
        const float r[2] = {own2.x, own2.y};
        float* o = dst + L.at(0, 0, x, y, z);
        auto nb = [&](int s, int dx, int dy, int dz) {
            const float2 v = near(dx, dy, dz);
            return s ? v.y : v.x;
        };
        tile_collide<float, MRT>(f, r, m, nb, [&](int s, const float (&out)[19]) {
            float others = 0.f;  // the rest population closes the mass balance
#pragma unroll
            for (int i = 1; i < 19; ++i) {
                __stcs(o + (19 * s + i) * L.pitch, out[i]);
                others += out[i];
            }
            __stcs(o + 19 * s * L.pitch, r[s] - others);
        });
        if (!(isfinite(r[0]) && isfinite(r[1]))) atomicOr(d_err, 1);
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

// Any float32 box: one node per thread.  Keeps the tile kernel's shape, by
// which the centre sums are ordered.  Their CTAs come first where the grid
// takes more than one wave, so that none is left over at its end (per step,
// first against last: 60 x 50 x 44 17.0 us and 19.2, 130^3 206 and 240; 37 x 29 x
// 23, one wave, 13.9 and 13.8).
Shape flat_any_shape(const Layout& L, const Shape& tile, int num_sms) {
    Shape sh = tile;
    sh.flat = kFlatAny;
    sh.centre_first = any_colliders(L) > kAnyPerSM * (num_sms > 0 ? num_sms : 152);
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
    const int per_plane = any_per_plane(L), colliders = any_colliders(L);
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
    const AnyTiles a = {sh.tx, sh.ty, sh.zchunk, (int)sh.grid.x, (int)sh.grid.y,
                        (int)(sh.grid.x * sh.grid.y * sh.grid.z)};
    cfg.gridDim = dim3(colliders + a.ctas, 1, 1);
    return cudaLaunchKernelEx(&cfg, m.mrt ? k_any_collide<true> : k_any_collide<false>, f, (float*)dst, L,
                              model_c<float>(m), (const float2*)rho, g, per_plane, a,
                              sh.centre_first ? 0 : colliders, cp, d_err);
}

}  // namespace lbmgb
