// Two-pass stream-collide step for float32 and 16-bit deviation storage with
// the ghost boundary (Sec. 2, Eqs. 6-10 of Milan et al., arXiv:2112.09972):
// a density pass and a collision pass, one thread per node and plane, as
// lbm_flat.cu does for float64.  Two forms:
//
//   k_row_rho / k_row_collide -- the row-tiled widths (Lx = TX in {32, 64, 128,
//       256}) for small boxes.  The cluster kernels (lbm_fast.cu) march a
//       chunk of z planes one after another, about 3 us a plane whatever the
//       box, so a box too small to fill the chip waits for that chain (10
//       planes at 64^3).  Here all planes of a chunk run at once; the second
//       read of the populations comes from L2, which such a box fits.  A CTA
//       has the row and the z chunk of a CTA of the cluster kernel, sums each
//       node's droplet indicator in that kernel's order and shares its node
//       arithmetic (collide_core), so both store bit-identical states.
//   k_any_rho / k_any_collide -- float32 boxes of any other extents, in place
//       of the tile kernel, whose tiles sum their halo's densities again
//       (about as many nodes as the tile has) and march in z.
//
// Density array: [Lz + 2][Ly + 2][Lx + 2] of {rho_A, rho_B}, its halo holding
// the ghost densities.
#include <cuda_runtime.h>

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

constexpr int kRowRhoThreads = 128;
template <int TX>
constexpr int row_rho_rows() {
    return TX >= kRowRhoThreads ? 1 : kRowRhoThreads / TX;
}
template <int TX, typename ST>
__global__ void __launch_bounds__(TX * row_rho_rows<TX>()) k_row_rho(const ST* __restrict__ src, Layout L,
                                                                     float2* __restrict__ rho, RhoGeo g) {
    pdl_wait();
    pdl_trigger();
    const int x = threadIdx.x % TX, y = blockIdx.x * row_rho_rows<TX>() + threadIdx.x / TX, z = blockIdx.y;
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
    float ra, rb;
    RowIO<TX, ST>::densities(node_planes<TX, ST>(src, L, x, y, z), pol, ra, rb);
    rho[g.at(x, y, z)] = make_float2(ra, rb);
}

// Grid and z chunks of the cluster kernel (1, Ly, chunks); TX x ZL threads,
// plane k of the chunk's march on z lane k mod ZL.
template <int TX, typename ST, bool MRT>
__global__ void __launch_bounds__(512) k_row_collide(const ST* __restrict__ src, ST* __restrict__ dst, Layout L,
                                                     FastModel m, const float2* __restrict__ rho, RhoGeo g,
                                                     int zchunk, CentreParts cp, int* __restrict__ d_err) {
    using IO = RowIO<TX, ST>;
    extern __shared__ float wk[];  // [zchunk][TX] droplet indicators, in march order
    __shared__ float red[4 * 16];
    pdl_wait();
    const int x = threadIdx.x % TX, zl = threadIdx.x / TX, ZL = blockDim.x / TX, y = blockIdx.y;
    const int zc0 = blockIdx.z * zchunk, zc1 = min(zc0 + zchunk, L.Lz), n = zc1 - zc0;
    const bool down = blockIdx.z & 1;  // odd chunks march down, as the cluster kernel's do
    const float px = (float)x - 0.5f * (float)(L.Lx - 1), py = (float)y - 0.5f * (float)(L.Ly - 1);
    int bad = 0;
    for (int k = zl; k < n; k += ZL) {
        const int z = down ? zc1 - 1 - k : zc0 + k;
        float f[2][19], rs[2], cw[4] = {0.f, 0.f, 0.f, 0.f};
        IO::populations(node_planes<TX, ST>(src, L, x, y, z), f, rs);
        const float2* r = rho + g.at(x, y, z);
        collide_core<IO, ST, MRT>(RhoNb{r, g.nx, g.nx * g.ny}, __ldg(r), f, rs, m, IO::out(dst, L, x, y, z), cw, bad,
                                  px, py, (float)z - 0.5f * (float)(L.Lz - 1));
        wk[k * TX + x] = cw[0];
    }
    pdl_trigger();
    if (bad) atomicOr(d_err, bad);
    __syncthreads();
    // the sums of the cluster kernel's thread x, in its order
    float cm[4] = {0.f, 0.f, 0.f, 0.f};
    if (zl == 0)
        for (int k = 0; k < n; ++k) {
            const float w = wk[k * TX + x], pz = (float)(down ? zc1 - 1 - k : zc0 + k) - 0.5f * (float)(L.Lz - 1);
            cm[0] += w;
            cm[1] = fmaf(w, px, cm[1]);
            cm[2] = fmaf(w, py, cm[2]);
            cm[3] = fmaf(w, pz, cm[3]);
        }
    centre_epilogue(cm, cp, red);
}

template <int TX, typename ST, bool MRT>
cudaError_t launch_row_t(const void* src, void* dst, void* rho, const Layout& L, const Model& m, const Shape& sh,
                         CentreParts cp, int* d_err, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1] = {pdl_attribute()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.stream = s;
    cfg.gridDim = dim3(L.Ly / row_rho_rows<TX>(), L.Lz, 1);
    cfg.blockDim = dim3(TX * row_rho_rows<TX>(), 1, 1);
    const RhoGeo g = rho_geo(L);
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_row_rho<TX, ST>, (const ST*)src, L, (float2*)rho, g);
    if (e != cudaSuccess) return e;
    cfg.gridDim = sh.grid;
    cfg.blockDim = dim3(sh.threads, 1, 1);
    cfg.dynamicSmemBytes = sh.smem;
    return cudaLaunchKernelEx(&cfg, k_row_collide<TX, ST, MRT>, (const ST*)src, (ST*)dst, L, fast_model(m),
                              (const float2*)rho, g, sh.zchunk, cp, d_err);
}

template <int TX>
cudaError_t launch_row_w(int prec, const void* src, void* dst, void* rho, const Layout& L, const Model& m,
                         const Shape& sh, CentreParts cp, int* d_err, cudaStream_t s) {
    if (prec == kFP32)
        return m.mrt ? launch_row_t<TX, float, true>(src, dst, rho, L, m, sh, cp, d_err, s)
                     : launch_row_t<TX, float, false>(src, dst, rho, L, m, sh, cp, d_err, s);
    if (m.mrt) return cudaErrorInvalidValue;
    if (prec == kFP16Dev) return launch_row_t<TX, Dev<__half>, false>(src, dst, rho, L, m, sh, cp, d_err, s);
    return launch_row_t<TX, Dev<__nv_bfloat16>, false>(src, dst, rho, L, m, sh, cp, d_err, s);
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
__global__ void __launch_bounds__(kAnyThreads) k_any_rho(const float* __restrict__ src, Layout L,
                                                         float2* __restrict__ rho, RhoGeo g, int zchunk) {
    pdl_wait();
    pdl_trigger();
    const int p = blockIdx.x * kAnyThreads + threadIdx.x;
    if (p >= L.Lx * L.Ly) return;
    const int y = p / L.Lx, x = p - y * L.Lx;
    const Puller<float, float, false> P{src, L};
    const int z1 = min(((int)blockIdx.y + 1) * zchunk, L.Lz);
    for (int z = blockIdx.y * zchunk; z < z1; ++z) {
        float f[2][19];
        P.pull(x, y, z, f);
        rho[g.at(x, y, z)] = make_float2(sum19<float>(f[0]), sum19<float>(f[1]));
    }
}

template <bool MRT>
__global__ void __launch_bounds__(kAnyThreads, 5)
    k_any_collide(const float* __restrict__ src, float* __restrict__ dst, Layout L, FastModel m,
                  const float2* __restrict__ rho, RhoGeo g, int zchunk, CentreParts cp, int* __restrict__ d_err) {
    __shared__ float scratch[4 * (kAnyThreads / 32)];
    pdl_wait();
    const int p = blockIdx.x * kAnyThreads + threadIdx.x;
    const int y = p / L.Lx, x = p - y * L.Lx;
    const Puller<float, float, false> P{src, L};
    float cm[4] = {0.f, 0.f, 0.f, 0.f};
    int bad = 0;
    if (p < L.Lx * L.Ly) {
        const float px = (float)x - 0.5f * (float)(L.Lx - 1), py = (float)y - 0.5f * (float)(L.Ly - 1);
        const int z1 = min(((int)blockIdx.y + 1) * zchunk, L.Lz);
        for (int z = blockIdx.y * zchunk; z < z1; ++z) {
            float f[2][19];
            const float rs[2] = {0.f, 0.f};
            P.pull(x, y, z, f);
            const float2* r = rho + g.at(x, y, z);
            collide_core<AnyIO, float, MRT>(RhoNb{r, g.nx, g.nx * g.ny}, __ldg(r), f, rs, m,
                                            AnyIO::Out{dst + L.at(0, 0, x, y, z), L.pitch}, cm, bad, px, py,
                                            (float)z - 0.5f * (float)(L.Lz - 1));
        }
    }
    pdl_trigger();
    if (bad) atomicOr(d_err, bad);
    const unsigned cta = blockIdx.y * gridDim.x + blockIdx.x, total = gridDim.x * gridDim.y;
    const bool any = __syncthreads_or(cm[0] != 0.f) != 0;
    centre_reduce_last<kAnyThreads>(cm, any, reinterpret_cast<float*>(cp.p), cta, total, cp.counter, cp.sum, cp.frame,
                                    scratch);
}

}  // namespace

long long flat32_rho_bytes(const Layout& L) {
    return (long long)sizeof(float2) * (L.Lx + 2) * (L.Ly + 2) * (L.Lz + 2);
}

// The two-pass launch of a row-tiled shape: its grid and z chunks, with as
// many planes of a chunk at once as 512 threads hold.
Shape flat_rows_shape(const Shape& rows) {
    Shape sh = rows;
    int zl = 512 / rows.tx;
    if (zl > rows.zchunk) zl = rows.zchunk;
    sh.flat = kFlatRows;
    sh.threads = zl * rows.tx;
    sh.smem = sizeof(float) * (size_t)rows.zchunk * rows.tx;
    return sh;
}

// Any float32 box: one node per thread; the z extent is cut so that the
// launch has at most about 32 CTAs per SM (the last CTA sums their partials).
Shape flat_any_shape(const Layout& L, int num_sms) {
    Shape sh = {};
    const long long per_plane = ((long long)L.Lx * L.Ly + kAnyThreads - 1) / kAnyThreads;
    const long long want = 32LL * (num_sms > 0 ? num_sms : 152);
    long long zc = (per_plane * L.Lz + want - 1) / want;
    if (zc < 1) zc = 1;
    sh.flat = kFlatAny;
    sh.tx = L.Lx;
    sh.ty = L.Lx >= kAnyThreads ? 1 : kAnyThreads / L.Lx;
    sh.zchunk = (int)zc;
    sh.grid = dim3((unsigned)per_plane, (unsigned)((L.Lz + zc - 1) / zc), 1);
    sh.threads = kAnyThreads;
    return sh;
}

cudaError_t launch_flat32_fill(void* rho, const Layout& L, const Model& m, cudaStream_t s) {
    const long long n = flat32_rho_bytes(L) / (long long)sizeof(float2);
    k_fill2<<<(unsigned)((n + 255) / 256), 256, 0, s>>>((float2*)rho, n, (float)m.rho_b[0], (float)m.rho_b[1]);
    return cudaGetLastError();
}

cudaError_t launch_flat_rows(int prec, const void* src, void* dst, void* rho, const Layout& L, const Model& m,
                             const Shape& sh, CentreParts cp, int* d_err, cudaStream_t s) {
    switch (L.Lx) {
        case 32: return launch_row_w<32>(prec, src, dst, rho, L, m, sh, cp, d_err, s);
        case 64: return launch_row_w<64>(prec, src, dst, rho, L, m, sh, cp, d_err, s);
        case 128: return launch_row_w<128>(prec, src, dst, rho, L, m, sh, cp, d_err, s);
        case 256: return launch_row_w<256>(prec, src, dst, rho, L, m, sh, cp, d_err, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_flat_any(const void* src, void* dst, void* rho, const Layout& L, const Model& m, const Shape& sh,
                            CentreParts cp, int* d_err, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = sh.grid;
    cfg.blockDim = dim3(kAnyThreads, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1] = {pdl_attribute()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const RhoGeo g = rho_geo(L);
    const float* f = (const float*)src;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_any_rho, f, L, (float2*)rho, g, sh.zchunk);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, m.mrt ? k_any_collide<true> : k_any_collide<false>, f, (float*)dst, L,
                              fast_model(m), (const float2*)rho, g, sh.zchunk, cp, d_err);
}

}  // namespace lbmgb
