// Centre-of-mass partials of a stream-collide launch, reduced in a fixed
// order (warp shuffles, then the last CTA to finish), and the frame origin
// for the next step.  Shared by the row kernels and the generic tile kernel.
// Not part of the C ABI.
#pragma once

#include <cuda_runtime.h>

#include "lbm_internal.h"

namespace lbmgb {
namespace {

// The final sum by one warp: slots 0 .. total - 1 in order.
template <typename C>
__device__ void centre_total(const C* parts, unsigned total, unsigned* counter, double* sum8, float* frame) {
    const int lane = threadIdx.x & 31;
    __threadfence();
    // eight slots' loads in flight at once (one after another, the L2
    // latency of each made this sum several microseconds of every launch)
    C s4[4] = {C(0), C(0), C(0), C(0)};
    for (unsigned b0 = lane; b0 < total; b0 += 256u) {
        C v[8][4];
#pragma unroll
        for (unsigned u = 0; u < 8; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) v[u][q] = b0 + 32u * u < total ? __ldcg(parts + 4LL * (b0 + 32u * u) + q) : C(0);
#pragma unroll
        for (unsigned u = 0; u < 8; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) s4[q] += v[u][q];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s4[q] += __shfl_down_sync(0xffffffffu, s4[q], o);
    }
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) sum8[q] = (double)s4[q];
        // frame origin x_c = sum w x / sum w (box centre when there is no droplet)
        const bool have = s4[0] > C(0);
        for (int q = 0; q < 3; ++q) {
            const C xc = have ? s4[1 + q] / s4[0] : C(0);
            sum8[4 + q] = (double)xc;
            frame[q] = (float)xc;
        }
        *counter = 0u;
    }
}

// Fixed-order reduction of centre partials by the last CTA to finish
// (threadfence-reduction pattern); every thread of the CTA calls it.  C is
// the reduction type (float32 for the float32 and 16-bit storage kernels, so
// that they run no FP64 instruction; float64 for the float64 kernel).  This
// CTA's partials go to parts[4 slot .. 4 slot + 3]; `total` CTAs share the
// counter; the last of them sums slots 0 .. total - 1 in order into sum8
// (the four sums, then x_c, y_c, z_c) and frame (x_c in float32), and resets
// the counter.  `scratch` holds 4 values of C per warp of shared memory.
template <typename C>
__device__ void centre_reduce(C (&cm)[4], C* parts, long long slot, unsigned total, unsigned* counter, double* sum8,
                              float* frame, C* scratch) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nwarps = (blockDim.x + 31) >> 5;
    __shared__ unsigned last;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        C a = cm[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        if (lane == 0) scratch[4 * warp + q] = a;
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            C a = lane < nwarps ? scratch[4 * lane + q] : C(0);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
            if (lane == 0) parts[4 * slot + q] = a;
        }
        if (lane == 0) {
            __threadfence();
            last = atomicAdd(counter, 1u) == total - 1 ? 1u : 0u;
        }
    }
    __syncthreads();
    if (last && warp == 0) centre_total(parts, total, counter, sum8, frame);
}

// The same over every CTA of the launch, in CTA order, into CentreParts.
template <typename C>
__device__ void centre_epilogue(C (&cm)[4], CentreParts cp, C* scratch) {
    const long long cta = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    const unsigned total = gridDim.x * gridDim.y * gridDim.z;
    centre_reduce(cm, reinterpret_cast<C*>(cp.p), cta, total, cp.counter, cp.sum, cp.frame, scratch);
}

// Centre-of-mass partials of `units` pieces of the box by the `ctas` CTAs of a
// launch that this is the cta-th of, from a density array, one warp to a unit
// (the two-pass kernels).  unit(u, cm) leaves the sums of unit u in its lane
// 0.  The CTAs that collide then hold nothing back for a reduction and end
// when their nodes are stored; these few run beside them.
template <typename C, typename U>
__device__ void centre_units(U&& unit, int units, int cta, int ctas, CentreParts cp) {
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, warps = blockDim.x / 32;
    __shared__ unsigned last;
    C* parts = reinterpret_cast<C*>(cp.p);
    for (int u = cta * warps + warp; u < units; u += ctas * warps) {
        C cm[4] = {C(0), C(0), C(0), C(0)};
        unit(u, cm);
        if (lane == 0)
#pragma unroll
            for (int q = 0; q < 4; ++q) parts[4LL * u + q] = cm[q];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(cp.counter, 1u) == (unsigned)ctas - 1u ? 1u : 0u;
    }
    __syncthreads();
    if (last && warp == 0) centre_total<C>(parts, (unsigned)units, cp.counter, cp.sum, cp.frame);
}
template <typename C>
__device__ __forceinline__ C warp_total(C a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    return a;
}

}  // namespace
}  // namespace lbmgb
