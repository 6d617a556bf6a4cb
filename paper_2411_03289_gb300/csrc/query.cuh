// The query rollout: Alg. 1 Step 1 without its serial variance.
//
// The mean of Eq. 6 never reads the covariance of Eq. 10, so a rollout is
// three passes instead of one recurrence of everything:
//   chain.cu          the means of all samples, step by step (O(N) work per
//                     step: kernel row and k* . alpha), recording the GP
//                     query of every (step, sample);
//   variance_*.cu     |L^-1 k*|^2 of all T K queries at once: a matrix product
//                     with no recurrence, tiled over queries, so every tile is
//                     full and every SM has work whatever K is;
//   stage_cost.cu     the covariance recurrence and the stage costs (O(1) and
//                     O(candidates) per step).
// Shared device helpers of those kernels.
#pragma once

#include "common.cuh"
#include "tc05.cuh"

namespace gpm {
namespace qr {

// 2^x on the SFU; results below the normal range flush to zero, where a kernel
// value is at least 2^-126 of the signal variance's scale
__device__ __forceinline__ float ex2(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// kernel values exp2(-|z - x|^2) of two points in pair layout: a = (x0, x0',
// x1, x1'), b = (x2, x2', x3, x3'); zz_d = (z_d, z_d)
__device__ __forceinline__ void kernel_pair(const uint64_t (&zz)[4], const ulonglong2& a, const ulonglong2& b,
                                            float& k0, float& k1) {
    const uint64_t d0 = tc::f2sub(zz[0], a.x), d1 = tc::f2sub(zz[1], a.y);
    const uint64_t d2 = tc::f2sub(zz[2], b.x), d3 = tc::f2sub(zz[3], b.y);
    uint64_t t = tc::f2mul(d0, d0);
    t = tc::f2fma(d1, d1, t);
    t = tc::f2fma(d2, d2, t);
    t = tc::f2fma(d3, d3, t);
    float t0, t1;
    tc::f2unpack(t, t0, t1);
    k0 = ex2(-t0);
    k1 = ex2(-t1);
}

// Squares of a row of v (column i at v[i ld]) as a warp would sum them: 32 chains
// over the columns i0 + l, i0 + l + STEP, ..., then the shuffle tree.
template <int STEP>
__device__ __forceinline__ float lane_squares(const float* v, int ld, int i0, int n) {
    float s[32];
#pragma unroll
    for (int l = 0; l < 32; ++l) s[l] = 0.0f;
    for (int i = i0; i < n; i += STEP) {
#pragma unroll
        for (int l = 0; l < 32; ++l) {
            const float x = i + l < n ? __ldcg(v + (size_t)(i + l) * ld) : 0.0f;
            s[l] = fmaf(x, x, s[l]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int l = 0; l < o; ++l) s[l] += s[l + o];
    return s[0];
}

// wait for the kernel before this one in the stream (launched with programmatic
// serialisation); a no-op after an ordinary launch
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            tc::smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(tc::smem_addr(bar))
        : "memory");
}

}  // namespace qr

// Launch with optional programmatic serialisation after the previous kernel of
// the stream.
template <typename... KA, typename... A>
inline cudaError_t launch_ex(void (*kern)(KA...), dim3 grid, int threads, size_t smem, cudaStream_t st, bool dependent,
                             A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

}  // namespace gpm
