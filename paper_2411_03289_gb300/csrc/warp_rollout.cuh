// Building blocks of the adjoint's warp-per-sample kernels: a CTA of GMT warps
// carries GMT samples, so that a sample's scalar work (covariance, costs) stays
// in one warp.
#pragma once

#include <cfloat>

#include "common.cuh"

namespace gpm {
namespace wr {
namespace {

constexpr int GMT = 8;              // samples per CTA (one warp each)
constexpr int GT = GMT * 32;        // threads per CTA

// upper-triangle position of Sigma[i][j], i <= j: rows hold 5, 4, 3, 2, 1 entries
__host__ __device__ constexpr int sidx(int i, int j) { return i * 5 - (i * (i - 1)) / 2 + (j - i); }

__device__ __forceinline__ float wsum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// warp-wide minimum with the smallest index among equal values
__device__ __forceinline__ void wargmin(float& v, int& i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int oi = __shfl_xor_sync(0xffffffffu, i, o);
        if (ov < v || (ov == v && oi < i)) {
            v = ov;
            i = oi;
        }
    }
}

__device__ __forceinline__ float sigm(float x) { return 1.0f / (1.0f + expf(-x)); }

__device__ __forceinline__ float4 ldg4(const float* p) {
    return __ldg(reinterpret_cast<const float4*>(p));
}

struct Lam {
    float lmax, sq;          // clamped eigenvalue and its square root
    float dxx, dxy, dyy;     // d sqrt(lmax) / d (Sxx, Sxy, Syy)
};

__device__ __forceinline__ Lam lam_max(float sxx, float sxy, float syy) {
    Lam L;
    const float d = 0.5f * (sxx - syy);
    const float h = hypotf(d, sxy);
    const float raw = 0.5f * (sxx + syy) + h;
    L.lmax = fmaxf(0.0f, raw);
    L.sq = sqrtf(L.lmax);
    // derivative of the square root: zero where it is undefined (Sigma_XY = 0)
    const float ds = (raw > 0.0f && L.sq > 0.0f) ? 0.5f / L.sq : 0.0f;
    const float gx = (h > 0.0f) ? 0.5f + 0.5f * d / h : 0.5f;
    const float gy = (h > 0.0f) ? 0.5f - 0.5f * d / h : 0.5f;
    const float gxy = (h > 0.0f) ? sxy / h : 0.0f;
    L.dxx = ds * gx;
    L.dxy = ds * gxy;
    L.dyy = ds * gy;
    return L;
}

// nearest lane segment of point (px, py): squared distance and index (warp-wide)
__device__ __forceinline__ void lane_nearest(const RolloutArgs& a, float px, float py, float& best,
                                             int& bi) {
    const int lane = threadIdx.x & 31;
    best = FLT_MAX;
    bi = 0x7fffffff;
    const int2 oc = lane_cands(a, px, py);                 // candidate segments of this position
    for (int i = lane; i < oc.y; i += 32) {
        const int gI = lane_seg(a, oc, i);
        const float4 sg = __ldg(a.seg + gI);
        const float il2 = __ldg(a.seg_il2 + gI);
        const float qx0 = px - sg.x, qy0 = py - sg.y;
        const float t = fminf(fmaxf((qx0 * sg.z + qy0 * sg.w) * il2, 0.0f), 1.0f);
        const float qx = qx0 - t * sg.z, qy = qy0 - t * sg.w;
        const float d2 = qx * qx + qy * qy;
        if (d2 < best) {
            best = d2;
            bi = gI;
        }
    }
    wargmin(best, bi);
}

// obstacle margin d_bar (Eq. 15-16) of obstacle o at (px, py)
__device__ __forceinline__ float obstacle_margin(const RolloutArgs& a, int o, float px, float py,
                                                 float sxx, float sxy, float syy, float sqlam) {
    const float cx = __ldg(a.obst + 3 * o), cy = __ldg(a.obst + 3 * o + 1), R = __ldg(a.obst + 3 * o + 2);
    const float dx = px - cx, dy = py - cy;
    const float rho = sqrtf(dx * dx + dy * dy);
    float spread;
    if (rho > 1e-9f) {
        const float nx = dx / rho, ny = dy / rho;
        spread = sqrtf(fmaxf(0.0f, nx * nx * sxx + 2.0f * nx * ny * sxy + ny * ny * syy));
    } else {
        spread = sqrtf(fmaxf(0.0f, sqlam * sqlam));
    }
    return (rho - R) - a.phi_inv * spread;
}

__device__ __forceinline__ void obstacle_nearest(const RolloutArgs& a, float px, float py, float sxx,
                                                 float sxy, float syy, float sqlam, float& best,
                                                 int& bi) {
    const int lane = threadIdx.x & 31;
    best = FLT_MAX;
    bi = 0x7fffffff;
    for (int o = lane; o < a.O; o += 32) {
        const float m = obstacle_margin(a, o, px, py, sxx, sxy, syy, sqlam);
        if (m < best) {
            best = m;
            bi = o;
        }
    }
    wargmin(best, bi);
}

}  // namespace
}  // namespace wr
}  // namespace gpm
