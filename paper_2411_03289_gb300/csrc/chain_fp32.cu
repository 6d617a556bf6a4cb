// The mean chain of the FP32 query rollout: all samples' means through the
// horizon and the GP query of every step, every mean term added with
// compensation.
//
// G lanes carry a sample; lane g sums the points g, g + G, ... .  Three rules by
// training-set size, as the sums' orders are part of the results: 8 lanes up to
// 1024 points, 16 up to 2048, 32 beyond, their sums added in lane order; and for
// terrain ensembles and the adjoint 32 lanes and the shuffle tree (ChainSums).  The CTA
// draws the perturbed controls of its samples and steps first, as they do not
// depend on the state.
// What bounds it: the issue slots of the point loop (about 30 instructions a
// point, two thirds of them the two compensated additions) and, below two warps a
// scheduler, their latency.  K = 4096 T = 50 N = 500: 143 us.
#include "query.cuh"

namespace gpm {
namespace {

using namespace qr;

// sum over the warp's lanes
__device__ __forceinline__ float tree_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// TREE: the sums by the shuffle tree (G = 32), the GPs mixed by their weights.
// FUSEZ: a difference z - x is one rounding, fma(z, scale, -x), instead of two.
// SMEM: the training sets of all GPs staged in shared memory.
template <int G, bool TREE, bool FUSEZ, bool SMEM, int CW>
__global__ void __launch_bounds__(32 * CW) k_chain32(const RolloutArgs a, const GpSet gs, const QueryWs ws) {
    extern __shared__ __align__(16) unsigned char csm[];
    constexpr int CT = 32 * CW, SPW = 32 / G, SPC = CW * SPW;    // samples per warp, per CTA
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int l0 = blockIdx.x * SPC;
    const int ls = l0 + warp * SPW + lane / G, g = lane % G;
    const int l = min(ls, ws.Ks - 1);              // spare ones repeat the last sample
    const bool writer = g == 0 && ls < ws.Ks;
    const int s = ws.s0 + l;
    const int T = a.T, Ks = ws.Ks;

    float mu0 = a.x0[0], mu1 = a.x0[1], mu2 = a.x0[2], mu3 = a.x0[3], mu4 = a.x0[4];
    uint32_t it0 = a.it0, it1 = a.it1;
    if (a.x0_dev) {
        mu0 = a.x0_dev[0]; mu1 = a.x0_dev[1]; mu2 = a.x0_dev[2]; mu3 = a.x0_dev[3]; mu4 = a.x0_dev[4];
    }
    if (a.it_dev) {
        const unsigned long long v = *a.it_dev;
        it0 = (uint32_t)v;
        it1 = (uint32_t)(v >> 32);
    }
    if (SMEM) {
        float4* dx = reinterpret_cast<float4*>(csm);
        for (int t = 0; t < gs.M; ++t) {
            const int N = gs.gp[t].N;
            float2* da = reinterpret_cast<float2*>(dx + N);
            for (int i = tid; i < N; i += CT) {
                dx[i] = __ldg(reinterpret_cast<const float4*>(gs.gp[t].Xs) + i);
                da[i] = __ldg(reinterpret_cast<const float2*>(gs.gp[t].alpha) + i);
            }
            dx = reinterpret_cast<float4*>(da + (N + 1) / 2 * 2);
        }
    }
    // clamped perturbed controls (Eq. 8) of this CTA's samples, every step
    {
        const int n = min(SPC, Ks - l0);
        for (int i = tid; i < SPC * T; i += CT) {
            const int k = i / SPC, q = i % SPC;
            if (q >= n) continue;
            const float2 e = control_eps((uint32_t)k, (uint32_t)(ws.s0 + l0 + q), it0, it1, a.key0, a.key1, a.sig_v,
                                         a.sig_w);
            float2 u;
            u.x = fminf(fmaxf(__ldg(a.U + 2 * k) + e.x, a.umin0), a.umax0);
            u.y = fminf(fmaxf(__ldg(a.U + 2 * k + 1) + e.y, a.umin1), a.umax1);
            a.u_tilde[(size_t)k * a.K + ws.s0 + l0 + q] = u;
        }
    }
    __syncthreads();
    float2 un = a.u_tilde[s];
    for (int k = 0; k < T; ++k) {
        const float2 ut = un;
        if (k + 1 < T) un = a.u_tilde[(size_t)(k + 1) * a.K + s];
        float mean_v = 0.0f, mean_w = 0.0f;
        const float4* xs = reinterpret_cast<const float4*>(csm);
        for (int t = 0; t < gs.M; ++t) {
            const GpSet::One& P = gs.gp[t];
            const float z0 = mu3 * P.zscale[0], z1 = mu4 * P.zscale[1], z2 = ut.x * P.zscale[2], z3 = ut.y * P.zscale[3];
            const float2* al = reinterpret_cast<const float2*>(xs + P.N);
            float mv = 0.0f, mw = 0.0f, cv = 0.0f, cw = 0.0f;
#pragma unroll 4
            for (int j = g; j < P.N; j += G) {
                const float4 x = SMEM ? xs[j] : __ldg(reinterpret_cast<const float4*>(P.Xs) + j);
                const float2 b = SMEM ? al[j] : __ldg(reinterpret_cast<const float2*>(P.alpha) + j);
                float e0, e1, e2, e3;
                if (FUSEZ) {
                    e0 = fmaf(mu3, P.zscale[0], -x.x);
                    e1 = fmaf(mu4, P.zscale[1], -x.y);
                    e2 = fmaf(ut.x, P.zscale[2], -x.z);
                    e3 = fmaf(ut.y, P.zscale[3], -x.w);
                } else {
                    e0 = z0 - x.x;
                    e1 = z1 - x.y;
                    e2 = z2 - x.z;
                    e3 = z3 - x.w;
                }
                const float kv = P.sf2 * ex2(-(e0 * e0 + e1 * e1 + e2 * e2 + e3 * e3));
                kahan_add(mv, cv, kv * b.x);
                kahan_add(mw, cw, kv * b.y);
            }
            mv += cv;
            mw += cw;
            if (TREE) {
                mean_v += P.w * tree_sum(mv);
                mean_w += P.w * tree_sum(mw);
            } else {
                float tv = 0.0f, tw = 0.0f, dv = 0.0f, dw = 0.0f;
#pragma unroll 8
                for (int i = 0; i < G; ++i) {
                    kahan_add(tv, dv, __shfl_sync(0xffffffffu, mv, i, G));
                    kahan_add(tw, dw, __shfl_sync(0xffffffffu, mw, i, G));
                }
                mean_v = tv + dv;
                mean_w = tw + dw;
            }
            xs = reinterpret_cast<const float4*>(al + (P.N + 1) / 2 * 2);
        }
        float sn, cs;
        sincosf(mu2, &sn, &cs);
        const float nX = __fadd_rn(mu0, __fmul_rn(__fmul_rn(a.dt, mu3), cs));    // (two roundings)
        const float nY = mu1 + a.dt * mu3 * sn;
        const float nT = mu2 + a.dt * mu4;
        const float nV = mu3 + a.kv * (ut.x - mu3) + mean_v;
        const float nW = mu4 + a.kw * (ut.y - mu4) + mean_w;
        if (writer) {
            ws.zq[(size_t)k * Ks + l] = make_float4(mu3, mu4, ut.x, ut.y);
            ws.st[(size_t)k * Ks + l] = make_float4(nX, nY, nT, nV);
        }
        mu0 = nX; mu1 = nY; mu2 = nT; mu3 = nV; mu4 = nW;
    }
    if (writer) ws.zq[(size_t)T * Ks + l] = make_float4(mu3, mu4, 0.0f, 0.0f);
}

template <int G, bool TREE, bool FUSEZ, bool SMEM, int CW>
int launch_w(const RolloutArgs& a, const GpSet& gs, const QueryWs& ws, size_t bytes, cudaStream_t st) {
    constexpr int SPC = CW * 32 / G;
    auto kern = k_chain32<G, TREE, FUSEZ, SMEM, CW>;
    GPM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024));
    kern<<<(unsigned)((ws.Ks + SPC - 1) / SPC), 32 * CW, bytes, st>>>(a, gs, ws);
    GPM_CUDA(cudaGetLastError());
    return GPMPPI_OK;
}

template <int G, bool TREE, bool FUSEZ>
int launch_t(const RolloutArgs& a, const GpSet& gs, const QueryWs& ws, cudaStream_t st) {
    size_t bytes = 0;
    for (int t = 0; t < gs.M; ++t) bytes += (size_t)gs.gp[t].N * 16 + (size_t)(gs.gp[t].N + 1) / 2 * 16;
    // Eight-lane samples: CTAs of one warp (four samples) spread the warps over the
    // schedulers evenly, where 256 CTAs of four are two on most SMs and one on the
    // rest (K = 4096 T = 50 N = 500: 143 against 214 us).  With a sample a warp their
    // copies of the training set cost more (N = 1000: 322 against 267 us).
    // Training sets of up to 4096 points go to shared memory.
    if (G == 8) return launch_w<G, TREE, FUSEZ, true, 1>(a, gs, ws, bytes, st);
    if (bytes <= 100 * 1024) return launch_w<G, TREE, FUSEZ, true, 4>(a, gs, ws, bytes, st);
    return launch_w<G, TREE, FUSEZ, false, 4>(a, gs, ws, 0, st);
}

}  // namespace

int launch_chain_fp32(const RolloutArgs& a, const GpSet& gs, ChainSums sums, const QueryWs& ws, cudaStream_t st) {
    if (sums == kChainTree) return launch_t<32, true, false>(a, gs, ws, st);
    if (sums == kChainTreeFused) return launch_t<32, true, true>(a, gs, ws, st);
    const int N = gs.gp[0].N;
    if (N <= 1024) return launch_t<8, false, false>(a, gs, ws, st);
    return N <= 2048 ? launch_t<16, false, false>(a, gs, ws, st) : launch_t<32, false, false>(a, gs, ws, st);
}

}  // namespace gpm
