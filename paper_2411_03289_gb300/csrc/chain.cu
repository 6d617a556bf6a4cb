// The mean chain of the query rollout (Alg. 1 Step 1: noise, clamp, Eq. 1-3,
// 6): all samples' means through the horizon, and the GP query of every step.
//
// A warp carries SG samples; its lanes share the training points, so that every
// point read from shared memory serves SG samples.  A step is the samples'
// kernel rows and their two mean sums (two points per packed instruction) in parts,
// the parts' sums, and the unicycle.  The perturbed controls do not depend on the
// state, so the CTA draws those of all its samples and steps first.
// What bounds it: the latency of a step's serial chain (row -> sums ->
// dynamics -> next row) while K leaves few warps per scheduler, the issue slots
// of the kernel rows (about 10 instructions for two points) once it does not.
// With one sample per 16 lanes the shared-memory reads of the points bounded it
// (12 KB per sample and step at N = 500): 112 us at K = 4096, T = 50, N = 500
// against 71 us with four samples a warp (85 with the lanes' sums as a tree).
#include "query.cuh"

namespace gpm {
namespace {

using namespace qr;

constexpr int CT = 128;          // threads
constexpr int CW = CT / 32;

// The sums of the mean are those of the rollouts that carried a sample tile through the
// horizon (VarSums): parts of consecutive points, each one chain of products of pairs,
// added with compensation by a lane a chain; the chains plainly.
//   R = 2, 4, 8  the batched rollout's R threads a sample (rollout_mma.cu): R parts of
//                32 / R points of every 32-point stage, R chains, stages ascending
//   R = 1        kSumsShares: 16-point chunks; chains of the even and the odd chunks of
//                each share, 257 to 512 points: 24-27, 12-23, then 28-31 with 0-11; 129
//                to 256: 12-15, 0-11; fewer: 0-7
// A lane forms the parts of its stages, and a lane a chain then adds them: for R > 1 a
// serial sum of N / 32 terms a step that a tree would not have.  K = 16384 T = 100 N =
// 2048 (R = 2): 1.62 ms (1.64 with the lanes' sums as a tree); K = 5000 T = 60 N = 1500
// (R = 8): 380 us (313); K = 1500 T = 37 N = 777 (R = 8): 76 us (55).
__host__ __device__ constexpr int part_pairs(int R) { return R == 1 ? 8 : 16 / R; }
// R > 1: parts a lane forms before they are added, 16 or 32 stages (a batch's hand-over
// costs as much as the sums of some 20 stages); R = 1: all of them
__host__ __device__ constexpr int batch_parts(int SG, int R) { return R == 1 ? 1 : SG == 1 ? R : R / 2; }
__host__ __device__ constexpr int batch_stages(int SG, int R) { return R == 1 ? 32 : batch_parts(SG, R) * 32 / R; }
// A warp's partial sums: 2 SG R chains, a word of padding between them; R = 1: 32 chunks
// of 2 SG values (kShareLd words each: the lanes' reads in different banks), and the sums
// of their six chains.  1 to 4 KB.
constexpr int kShareChains = 6, kShareLd = 42;
__host__ __device__ constexpr int part_bytes(int SG, int R) {
    return (2 * SG * (R == 1 ? kShareLd + kShareChains : R * (batch_stages(SG, R) + 1)) * 4 + 15) / 16 * 16;
}

// SMEM: the training sets of all GPs staged in shared memory (x in two arrays
// of 16-byte halves, the pairs of the lanes' parts next to each other).
template <int SG, int R, bool SMEM>
__global__ void __launch_bounds__(CT) k_chain(const RolloutArgs a, const GpSet gs, const QueryWs ws) {
    extern __shared__ __align__(16) unsigned char csm[];
    constexpr int SPC = CW * SG;               // samples per CTA
    constexpr int NV = 2 * SG;
    constexpr int PU = part_pairs(R);          // pairs of a part
    constexpr int SPB = batch_stages(SG, R);   // stages of a batch
    constexpr int LD = R == 1 ? kShareLd : SPB + 1, NCH = NV * R;      // chains and their spacing
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float4* zs = reinterpret_cast<float4*>(csm) + warp * SG;            // the warp's queries
    float* ps = reinterpret_cast<float*>(csm + CW * SG * 16 + warp * part_bytes(SG, R));
    ulonglong2* xs = reinterpret_cast<ulonglong2*>(csm + CW * (SG * 16 + part_bytes(SG, R)));
    const int l0 = blockIdx.x * SPC;
    const int j = lane % SG;                                            // the sample whose state this lane carries
    const int l = min(l0 + warp * SG + j, ws.Ks - 1);                   // spare ones repeat the last sample
    const bool writer = lane < SG && l0 + warp * SG + j < ws.Ks;
    const int s = ws.s0 + l;
    const int K = a.K, T = a.T, Ks = ws.Ks;

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
        ulonglong2* dst = xs;
        for (int t = 0; t < gs.M; ++t) {
            const int np = gs.gp[t].npad / 2;           // pairs
            const ulonglong2* src = reinterpret_cast<const ulonglong2*>(gs.gp[t].xq);
            for (int i = tid; i < np; i += CT) {
                const int to = (i % PU) * (np / PU) + i / PU;
                dst[to] = __ldg(src + 2 * i);
                dst[np + to] = __ldg(src + 2 * i + 1);
                dst[2 * np + to] = __ldg(src + 2 * np + i);
            }
            dst += 3 * np;
        }
    }
    // clamped perturbed controls (Eq. 8) of this CTA's samples, every step
    const int n = min(SPC, Ks - l0);
    for (int i = tid; i < SPC * T; i += CT) {
        const int k = i / SPC, q = i % SPC;
        if (q >= n) continue;
        const float2 e = control_eps((uint32_t)k, (uint32_t)(ws.s0 + l0 + q), it0, it1, a.key0, a.key1, a.sig_v,
                                     a.sig_w);
        float2 u;
        u.x = fminf(fmaxf(__ldg(a.U + 2 * k) + e.x, a.umin0), a.umax0);
        u.y = fminf(fmaxf(__ldg(a.U + 2 * k + 1) + e.y, a.umin1), a.umax1);
        a.u_tilde[(size_t)k * K + ws.s0 + l0 + q] = u;
    }
    // R = 1: four lanes a value; lanes 0 and 1 (the parity) sum the first shares (two
    // chains: two chunks from c0, six from c1), lanes 2 and 3 the last one (one chain)
    int c0_ = 0, c1_ = 4;
    bool apart = false, none = false;
    if (R == 1) {
        const int N = gs.gp[0].N;
        const bool last = lane & 2;
        apart = N > 128 && !last;
        none = N <= 256 && last;
        if (N > 256) c0_ = last ? 28 : 24, c1_ = last ? 0 : 12;
        else if (N > 128) c0_ = 12, c1_ = 0;
        c0_ += lane & 1;
        c1_ += lane & 1;
    }
    __syncthreads();
    float2 un = a.u_tilde[s];
    for (int k = 0; k < T; ++k) {
        const float2 ut = un;
        if (k + 1 < T) un = a.u_tilde[(size_t)(k + 1) * K + s];
        if (lane < SG) zs[lane] = make_float4(mu3, mu4, ut.x, ut.y);
        __syncwarp();
        float mean_v = 0.0f, mean_w = 0.0f;
        const ulonglong2* base = xs;
        for (int t = 0; t < gs.M; ++t) {
            const GpSet::One& G = gs.gp[t];
            const int np = G.npad / 2;
            const ulonglong2* xg = reinterpret_cast<const ulonglong2*>(G.xq);
            uint64_t zz[SG][4];
#pragma unroll
            for (int q = 0; q < SG; ++q) {
                const float4 z = zs[q];
                const float z0 = z.x * G.zscale[0], z1 = z.y * G.zscale[1];
                const float z2 = z.z * G.zscale[2], z3 = z.w * G.zscale[3];
                zz[q][0] = tc::f2pack(z0, z0);
                zz[q][1] = tc::f2pack(z1, z1);
                zz[q][2] = tc::f2pack(z2, z2);
                zz[q][3] = tc::f2pack(z3, z3);
            }
            const float wsf = G.w * G.sf2;
            const int C = R == 1 ? (G.N + 15) / 16 : (G.N + 31) / 32, U = C * R;       // stages and parts
            float cs_[(NCH + 31) / 32], cc_[(NCH + 31) / 32];
#pragma unroll
            for (int h = 0; h < (NCH + 31) / 32; ++h) {
                cs_[h] = 0.0f;
                cc_[h] = 0.0f;
            }
            for (int c0 = 0; c0 < C; c0 += SPB) {
                // IU parts of a lane interleaved; past the last one that part again
                constexpr int IU = SG < 4 && batch_parts(SG, R) > 1 ? 2 : 1;
                for (int b0 = 0; b0 < batch_parts(SG, R) && c0 * R + 32 * b0 < U; b0 += IU) {
                    uint64_t pv[IU][SG], pw[IU][SG];
                    int at[IU];
#pragma unroll
                    for (int b = 0; b < IU; ++b) {
                        const int unit = min(c0 * R + 32 * (b0 + b) + lane, U - 1);
                        at[b] = SMEM ? unit : unit * PU;
#pragma unroll
                        for (int q = 0; q < SG; ++q) {
                            pv[b][q] = 0ull;
                            pw[b][q] = 0ull;
                        }
                    }
#pragma unroll
                    for (int i = 0; i < PU; ++i) {
#pragma unroll
                        for (int b = 0; b < IU; ++b) {
                            const int p = SMEM ? i * (np / PU) + at[b] : at[b] + i;
                            const ulonglong2 xa = SMEM ? base[p] : __ldg(xg + 2 * p);
                            const ulonglong2 xb = SMEM ? base[np + p] : __ldg(xg + 2 * p + 1);
                            const ulonglong2 al = SMEM ? base[2 * np + p] : __ldg(xg + 2 * np + p);
#pragma unroll
                            for (int q = 0; q < SG; ++q) {
                                float k0, k1;
                                kernel_pair(zz[q], xa, xb, k0, k1);
                                const uint64_t kk = tc::f2pack(k0, k1);
                                pv[b][q] = tc::f2fma(kk, al.x, pv[b][q]);
                                pw[b][q] = tc::f2fma(kk, al.y, pw[b][q]);
                            }
                        }
                    }
#pragma unroll
                    for (int b = 0; b < IU; ++b) {
                        float* o = ps + (lane % R) * LD + (32 / R) * (b0 + b) + lane / R;
#pragma unroll
                        for (int q = 0; q < SG; ++q) {
                            const bool in = R > 1 || lane < U;
                            float x, y;
                            tc::f2unpack(pv[b][q], x, y);
                            o[2 * q * R * LD] = in ? x + y : 0.0f;
                            tc::f2unpack(pw[b][q], x, y);
                            o[(2 * q + 1) * R * LD] = in ? x + y : 0.0f;
                        }
                    }
                }
                __syncwarp();
                if constexpr (R > 1) {
                    const int nc = min(SPB, C - c0);
                    if (NCH >= 32 || lane < NCH) {
#pragma unroll 8
                        for (int c = 0; c < nc; ++c)
#pragma unroll
                            for (int h = 0; h < (NCH + 31) / 32; ++h) kahan_add(cs_[h], cc_[h], ps[(lane + 32 * h) * LD + c]);
                    }
                    __syncwarp();
                }
            }
            float mv = 0.0f, mw = 0.0f;
            if constexpr (R > 1) {
#pragma unroll
                for (int h = 0; h < (NCH + 31) / 32; ++h)
                    if (lane + 32 * h < NCH) ps[lane + 32 * h] = cs_[h] + cc_[h];
                __syncwarp();
                mv = ps[2 * j * R];
                mw = ps[(2 * j + 1) * R];
#pragma unroll
                for (int u = 1; u < R; ++u) {
                    mv += ps[2 * j * R + u];
                    mw += ps[(2 * j + 1) * R + u];
                }
            } else {
                // eight terms a lane; chunks past the last one are zero
                float* sum = ps + NV * LD;
                const int val = lane >> 2;
                if (val < NV) {
                    const float* o = ps + val * LD;
                    float x[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) x[i] = i < 2 ? o[c0_ + 2 * i] : o[c1_ + 2 * (i - 2)];
                    float s0 = x[0], k0 = 0.0f;
                    kahan_add(s0, k0, x[1]);
                    const float first = s0 + k0;
                    if (apart) {
                        s0 = 0.0f;
                        k0 = 0.0f;
                    }
#pragma unroll
                    for (int i = 2; i < 8; ++i) kahan_add(s0, k0, x[i]);
                    const float rest = s0 + k0;
                    // order: the shares one after the other, even and odd chunks
                    float* r = sum + val * kShareChains + (lane & 1);
                    if (lane & 2) {
                        r[4] = none ? 0.0f : rest;
                    } else {
                        r[0] = apart ? first : rest;
                        r[2] = apart ? rest : 0.0f;
                    }
                }
                __syncwarp();
#pragma unroll
                for (int i = 0; i < kShareChains; ++i) {
                    mv += sum[2 * j * kShareChains + i];
                    mw += sum[(2 * j + 1) * kShareChains + i];
                }
            }
            mean_v = R == 1 ? mv : mean_v + wsf * mv;      // (R = 1: one GP; scaled below)
            mean_w = R == 1 ? mw : mean_w + wsf * mw;
            __syncwarp();                          // read before the next GP's parts
            base += 3 * np;
        }
        float sn, cs;
        sincosf(mu2, &sn, &cs);
        // R > 1: the two roundings of the batched rollout
        const float nX = R > 1 ? __fadd_rn(mu0, __fmul_rn(__fmul_rn(a.dt, mu3), cs)) : mu0 + a.dt * mu3 * cs;
        const float nY = mu1 + a.dt * mu3 * sn;
        const float nT = mu2 + a.dt * mu4;
        float nV = mu3 + a.kv * (ut.x - mu3), nW = mu4 + a.kw * (ut.y - mu4);
        nV = R == 1 ? fmaf(a.sf2, mean_v, nV) : nV + mean_v;
        nW = R == 1 ? fmaf(a.sf2, mean_w, nW) : nW + mean_w;
        if (writer) {
            ws.zq[(size_t)k * Ks + l] = make_float4(mu3, mu4, ut.x, ut.y);
            ws.st[(size_t)k * Ks + l] = make_float4(nX, nY, nT, nV);
        }
        mu0 = nX; mu1 = nY; mu2 = nT; mu3 = nV; mu4 = nW;
        __syncwarp();                          // every lane has read zs
    }
    if (writer) ws.zq[(size_t)T * Ks + l] = make_float4(mu3, mu4, 0.0f, 0.0f);
}

}  // namespace

int launch_chain(const RolloutArgs& a, const GpSet& gs, const QueryWs& ws, cudaStream_t st) {
    size_t points = 0;
    for (int t = 0; t < gs.M; ++t) points += (size_t)gs.gp[t].npad;
    // two CTAs per SM keep their training sets in shared memory up to 4096 points
    const bool sm = points * 24 <= 100 * 1024;
    // Samples per warp (the sums do not depend on them; a.K: the same in every piece of
    // the samples).  Measured (us, 1 / 2 / 4 samples): K = 256 T = 20 N = 50: 14.3 /
    // 16.9 / 22.6; K = 1000 T = 40 N = 300: 35.1 / 31.8 / 43.7, N = 1200: 85.9 / 77.8 /
    // 118; K = 2000 T = 40 N = 1000: 110 / 78.9 / 95.1; K = 4096 T = 50 N = 500: 99.4 /
    // 79.3 / 70.9, N = 1200: 294 / 201 / 199; K = 16384 T = 100 N = 2048: 2954 / 1954 / 1580.
    const int sg = a.K >= 3600 ? 4 : a.K >= 900 ? 2 : 1;
#define GPM_CHAIN(L, R)                                                                                         \
    do {                                                                                                        \
        const dim3 grid((unsigned)((ws.Ks + CW * L - 1) / (CW * L)));                                           \
        const size_t smem = CW * (L * 16 + part_bytes(L, R)) + (sm ? points * 24 : 0);                          \
        if (sm) {                                                                                               \
            GPM_CUDA(cudaFuncSetAttribute(k_chain<L, R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,     \
                                          120 * 1024));                                                         \
            k_chain<L, R, true><<<grid, CT, smem, st>>>(a, gs, ws);                                             \
        } else {                                                                                                \
            k_chain<L, R, false><<<grid, CT, smem, st>>>(a, gs, ws);                                            \
        }                                                                                                       \
    } while (0)
#define GPM_CHAIN_R(R)                     \
    do {                                   \
        if (sg == 1) GPM_CHAIN(1, R);      \
        else if (sg == 2) GPM_CHAIN(2, R); \
        else GPM_CHAIN(4, R);              \
    } while (0)
    if (ws.sums == kSumsShares) GPM_CHAIN_R(1);
    else if (ws.rps == 2) GPM_CHAIN_R(2);
    else if (ws.rps == 4) GPM_CHAIN_R(4);
    else GPM_CHAIN_R(8);
#undef GPM_CHAIN_R
#undef GPM_CHAIN
    GPM_CUDA(cudaGetLastError());
    return GPMPPI_OK;
}

}  // namespace gpm
