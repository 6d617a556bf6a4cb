// The mean chain of the query rollout (Alg. 1 Step 1: noise, clamp, Eq. 1-3,
// 6): all samples' means through the horizon, and the GP query of every step.
//
// A warp carries SG samples; its lanes share the training points, so that every
// point read from shared memory serves SG samples.  A step is the samples'
// kernel rows and their two mean sums (two points per packed instruction), a
// reduction that scatters the 2 SG sums over the lanes, and the unicycle.  The
// perturbed controls do not depend on the state, so the CTA draws those of all
// its samples and steps first.
// What bounds it: the latency of a step's serial chain (row -> reduction ->
// dynamics -> next row) while K leaves few warps per scheduler, the issue slots
// of the kernel rows (about 10 instructions for two points) once it does not.
// With one sample per 16 lanes the shared-memory reads of the points bounded it
// (12 KB per sample and step at N = 500): 112 us at K = 4096, T = 50, N = 500
// against 87 us now.
#include "query.cuh"

namespace gpm {
namespace {

using namespace qr;

constexpr int CT = 128;          // threads
constexpr int CW = CT / 32;
constexpr int GRP = 8;           // pairs of points summed plainly between compensated additions

// Compensated sums over the warp's lanes of the NV values (v[i], c[i]): on
// return v[0] holds the total of one of them, the one sum_lane maps to this
// lane (the exchange halves the values a lane holds while it has several).
template <int NV>
__device__ __forceinline__ void scatter_sum(float (&v)[NV], float (&c)[NV]) {
    const int lane = threadIdx.x & 31;
    int n = NV;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (n > 1) {
            n /= 2;
            const bool up = lane & o;
#pragma unroll
            for (int i = 0; i < NV / 2; ++i) {
                if (i >= n) break;
                const float sv = up ? v[i] : v[i + n], sc = up ? c[i] : c[i + n];
                float kv = up ? v[i + n] : v[i], kc = up ? c[i + n] : c[i];
                const float ov = __shfl_xor_sync(0xffffffffu, sv, o), oc = __shfl_xor_sync(0xffffffffu, sc, o);
                kahan_add(kv, kc, ov);
                v[i] = kv;
                c[i] = kc + oc;
            }
        } else {
            const float ov = __shfl_xor_sync(0xffffffffu, v[0], o), oc = __shfl_xor_sync(0xffffffffu, c[0], o);
            kahan_add(v[0], c[0], ov);
            c[0] += oc;
        }
    }
    v[0] += c[0];
}

// the lane that holds value i of scatter_sum<NV>
template <int NV>
__device__ __forceinline__ int sum_lane(int i) {
    int lane = 0;
#pragma unroll
    for (int o = 16, n = NV; n > 1; o >>= 1) {
        n /= 2;
        if (i & n) lane |= o;
    }
    return lane;
}

// A warp's partial sums (R > 0): 2 SG R chains, 16 or 32 stages at a time (a batch's
// hand-over costs as much as the sums of some 20 stages), a word of padding between
// chains; 1 to 4 KB.
__host__ __device__ constexpr int batch_parts(int SG, int R) { return SG == 1 ? R : R / 2; }    // parts a lane
__host__ __device__ constexpr int batch_stages(int SG, int R) { return R ? batch_parts(SG, R) * 32 / R : 0; }
__host__ __device__ constexpr int part_bytes(int SG, int R) { return R ? (2 * SG * R * (batch_stages(SG, R) + 1) * 4 + 15) / 16 * 16 : 0; }

// SMEM: the training sets of all GPs staged in shared memory (x in two arrays
// of 16-byte halves, so that neighbouring lanes read neighbouring lines).
// R = 0: every lane sums its own pairs, the lanes' sums are added as a tree.
// R > 0: the sums of the batched rollout's R threads a sample (rollout_mma.cu),
// so that a controller's costs are the same bits there and here: R parts of 32 / R
// points of every 32-point stage, each one chain of products, added with
// compensation in the order of the stages; the R sums plainly.  A lane forms the
// parts of its stages, and a lane a chain then adds them: a serial sum of N / 32
// terms a step that the tree does not have.  K = 16384 T = 100 N = 2048 (R = 2):
// 1.64 ms (1.64 as R = 0); K = 5000 T = 60 N = 1500 (R = 8): 397 us (313); K = 1500
// T = 37 N = 777 (R = 8): 77 us (55).
template <int SG, int R, bool SMEM>
__global__ void __launch_bounds__(CT) k_chain(const RolloutArgs a, const GpSet gs, const QueryWs ws) {
    extern __shared__ __align__(16) unsigned char csm[];
    constexpr int SPC = CW * SG;               // samples per CTA
    constexpr int NV = 2 * SG;
    constexpr int RR = R ? R : 1;
    constexpr int PU = 16 / RR;                // pairs of a part
    constexpr int SPB = batch_stages(SG, R);   // stages of a batch
    constexpr int LD = SPB + 1, NCH = NV * RR; // chains and their spacing
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
                // R > 0: the pairs of the lanes' parts next to each other
                const int to = R ? (i % PU) * (np / PU) + i / PU : i;
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
            const int np = G.npad / 2, pairs = (G.N + 1) / 2;
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
            if constexpr (R > 0) {
                const int C = (G.N + 31) / 32, U = C * R;       // stages and parts
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
                            float* o = ps + (lane % R) * LD + (32 / RR) * (b0 + b) + lane / R;
#pragma unroll
                            for (int q = 0; q < SG; ++q) {
                                float x, y;
                                tc::f2unpack(pv[b][q], x, y);
                                o[2 * q * R * LD] = x + y;
                                tc::f2unpack(pw[b][q], x, y);
                                o[(2 * q + 1) * R * LD] = x + y;
                            }
                        }
                    }
                    __syncwarp();
                    const int nc = min(SPB, C - c0);
#pragma unroll
                    for (int h = 0; h < (NCH + 31) / 32; ++h)
                        if (lane + 32 * h < NCH) {
                            const float* o = ps + (lane + 32 * h) * LD;
#pragma unroll 8
                            for (int c = 0; c < nc; ++c) kahan_add(cs_[h], cc_[h], o[c]);
                        }
                    __syncwarp();
                }
#pragma unroll
                for (int h = 0; h < (NCH + 31) / 32; ++h)
                    if (lane + 32 * h < NCH) ps[lane + 32 * h] = cs_[h] + cc_[h];
                __syncwarp();
                float mv = ps[2 * j * R], mw = ps[(2 * j + 1) * R];
#pragma unroll
                for (int u = 1; u < R; ++u) {
                    mv += ps[2 * j * R + u];
                    mw += ps[(2 * j + 1) * R + u];
                }
                mean_v += wsf * mv;
                mean_w += wsf * mw;
                __syncwarp();                      // read before the next GP's parts
                base += 3 * np;
                continue;
            }
            float v[NV], c[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                v[i] = 0.0f;
                c[i] = 0.0f;
            }
            for (int p0 = 0; p0 < pairs; p0 += 32 * GRP) {
                uint64_t pv[SG], pw[SG];
#pragma unroll
                for (int q = 0; q < SG; ++q) {
                    pv[q] = 0ull;
                    pw[q] = 0ull;
                }
                const int pe = min(pairs, p0 + 32 * GRP);
#pragma unroll 2
                for (int p = p0 + lane; p < pe; p += 32) {
                    const ulonglong2 xa = SMEM ? base[p] : __ldg(xg + 2 * p);
                    const ulonglong2 xb = SMEM ? base[np + p] : __ldg(xg + 2 * p + 1);
                    const ulonglong2 al = SMEM ? base[2 * np + p] : __ldg(xg + 2 * np + p);
#pragma unroll
                    for (int q = 0; q < SG; ++q) {
                        float k0, k1;
                        kernel_pair(zz[q], xa, xb, k0, k1);
                        const uint64_t kk = tc::f2pack(k0, k1);
                        pv[q] = tc::f2fma(kk, al.x, pv[q]);
                        pw[q] = tc::f2fma(kk, al.y, pw[q]);
                    }
                }
#pragma unroll
                for (int q = 0; q < SG; ++q) {
                    float x, y;
                    tc::f2unpack(pv[q], x, y);
                    kahan_add(v[2 * q], c[2 * q], x + y);
                    tc::f2unpack(pw[q], x, y);
                    kahan_add(v[2 * q + 1], c[2 * q + 1], x + y);
                }
            }
            scatter_sum<NV>(v, c);
            mean_v += wsf * __shfl_sync(0xffffffffu, v[0], sum_lane<NV>(2 * j));
            mean_w += wsf * __shfl_sync(0xffffffffu, v[0], sum_lane<NV>(2 * j + 1));
            base += 3 * np;
        }
        float sn, cs;
        sincosf(mu2, &sn, &cs);
        // R > 0: the two roundings of the batched rollout
        const float nX = R ? __fadd_rn(mu0, __fmul_rn(__fmul_rn(a.dt, mu3), cs)) : mu0 + a.dt * mu3 * cs;
        const float nY = mu1 + a.dt * mu3 * sn;
        const float nT = mu2 + a.dt * mu4;
        const float nV = mu3 + a.kv * (ut.x - mu3) + mean_v;
        const float nW = mu4 + a.kw * (ut.y - mu4) + mean_w;
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
    // samples per warp: as many as leave every scheduler a warp and a half.
    // Measured (us, 1 / 2 / 4 / 8 samples): K = 256 T = 20 N = 50: 14 / 16 / 16 /
    // 20; K = 1000 T = 40 N = 300: 34 / 36 / 40 / 54; K = 4096 T = 50 N = 500:
    // 114 / 98 / 87 / 87; K = 16384 T = 100 N = 2048: 2379 / 1683 / 1414 / 1509.
    int sg = 1;
    while (sg < 4 && a.K / (2 * sg) >= 900) sg *= 2;     // (a.K: the same in every piece of the samples)
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
    if (ws.rps == 0) GPM_CHAIN_R(0);
    else if (ws.rps == 2) GPM_CHAIN_R(2);
    else if (ws.rps == 4) GPM_CHAIN_R(4);
    else GPM_CHAIN_R(8);
#undef GPM_CHAIN_R
#undef GPM_CHAIN
    GPM_CUDA(cudaGetLastError());
    return GPMPPI_OK;
}

}  // namespace gpm
