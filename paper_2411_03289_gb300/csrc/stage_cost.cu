// The covariance recurrence and the stage costs of the query rollout (Eq. 10,
// 11-16, the goal terms of Eq. 12), from the recorded means and variances.
//
// A CTA carries 32 samples (lane = sample) through the horizon in chunks of
// steps.  Per chunk all warps form what a step's Jacobian and variance need,
// then warp 0 runs the covariance recurrence, which is all that is serial
// here, while the other warps score the chunk before it, one step each: the
// lane distance (candidate segments) and the obstacles dominate.
// What bounds it: the latency of a chunk (the recurrence, about 100 instructions
// a step on one warp, beside one or two scored steps a warp).  Measured at
// K = 4096, T = 50, 16 obstacles: 23 us (47 us with the candidate segments read
// one after the other and every obstacle's margin in full).
#include <cfloat>

#include "query.cuh"

namespace gpm {
namespace {

using namespace qr;

constexpr int SW = 16;                   // scoring warps
constexpr int ST = 32 * (SW + 1);        // threads: warp 0 carries the covariance
constexpr int CK = 16;                   // steps per chunk
constexpr int SU = 8;                    // lane segments per round

struct ScoreScale {
    int M, nparts;
    bool two;            // the variances are added in a rounding of their own (FP32 terrain ensembles)
    float w2[kMaxTerrains], sf2[kMaxTerrains], qscale[kMaxTerrains];
};

struct SLayout {
    // two buffers of each, by chunk parity
    static constexpr int pre = 0;                            // CK x 32 float4: sin, cos, v, variance (before the step)
    static constexpr int sxy = pre + 2 * CK * 32 * 16;         // CK x 32 x 3 floats: tightening covariance
    static constexpr int var = sxy + 2 * CK * 32 * 12;       // CK x 32 floats
    static constexpr int stage = var + 2 * CK * 32 * 4;      // CK x 32 floats
    static constexpr int disc = stage + 2 * CK * 32 * 4;     // CK floats
    static constexpr int obst = disc + 2 * CK * 4;           // O x 3 floats
};

// Sigma' = A Sigma A^T + diag(0, 0, 0, s, s) (Eq. 10), A the Jacobian of the
// unicycle step at heading (sn, cs) and speed v
__device__ __forceinline__ void cov_step(const RolloutArgs& a, bool two, float sn, float cs, float v, float s, float& S00,
                                         float& S01, float& S02, float& S03, float& S04, float& S11, float& S12,
                                         float& S13, float& S14, float& S22, float& S23, float& S24, float& S33,
                                         float& S34, float& S44) {
    const float a02 = -a.dt * v * sn, a03 = a.dt * cs;
    const float a12 = a.dt * v * cs, a13 = a.dt * sn;
    // B = A Sigma (rows), then Sigma' = B A^T + diag(0,0,0,s,s)
    const float B00 = S00 + a02 * S02 + a03 * S03, B01 = S01 + a02 * S12 + a03 * S13,
                B02 = S02 + a02 * S22 + a03 * S23, B03 = S03 + a02 * S23 + a03 * S33,
                B04 = S04 + a02 * S24 + a03 * S34;
    const float B11 = S11 + a12 * S12 + a13 * S13, B12 = S12 + a12 * S22 + a13 * S23,
                B13 = S13 + a12 * S23 + a13 * S33, B14 = S14 + a12 * S24 + a13 * S34;
    const float B22 = S22 + a.dt * S24, B23 = S23 + a.dt * S34, B24 = S24 + a.dt * S44;
    const float B33 = a.av * S33, B34 = a.av * S34;
    const float B44 = a.aw * S44;
    S00 = B00 + a02 * B02 + a03 * B03;
    S01 = B01 + a12 * B02 + a13 * B03;
    S02 = B02 + a.dt * B04;
    S03 = a.av * B03;
    S04 = a.aw * B04;
    S11 = B11 + a12 * B12 + a13 * B13;
    S12 = B12 + a.dt * B14;
    S13 = a.av * B13;
    S14 = a.aw * B14;
    S22 = B22 + a.dt * B24;
    S23 = a.av * B23;
    S24 = a.aw * B24;
    S33 = two ? __fadd_rn(__fmul_rn(a.av, B33), s) : a.av * B33 + s;
    S34 = a.aw * B34;
    S44 = two ? __fadd_rn(__fmul_rn(a.aw, B44), s) : a.aw * B44 + s;
}

template <bool TRACE>
__global__ void __launch_bounds__(ST) k_stage_cost(const RolloutArgs a, const ScoreScale sc, const QueryWs ws) {
    extern __shared__ __align__(16) unsigned char ssm[];
    float4* pre = reinterpret_cast<float4*>(ssm + SLayout::pre);
    float* sxy_s = reinterpret_cast<float*>(ssm + SLayout::sxy);
    float* var_s = reinterpret_cast<float*>(ssm + SLayout::var);
    float* stage_s = reinterpret_cast<float*>(ssm + SLayout::stage);
    float* disc_s = reinterpret_cast<float*>(ssm + SLayout::disc);
    float* obst_s = reinterpret_cast<float*>(ssm + SLayout::obst);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int l = min(blockIdx.x * 32 + lane, ws.Ks - 1);
    const bool act = (int)blockIdx.x * 32 + lane < ws.Ks;
    const int Ks = ws.Ks, T = a.T;
    const size_t Q = (size_t)T * Ks;
    for (int i = tid; i < 3 * a.O; i += ST) obst_s[i] = __ldg(a.obst + i);
    float th0 = a.x0[2], v0 = a.x0[3];
    if (a.x0_dev) {
        th0 = a.x0_dev[2];
        v0 = a.x0_dev[3];
    }
    grid_wait();

    float S00 = 0, S01 = 0, S02 = 0, S03 = 0, S04 = 0, S11 = 0, S12 = 0, S13 = 0, S14 = 0, S22 = 0, S23 = 0, S24 = 0,
          S33 = 0, S34 = 0, S44 = 0;
    float cost = 0.0f, disc = 1.0f;
    const int nchunk = (T + CK - 1) / CK;
    for (int c = 0; c <= nchunk; ++c) {
        // the variance and the Jacobian's state of chunk c
        for (int i = warp; i < CK; i += SW + 1) {
            const int k = c * CK + i;
            if (k >= T) break;
            float th = th0, v = v0;
            if (k > 0) {
                const float4 p = ws.st[(size_t)(k - 1) * Ks + l];
                th = p.z;
                v = p.w;
            }
            float s = 0.0f;
            const float* qp = ws.q + (size_t)k * Ks + l;
            for (int t = 0; t < sc.M; ++t) {
                const float q = *qp;
                qp += (size_t)sc.nparts * Q;
                s += sc.w2[t] * fmaxf(0.0f, sc.sf2[t] - sc.qscale[t] * q);
            }
            float sn, cs;
            sincosf(th, &sn, &cs);
            pre[((c & 1) * CK + i) * 32 + lane] = make_float4(sn, cs, v, s);
        }
        __syncthreads();
        if (warp == 0) {
            // the scores of chunk c - 2, in step order
            if (c >= 2)
                for (int i = 0; i < CK; ++i) cost += stage_s[((c & 1) * CK + i) * 32 + lane];
            float* sx = sxy_s + (c & 1) * (CK * 32 * 3);
            float* vr = var_s + (c & 1) * (CK * 32);
            for (int i = 0; i < CK; ++i) {
                const int k = c * CK + i;
                if (k >= T) break;
                const float4 p = pre[((c & 1) * CK + i) * 32 + lane];
                const float sn = p.x, cs = p.y, v = p.z, s = p.w;
                cov_step(a, sc.two, sn, cs, v, s, S00, S01, S02, S03, S04, S11, S12, S13, S14, S22, S23, S24, S33, S34, S44);
                float xx = S00, xy = S01, yy = S11;
                if (a.nom_sxy) {
                    xx = __ldg(a.nom_sxy + 3 * k);
                    xy = __ldg(a.nom_sxy + 3 * k + 1);
                    yy = __ldg(a.nom_sxy + 3 * k + 2);
                }
                sx[i * 32 + lane] = xx;
                sx[(CK + i) * 32 + lane] = xy;
                sx[(2 * CK + i) * 32 + lane] = yy;
                vr[i * 32 + lane] = s;
                if (lane == 0) disc_s[(c & 1) * CK + i] = disc;
                disc *= 0.9f;
                if (TRACE && act && a.tr_sig) {
                    float* o = a.tr_sig + ((size_t)(ws.s0 + l) * T + k) * 15;
                    o[0] = S00; o[1] = S01; o[2] = S02; o[3] = S03; o[4] = S04;
                    o[5] = S11; o[6] = S12; o[7] = S13; o[8] = S14;
                    o[9] = S22; o[10] = S23; o[11] = S24;
                    o[12] = S33; o[13] = S34; o[14] = S44;
                }
            }
        } else if (c > 0) {
            const int cp = c - 1;
            const float* sx = sxy_s + (cp & 1) * (CK * 32 * 3);
            const float* vr = var_s + (cp & 1) * (CK * 32);
            for (int i = warp - 1; i < CK; i += SW) {
                const int k = cp * CK + i;
                if (k >= T) break;
                const float4 p = ws.st[(size_t)k * Ks + l];
                const float X = p.x, Y = p.y, v = p.w;
                const float xx = sx[i * 32 + lane], xy = sx[(CK + i) * 32 + lane], yy = sx[(2 * CK + i) * 32 + lane];
                const float s = vr[i * 32 + lane];
                const float lmax = fmaxf(0.0f, 0.5f * (xx + yy) + hypotf(0.5f * (xx - yy), xy));
                const float rbar = a.r - a.sq_chi2 * sqrtf(lmax);                    // Eq. 14
                float om = FLT_MAX;                                                  // Eq. 15-16
                const float reach = fmaxf(0.0f, a.phi_inv) * sqrtf(lmax);
                for (int o = 0; o < a.O; ++o) {
                    const float cx = obst_s[3 * o], cy = obst_s[3 * o + 1], R = obst_s[3 * o + 2];
                    const float dx = X - cx, dy = Y - cy;
                    // Sigma's spread along any normal is at most sqrt(lmax): beyond
                    // R + reach (with room for rounding) the margin is positive, and
                    // only its sign is asked for unless the margins are recorded
                    const float far = (R + reach) * 1.00001f;
                    if (!TRACE && dx * dx + dy * dy > far * far) continue;
                    const float rho = sqrtf(dx * dx + dy * dy);
                    float spread;
                    if (rho > 1e-9f) {
                        const float nx = dx / rho, ny = dy / rho;
                        spread = sqrtf(fmaxf(0.0f, nx * nx * xx + 2.0f * nx * ny * xy + ny * ny * yy));
                    } else {
                        spread = sqrtf(lmax);
                    }
                    om = fminf(om, (rho - R) - a.phi_inv * spread);
                }
                float best = FLT_MAX;
                const int2 oc = lane_cands(a, X, Y);
                // SU candidates at a time (the last one again past the end): their
                // loads are in flight together
                for (int j = 0; j < oc.y; j += SU) {
                    float4 sg[SU];
                    float il2[SU];
#pragma unroll
                    for (int u = 0; u < SU; ++u) {
                        const int g = lane_seg(a, oc, min(j + u, oc.y - 1));
                        sg[u] = __ldg(a.seg + g);
                        il2[u] = __ldg(a.seg_il2 + g);
                    }
#pragma unroll
                    for (int u = 0; u < SU; ++u) {
                        const float px = X - sg[u].x, py = Y - sg[u].y;
                        const float t = fminf(fmaxf((px * sg[u].z + py * sg[u].w) * il2[u], 0.0f), 1.0f);
                        const float qx = px - t * sg[u].z, qy = py - t * sg[u].w;
                        best = fminf(best, qx * qx + qy * qy);
                    }
                }
                const float e = sqrtf(best);
                const float lmargin = e - rbar;
                float stage = a.c_var * (s + s) + a.c_speed * (a.v_des - v) * (a.v_des - v);
                if (om <= 0.0f) stage += a.c_coll;
                stage += a.c_dev * e;
                if (lmargin > 0.0f) stage += a.c_lane * disc_s[(cp & 1) * CK + i];
                stage += goal_cost(a, k, X, Y);
                stage_s[((cp & 1) * CK + i) * 32 + lane] = stage;
                if (TRACE && act) {
                    const size_t sk = (size_t)(ws.s0 + l) * T + k;
                    if (a.tr_mu) {
                        float* o = a.tr_mu + sk * 5;
                        o[0] = X; o[1] = Y; o[2] = p.z; o[3] = v;
                        o[4] = ws.zq[(size_t)(k + 1) * Ks + l].y;
                    }
                    if (a.tr_stage) a.tr_stage[sk] = stage;
                    if (a.tr_margin) {
                        a.tr_margin[sk * 2] = lmargin;
                        a.tr_margin[sk * 2 + 1] = (a.O > 0) ? om : __int_as_float(0x7f800000);
                    }
                }
            }
        }
    }
    __syncthreads();
    if (warp == 0) {
        for (int i = 0; i < CK; ++i) {
            const int k = (nchunk - 1) * CK + i;
            if (k < T) cost += stage_s[(((nchunk - 1) & 1) * CK + i) * 32 + lane];
        }
        if (act && a.costs) a.costs[ws.s0 + l] = cost;
    }
}

// Alg. 1 Step 2: the covariance along the nominal trajectory, one warp.  Lanes
// load 32 steps' states and variances (ws.q) at a time; every lane carries the
// recurrence, lane 0 records Sigma_XY after each step.  Sigma in full, its two
// triangles by themselves: their roundings differ, and both go into the next step.
__global__ void __launch_bounds__(32) k_nominal_cov(const RolloutArgs a, const QueryWs ws,
                                                    float* __restrict__ sxy) {
    const int lane = threadIdx.x;
    grid_wait();
    float S[5][5] = {};
    for (int k0 = 0; k0 < a.T; k0 += 32) {
        const int kl = min(k0 + lane, a.T - 1);
        float th = a.x0[2], vl = a.x0[3];
        if (kl > 0) {
            const float4 p = ws.st[kl - 1];
            th = p.z;
            vl = p.w;
        }
        const float sl = ws.q[kl];
        float snl, csl;
        sincosf(th, &snl, &csl);
        for (int i = 0; i < 32 && k0 + i < a.T; ++i) {
            const float sn = __shfl_sync(0xffffffffu, snl, i), cs = __shfl_sync(0xffffffffu, csl, i);
            const float v = __shfl_sync(0xffffffffu, vl, i), s = __shfl_sync(0xffffffffu, sl, i);
            const float a02 = -a.dt * v * sn, a03 = a.dt * cs, a12 = a.dt * v * cs, a13 = a.dt * sn;
            float B[5][5];                     // A Sigma
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                B[0][j] = fmaf(a03, S[3][j], fmaf(a02, S[2][j], S[0][j]));
                B[1][j] = fmaf(a13, S[3][j], fmaf(a12, S[2][j], S[1][j]));
                B[2][j] = fmaf(a.dt, S[4][j], S[2][j]);
                B[3][j] = a.av * S[3][j];
                B[4][j] = a.aw * S[4][j];
            }
#pragma unroll
            for (int r = 0; r < 5; ++r) {      // times A^T
                S[r][0] = fmaf(B[r][3], a03, fmaf(B[r][2], a02, B[r][0]));
                S[r][1] = fmaf(B[r][3], a13, fmaf(B[r][2], a12, B[r][1]));
                S[r][2] = fmaf(B[r][4], a.dt, B[r][2]);
                S[r][3] = __fmul_rn(B[r][3], a.av);
                S[r][4] = __fmul_rn(B[r][4], a.aw);
            }
            S[3][3] = __fadd_rn(S[3][3], s);
            S[4][4] = __fadd_rn(S[4][4], s);
            if (lane == 0) {
                sxy[3 * (k0 + i)] = S[0][0];
                sxy[3 * (k0 + i) + 1] = S[0][1];
                sxy[3 * (k0 + i) + 2] = S[1][1];
            }
        }
    }
}

}  // namespace

int launch_nominal_cov(const RolloutArgs& a, const QueryWs& ws, float* sxy_out, cudaStream_t st) {
    GPM_CUDA(launch_ex(k_nominal_cov, dim3(1), 32, 0, st, true, a, ws, sxy_out));
    return GPMPPI_OK;
}

int launch_stage_cost(const RolloutArgs& a, const GpSet& gs, const QueryWs& ws, bool ensemble, cudaStream_t st) {
    ScoreScale sc = {};
    sc.M = gs.M;
    sc.nparts = ws.nparts;
    sc.two = ensemble;
    for (int t = 0; t < gs.M; ++t) {
        sc.w2[t] = gs.gp[t].w * gs.gp[t].w;
        sc.sf2[t] = gs.gp[t].sf2;
        sc.qscale[t] = gs.gp[t].qscale;
    }
    const int smem = SLayout::obst + 12 * a.O;
    const bool trace = a.tr_mu || a.tr_sig || a.tr_stage || a.tr_margin;
    auto kern = trace ? k_stage_cost<true> : k_stage_cost<false>;
    // the same limit whatever O is: it belongs to the function, which other threads launch too
    GPM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  SLayout::obst + 12 * GPMPPI_MAX_OBSTACLES));
    GPM_CUDA(launch_ex(kern, dim3((unsigned)((ws.Ks + 31) / 32)), ST, smem, st, true, a, sc, ws));
    return GPMPPI_OK;
}

}  // namespace gpm
