// Adjoint (reverse-mode) rollout: gradient of the smoothed chance-constrained
// MPPI cost with respect to the nominal controls U and the SE-ARD
// lengthscales of the residual GPs.
//
// Objective.  J = sum_s w_s S_s, where S_s is the rollout cost of sample s
// (Alg. 1 Step 1, Eq. 10-16) with the indicators of Eq. 11-12 replaced by
// logistic sigmoids of slope * margin, the control noise held fixed (the
// Philox draws of the current iteration) and w_s = 1/K unless the caller
// passes weights.
//
// The forward pass is a query rollout: the means of all samples (chain_fp32.cu),
// v = L^-1 k* and b = L^-T v = K^-1 k* of all T K queries as two triangular
// products (tri.cu), none of which needs the recurrence.  Then one warp per sample:
//   k_grad_fwd   covariances, S_s, and the records of every step;
//   k_grad_rev   the reverse steps, last first: stage-cost adjoint (lane distance,
//                lambda_max of Sigma_XY, obstacle spread), covariance adjoint
//                (Sigma' = A Sigma A^T + D: Sigma_bar = A^T G A, A_bar = 2 G A Sigma),
//                mean adjoint (Eq. 6), then the GP adjoint over the points:
//                k*_bar_j = m_bar . alpha_j - 2 s_bar b_j, z_bar, the direct
//                lengthscale terms and the terms that flow through alpha = K^-1 y.
// The terms that flow through K^-1 in the variance need G_o = sum_q s_bar_o,q
// b_q b_q^T; k_grad_rev stores the per-query adjoints, and a Gram kernel
// forms tr(dK/dl_d G_o) tile by tile.  A last kernel reduces the per-sample
// contributions in double in a fixed order, so results are deterministic.
#include <cfloat>

#include "common.cuh"
#include "warp_rollout.cuh"

namespace gpm {
namespace {

using namespace wr;

constexpr float kLn2 = 0.69314718055994530942f;

// Smoothed stage cost at the post-step state (warp-wide, lane-replicated).
__device__ float stage_cost(const GradArgs& g, int k, const float mu[5], const float S[15], float sraw) {
    const RolloutArgs& a = g.r;
    const float s = fmaxf(0.0f, sraw);
    float best;
    int bi;
    lane_nearest(a, mu[0], mu[1], best, bi);
    const float e = sqrtf(best);
    const Lam L = lam_max(S[sidx(0, 0)], S[sidx(0, 1)], S[sidx(1, 1)]);
    const float rbar = a.r - a.sq_chi2 * L.sq;                               // Eq. 14
    const float disc = exp2f((float)k * log2f(0.9f));
    float c = a.c_var * (s + s) + a.c_speed * (a.v_des - mu[3]) * (a.v_des - mu[3]) + a.c_dev * e +
              a.c_lane * disc * sigm(g.slope * (e - rbar));
    if (a.O > 0) {
        float om;
        int oi;
        obstacle_nearest(a, mu[0], mu[1], S[sidx(0, 0)], S[sidx(0, 1)], S[sidx(1, 1)], L.sq, om, oi);
        c += a.c_coll * sigm(-g.slope * om);
    }
    if (a.c_goal != 0.0f || a.c_term != 0.0f) {          // Eq. 12 goal terms, F smoothed
        const float dx = mu[0] - a.goal_x, dy = mu[1] - a.goal_y;
        const float d = sqrtf(dx * dx + dy * dy);
        c += a.c_goal * d;
        if (k == a.T - 1) c += a.c_term * sigm(g.slope * (d - a.goal_r));
    }
    return c;
}

// Adjoint of the smoothed stage cost at the post-step state, scaled by wt,
// added to the post-state adjoints mub (mean) and Sb (Sigma, stored upper
// triangle: the derivative with respect to each stored entry).  Returns the
// derivative with respect to the GP variance of each output.
__device__ float stage_cost_adjoint(const GradArgs& g, int k, const float mu[5], const float S[15],
                                    float wt, float mub[5], float Sb[15]) {
    const RolloutArgs& a = g.r;
    const float sxx = S[sidx(0, 0)], sxy = S[sidx(0, 1)], syy = S[sidx(1, 1)];
    const Lam L = lam_max(sxx, sxy, syy);
    float gX = 0.0f, gY = 0.0f, gxx = 0.0f, gxy = 0.0f, gyy = 0.0f;
    // lane deviation and tightened lane indicator (Eq. 11, 13-14)
    float best;
    int bi;
    lane_nearest(a, mu[0], mu[1], best, bi);
    const float e = sqrtf(best);
    float ex = 0.0f, ey = 0.0f;              // d e / d (X, Y)
    if (e > 0.0f && bi < a.S) {
        const float4 sg = __ldg(a.seg + bi);
        const float il2 = __ldg(a.seg_il2 + bi);
        const float qx0 = mu[0] - sg.x, qy0 = mu[1] - sg.y;
        const float t = fminf(fmaxf((qx0 * sg.z + qy0 * sg.w) * il2, 0.0f), 1.0f);
        ex = (qx0 - t * sg.z) / e;
        ey = (qy0 - t * sg.w) / e;
    }
    const float disc = exp2f((float)k * log2f(0.9f));
    const float sl = sigm(g.slope * (e - (a.r - a.sq_chi2 * L.sq)));
    const float gl = a.c_lane * disc * g.slope * sl * (1.0f - sl);    // d cost / d lane margin
    gX += (a.c_dev + gl) * ex;
    gY += (a.c_dev + gl) * ey;
    gxx += gl * a.sq_chi2 * L.dxx;
    gxy += gl * a.sq_chi2 * L.dxy;
    gyy += gl * a.sq_chi2 * L.dyy;
    // collision indicator (Eq. 12, 15-16) through the nearest tightened obstacle
    if (a.O > 0) {
        float om;
        int oi;
        obstacle_nearest(a, mu[0], mu[1], sxx, sxy, syy, L.sq, om, oi);
        const float sc = sigm(-g.slope * om);
        const float gc = -a.c_coll * g.slope * sc * (1.0f - sc);      // d cost / d margin
        if (oi < a.O) {
            const float cx = __ldg(a.obst + 3 * oi), cy = __ldg(a.obst + 3 * oi + 1);
            const float dx = mu[0] - cx, dy = mu[1] - cy;
            const float rho = sqrtf(dx * dx + dy * dy);
            if (rho > 1e-9f) {
                const float nx = dx / rho, ny = dy / rho;
                const float qn = nx * nx * sxx + 2.0f * nx * ny * sxy + ny * ny * syy;
                const float sp = sqrtf(fmaxf(0.0f, qn));
                float mx = nx, my = ny;           // d margin / d (X, Y)
                if (sp > 0.0f) {
                    const float snx = sxx * nx + sxy * ny, sny = sxy * nx + syy * ny;
                    mx -= a.phi_inv * (snx - qn * nx) / (rho * sp);
                    my -= a.phi_inv * (sny - qn * ny) / (rho * sp);
                    const float f = -a.phi_inv * 0.5f / sp;
                    gxx += gc * f * nx * nx;
                    gxy += gc * f * 2.0f * nx * ny;
                    gyy += gc * f * ny * ny;
                }
                gX += gc * mx;
                gY += gc * my;
            } else {
                gxx += gc * (-a.phi_inv) * L.dxx;
                gxy += gc * (-a.phi_inv) * L.dxy;
                gyy += gc * (-a.phi_inv) * L.dyy;
            }
        }
    }
    if (a.c_goal != 0.0f || a.c_term != 0.0f) {
        const float dx = mu[0] - a.goal_x, dy = mu[1] - a.goal_y;
        const float d = sqrtf(dx * dx + dy * dy);
        if (d > 0.0f) {
            float gd = a.c_goal;                            // d cost / d distance
            if (k == a.T - 1) {
                const float sg = sigm(g.slope * (d - a.goal_r));
                gd += a.c_term * g.slope * sg * (1.0f - sg);
            }
            gX += gd * dx / d;
            gY += gd * dy / d;
        }
    }
    mub[0] += wt * gX;
    mub[1] += wt * gY;
    mub[3] += wt * (-2.0f * a.c_speed * (a.v_des - mu[3]));
    Sb[sidx(0, 0)] += wt * gxx;
    Sb[sidx(0, 1)] += wt * gxy;
    Sb[sidx(1, 1)] += wt * gyy;
    return wt * a.c_var;
}

// Sigma' = A Sigma A^T + diag(0, 0, 0, s, s)  (Eq. 10), upper triangle in S
__device__ __forceinline__ void cov_forward(const RolloutArgs& a, float th, float v, float sv, float S[15]) {
    float sn, cs;
    sincosf(th, &sn, &cs);
    const float a02 = -a.dt * v * sn, a03 = a.dt * cs;
    const float a12 = a.dt * v * cs, a13 = a.dt * sn;
    float A[5][5] = {{1.f, 0.f, a02, a03, 0.f},
                     {0.f, 1.f, a12, a13, 0.f},
                     {0.f, 0.f, 1.f, 0.f, a.dt},
                     {0.f, 0.f, 0.f, a.av, 0.f},
                     {0.f, 0.f, 0.f, 0.f, a.aw}};
    float Sf[5][5];
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = 0; j < 5; ++j) Sf[i][j] = (i <= j) ? S[sidx(i, j)] : S[sidx(j, i)];
    float B[5][5];
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            float t = 0.0f;
#pragma unroll
            for (int m = 0; m < 5; ++m) t = fmaf(A[i][m], Sf[m][j], t);
            B[i][j] = t;
        }
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = i; j < 5; ++j) {
            float t = 0.0f;
#pragma unroll
            for (int m = 0; m < 5; ++m) t = fmaf(B[i][m], A[j][m], t);
            S[sidx(i, j)] = t;
        }
    S[sidx(3, 3)] += sv;
    S[sidx(4, 4)] += sv;
}

// the state before step k of sample l: (X, Y, theta, v) after step k - 1 and omega
__device__ __forceinline__ void state_before(const GradArgs& g, int k, int l, float mu[5]) {
    if (k == 0) {
#pragma unroll
        for (int i = 0; i < 5; ++i) mu[i] = g.r.x0[i];
        return;
    }
    const float4 p = g.ws.st[(size_t)(k - 1) * g.ws.Ks + l];
    mu[0] = p.x; mu[1] = p.y; mu[2] = p.z; mu[3] = p.w;
    mu[4] = g.ws.zq[(size_t)k * g.ws.Ks + l].y;
}

__global__ void __launch_bounds__(GT) k_grad_fwd(const GradArgs g) {
    const RolloutArgs& a = g.r;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int l = blockIdx.x * GMT + w;
    if (l >= g.ws.Ks) return;
    const int Ks = g.ws.Ks;
    float S[15];
#pragma unroll
    for (int i = 0; i < 15; ++i) S[i] = 0.0f;
    float Jsum = 0.0f, Jc = 0.0f;
    float th = a.x0[2], v = a.x0[3];
    for (int k = 0; k < a.T; ++k) {
        const float sraw = a.sf2 - g.ws.q[(size_t)k * Ks + l];
        const float4 p = g.ws.st[(size_t)k * Ks + l];
        cov_forward(a, th, v, fmaxf(0.0f, sraw), S);
        const float mu[5] = {p.x, p.y, p.z, p.w, 0.0f};      // the stage cost does not read omega
        kahan_add(Jsum, Jc, stage_cost(g, k, mu, S, sraw));
        float r = sraw;
#pragma unroll
        for (int i = 0; i < 15; ++i) r = lane == i ? S[i] : r;
        if (lane < 16) g.rec[((size_t)k * Ks + l) * 16 + lane] = r;
        th = p.z;
        v = p.w;
    }
    if (lane == 0) g.S_out[g.ws.s0 + l] = Jsum + Jc;
}

__global__ void __launch_bounds__(GT) k_grad_rev(const GradArgs g) {
    const RolloutArgs& a = g.r;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int l = blockIdx.x * GMT + w;
    const int Ks = g.ws.Ks, Np = a.Np, s = g.ws.s0 + l;
    if (l >= Ks) {
        // a padding row of a step: no adjoint (its b is never read)
        if (l < g.Kpad && lane == 0 && g.qbar)
            for (int k = 0; k < a.T; ++k) g.qbar[(size_t)k * g.Kpad + l] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const float wt = g.weight ? __ldg(g.weight + s) : g.inv_K;
    float mub[5], Sb[15], lsum[8];
#pragma unroll
    for (int i = 0; i < 5; ++i) mub[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < 15; ++i) Sb[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) lsum[i] = 0.0f;
    for (int k = a.T - 1; k >= 0; --k) {
        const float* post = g.rec + ((size_t)k * Ks + l) * 16;
        const float sraw = post[15];
        float sbv = 0.0f, sbw = 0.0f;
        {
            float m1[5], S1[15];
            state_before(g, k + 1, l, m1);
#pragma unroll
            for (int i = 0; i < 15; ++i) S1[i] = post[i];
            // stage cost of step k (scored on the post-step state)
            const float gs = stage_cost_adjoint(g, k, m1, S1, wt, mub, Sb);
            sbv = gs;
            sbw = gs;
        }
        float m0[5], S0[15];
        state_before(g, k, l, m0);
#pragma unroll
        for (int i = 0; i < 15; ++i) S0[i] = k > 0 ? post[i - (ptrdiff_t)Ks * 16] : 0.0f;
        const float4 zq = g.ws.zq[(size_t)k * Ks + l];
        // covariance adjoint: Sigma' = A Sigma A^T + diag(0,0,0,s,s)
        sbv += Sb[sidx(3, 3)];
        sbw += Sb[sidx(4, 4)];
        float sn, cs;
        sincosf(m0[2], &sn, &cs);
        const float v0 = m0[3];
        const float a02 = -a.dt * v0 * sn, a03 = a.dt * cs, a12 = a.dt * v0 * cs, a13 = a.dt * sn;
        const float A[5][5] = {{1.f, 0.f, a02, a03, 0.f},
                               {0.f, 1.f, a12, a13, 0.f},
                               {0.f, 0.f, 1.f, 0.f, a.dt},
                               {0.f, 0.f, 0.f, a.av, 0.f},
                               {0.f, 0.f, 0.f, 0.f, a.aw}};
        float G[5][5], Sf[5][5];
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                const int id = (i <= j) ? sidx(i, j) : sidx(j, i);
                G[i][j] = (i == j) ? Sb[id] : 0.5f * Sb[id];
                Sf[i][j] = S0[id];
            }
        float GA[5][5];
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                float t2 = 0.0f;
#pragma unroll
                for (int m = 0; m < 5; ++m) t2 = fmaf(G[i][m], A[m][j], t2);
                GA[i][j] = t2;
            }
        // A_bar = 2 G A Sigma at the entries of A that depend on the state
        float Ab02 = 0.f, Ab03 = 0.f, Ab12 = 0.f, Ab13 = 0.f;
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            Ab02 = fmaf(GA[0][m], Sf[m][2], Ab02);
            Ab03 = fmaf(GA[0][m], Sf[m][3], Ab03);
            Ab12 = fmaf(GA[1][m], Sf[m][2], Ab12);
            Ab13 = fmaf(GA[1][m], Sf[m][3], Ab13);
        }
        Ab02 *= 2.0f; Ab03 *= 2.0f; Ab12 *= 2.0f; Ab13 *= 2.0f;
        // Sigma_bar = A^T G A, returned to the stored-entry convention
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int j = i; j < 5; ++j) {
                float t2 = 0.0f;
#pragma unroll
                for (int m = 0; m < 5; ++m) t2 = fmaf(A[m][i], GA[m][j], t2);
                Sb[sidx(i, j)] = (i == j) ? t2 : 2.0f * t2;
            }
        // mean adjoint (Eq. 6 with the GP mean), with the A_bar terms
        const float mbv = mub[3], mbw = mub[4];
        float nm[5];
        nm[0] = mub[0];
        nm[1] = mub[1];
        nm[2] = mub[2] + mub[0] * (-a.dt * v0 * sn) + mub[1] * (a.dt * v0 * cs) +
                Ab02 * (-a.dt * v0 * cs) + Ab03 * (-a.dt * sn) + Ab12 * (-a.dt * v0 * sn) +
                Ab13 * (a.dt * cs);
        nm[3] = mub[0] * (a.dt * cs) + mub[1] * (a.dt * sn) + mub[3] * a.av +
                Ab02 * (-a.dt * sn) + Ab12 * (a.dt * cs);
        nm[4] = mub[2] * a.dt + mub[4] * a.aw;
        if (!(sraw > 0.0f)) {       // variance clamped at zero: no gradient through it
            sbv = 0.0f;
            sbw = 0.0f;
        }
        const float* bq = g.Bq + ((size_t)k * g.Kpad + l) * Np;
        if (lane == 0 && g.qbar) g.qbar[(size_t)k * g.Kpad + l] = make_float4(mbv, mbw, sbv, sbw);
        // GP adjoint: z_bar and the lengthscale terms
        float ubx = mbv * a.kv, uby = mbw * a.kw;
        const float z0 = m0[3] * a.zscale[0], z1 = m0[4] * a.zscale[1],
                    z2 = zq.z * a.zscale[2], z3 = zq.w * a.zscale[3];
        float zb[4] = {0.f, 0.f, 0.f, 0.f};
        float lb[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int j = lane; j < a.N; j += 32) {
            const float4 x = ldg4(a.Xs + 4 * j);
            const float d[4] = {z0 - x.x, z1 - x.y, z2 - x.z, z3 - x.w};
            const float kj = a.sf2 * exp2f(-(d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + d[3] * d[3]));
            const float bj = __ldcg(bq + j);
            const float2 al = __ldg(reinterpret_cast<const float2*>(a.alpha) + j);
            const float wv = kj * (mbv * al.x - 2.0f * sbv * bj);
            const float ww = kj * (mbw * al.y - 2.0f * sbw * bj);
            const float wz = wv + ww;
#pragma unroll
            for (int dd = 0; dd < 4; ++dd) {
                zb[dd] = fmaf(wz, d[dd], zb[dd]);
                const float d2 = d[dd] * d[dd];
                lb[dd] = fmaf(wv, d2, lb[dd]);
                lb[4 + dd] = fmaf(ww, d2, lb[4 + dd]);
            }
            if (g.ubar) {
#pragma unroll
                for (int dd = 0; dd < 4; ++dd) {
                    lb[dd] = fmaf(-mbv * bj, __ldg(g.ubar + (size_t)dd * Np + j), lb[dd]);
                    lb[4 + dd] = fmaf(-mbw * bj, __ldg(g.ubar + (size_t)(4 + dd) * Np + j), lb[4 + dd]);
                }
            }
        }
#pragma unroll
        for (int dd = 0; dd < 4; ++dd) zb[dd] = -2.0f * kLn2 * a.zscale[dd] * wsum(zb[dd]);
#pragma unroll
        for (int i = 0; i < 8; ++i) lb[i] = wsum(lb[i]);
        nm[3] += zb[0];
        nm[4] += zb[1];
        ubx += zb[2];
        uby += zb[3];
        if (lane == 0) {
            // no gradient through a control at its bound
            const bool in0 = zq.z > a.umin0 && zq.z < a.umax0, in1 = zq.w > a.umin1 && zq.w < a.umax1;
            g.dU_out[(size_t)(2 * k) * a.K + s] = in0 ? ubx : 0.0f;
            g.dU_out[(size_t)(2 * k + 1) * a.K + s] = in1 ? uby : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) lsum[i] += lb[i];
#pragma unroll
        for (int i = 0; i < 5; ++i) mub[i] = nm[i];
    }
    if (lane == 0 && g.dl_out) {
#pragma unroll
        for (int i = 0; i < 8; ++i) g.dl_out[(size_t)i * a.K + s] = lsum[i];
    }
}

// ubar[(o*4+d)][i] = sum_j Kf_ij (xs_id - xs_jd)^2 alpha_o[j]: (dK/dl_d) alpha_o
// up to the factor 2 ln2 / l_d; one warp per row i.
__global__ void k_dk_alpha(const float* __restrict__ Xs, const float* __restrict__ alpha, int N, int Np,
                           float sf2, float* __restrict__ ubar) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (i >= Np) return;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (i < N) {
        const float4 xi = ldg4(Xs + 4 * i);
        for (int j = lane; j < N; j += 32) {
            const float4 xj = ldg4(Xs + 4 * j);
            const float d[4] = {xi.x - xj.x, xi.y - xj.y, xi.z - xj.z, xi.w - xj.w};
            const float dd[4] = {d[0] * d[0], d[1] * d[1], d[2] * d[2], d[3] * d[3]};
            const float kf = sf2 * exp2f(-(dd[0] + dd[1] + dd[2] + dd[3]));
            const float2 al = __ldg(reinterpret_cast<const float2*>(alpha) + j);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                acc[e] = fmaf(kf * dd[e], al.x, acc[e]);
                acc[4 + e] = fmaf(kf * dd[e], al.y, acc[4 + e]);
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const float v = wsum(acc[e]);
        if (lane == 0) ubar[(size_t)e * Np + i] = v;
    }
}

// Final reductions in double, fixed order: blocks [0, 2T) -> dU, block 2T -> J,
// blocks 2T+1 .. 2T+8 -> dl (when requested).
__global__ void k_grad_reduce(const GradReduceArgs r) {
    __shared__ double red[256];
    const int b = blockIdx.x, tid = threadIdx.x;
    double acc = 0.0;
    float* dst = nullptr;
    double scale = 1.0;
    if (b < 2 * r.T) {
        for (int s = tid; s < r.K; s += 256) acc += (double)r.dU_out[(size_t)b * r.K + s];
        dst = r.dU + b;
    } else if (b == 2 * r.T) {
        for (int s = tid; s < r.K; s += 256)
            acc += (double)(r.weight ? r.weight[s] : r.inv_K) * (double)r.S_out[s];
        dst = r.J;
    } else {
        const int e = b - 2 * r.T - 1;
        for (int s = tid; s < r.K; s += 256) acc += (double)r.dl_out[(size_t)e * r.K + s];
        for (int p = tid; p < r.nparts; p += 256) acc += (double)r.parts[(size_t)p * 8 + e];
        dst = r.dl + e;
        scale = 2.0 * 0.69314718055994530942 / r.ell[e & 3];
    }
    red[tid] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (tid < o) red[tid] += red[tid + o];
        __syncthreads();
    }
    if (tid == 0 && dst) *dst = (float)(red[0] * scale);
}

}  // namespace

int launch_grad_forward(const GradArgs& g, cudaStream_t st) {
    k_grad_fwd<<<(g.ws.Ks + GMT - 1) / GMT, GT, 0, st>>>(g);
    GPM_CUDA(cudaGetLastError());
    return 0;
}

int launch_grad_reverse(const GradArgs& g, cudaStream_t st) {
    k_grad_rev<<<(g.Kpad + GMT - 1) / GMT, GT, 0, st>>>(g);
    GPM_CUDA(cudaGetLastError());
    return 0;
}

int launch_dk_alpha(const float* Xs, const float* alpha, int N, int Np, float sf2, float* ubar,
                    cudaStream_t st) {
    k_dk_alpha<<<(Np + 7) / 8, 256, 0, st>>>(Xs, alpha, N, Np, sf2, ubar);
    GPM_CUDA(cudaGetLastError());
    return 0;
}

int launch_grad_reduce(const GradReduceArgs& r, cudaStream_t st) {
    const int nb = 2 * r.T + 1 + (r.dl ? 8 : 0);
    k_grad_reduce<<<nb, 256, 0, st>>>(r);
    GPM_CUDA(cudaGetLastError());
    return 0;
}

}  // namespace gpm
