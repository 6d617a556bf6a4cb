// GP fit in FP64 on the GPU and the FP32 GP posterior.
//
// Sec. III-A fits two GPs (delta_v, delta_omega) on 4-D inputs; the rollout
// needs, per output, alpha = K^-1 y and L^-1 with L = chol(K_XX + sn2 I)
// (Rasmussen & Williams, Alg. 2.1), never L itself.  So one blocked elimination
// turns K into L^-1 in place (32 x 32 blocks): after block step k the block
// columns up to k hold rows of the inverse's right-hand side and those past k
// the trailing matrix, and the same rank-32 update serves both,
//     M_ij -= L_ik V_j,   V_j = L_jk^T (j > k)  or  (L^-1)_kj (j <= k).
// What bounds it: the FP64 pipe, two FMAs per clock and SM (N^3 / 3 of them:
// 1.9 ms at N = 1500), once a step has more blocks than SMs; the diagonal
// block of the next step is factored by the first CTA of an update while the
// others work on the rest.  N = 1500: updates 2.5 ms, panels 0.85 ms; with its
// allocations, packing and 200 predictions 4.5 ms (26.9 ms as a Cholesky factor, then
// its inverse, block by block).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cmath>
#include <vector>

#include <cstring>

#include "common.cuh"

namespace gpm {
namespace {

constexpr int NB = 32;

// K_XX + sn2 I in the lower triangle, zero above it.
__global__ void k_build_kxx(const double* __restrict__ X, int N, double il0, double il1, double il2, double il3,
                            double sf2, double sn2, double* __restrict__ M) {
    const int i = blockIdx.y * 8 + threadIdx.y, j = blockIdx.x * 32 + threadIdx.x;
    if (i >= N || j >= N) return;
    double v = 0.0;
    if (j <= i) {
        const double d0 = (X[i * 4 + 0] - X[j * 4 + 0]) * il0;
        const double d1 = (X[i * 4 + 1] - X[j * 4 + 1]) * il1;
        const double d2 = (X[i * 4 + 2] - X[j * 4 + 2]) * il2;
        const double d3 = (X[i * 4 + 3] - X[j * 4 + 3]) * il3;
        v = sf2 * exp(-0.5 * (d0 * d0 + d1 * d1 + d2 * d2 + d3 * d3));
        if (i == j) v += sn2;
    }
    M[(size_t)i * N + j] = v;
}

// a / b from r near 1 / b: two corrections by the exact remainder (Markstein 1990).
// Correctly rounded where r is the rounded reciprocal (the panels); within a unit in
// the last place with r a few of them off (the pivot's reciprocal root)
__device__ __forceinline__ double quotient(double a, double b, double r) {
    double q = a * r;
    q = fma(fma(-q, b, a), r, q);
    return fma(fma(-q, b, a), r, q);
}

// Cholesky factor of one 32 x 32 block, element (ty, tx) in m (the full
// symmetric block): row c past the pivot serves, by symmetry, as column c, so a
// step is one multiply-add a thread and one barrier.  D: the factor, lower
// triangle.
__device__ __forceinline__ void factor_diag(double m, double (*v)[NB + 1], double* __restrict__ D, int* flag) {
    const int tx = threadIdx.x, ty = threadIdx.y;
    for (int c = 0; c < NB; ++c) {
        if (ty == c) {
            double d = __shfl_sync(0xffffffffu, m, c);
            if (!(d > 0.0)) {
                if (tx == 0) atomicExch(flag, 1);   // the host reports NOT_PD; go on with finite values
                d = 1.0;
            }
            // square root by its remainder (Markstein) from the reciprocal root, which
            // then also serves the quotients: a third of the chain of sqrt and 1 / p
            const double y = rsqrt(d);
            double p = d * y;
            p = fma(fma(-p, p, d), 0.5 * y, p);
            m = tx == c ? p : quotient(m, p, y);
            v[c & 1][tx] = m;
            if (tx >= c) D[tx * NB + c] = m;
        }
        __syncthreads();
        if (ty > c) m -= v[c & 1][ty] * v[c & 1][tx];
    }
}

// element of block (kb, kb) with an identity extension beyond N
__device__ __forceinline__ double diag_value(const double* M, int N, int kb) {
    const int r = kb + max(threadIdx.x, threadIdx.y), c = kb + min(threadIdx.x, threadIdx.y);
    return r < N ? M[(size_t)r * N + c] : (r == c ? 1.0 : 0.0);
}

__global__ void __launch_bounds__(NB * NB) k_first_diag(const double* __restrict__ M, int N, double* __restrict__ D,
                                                         int* __restrict__ flag) {
    __shared__ double v[2][NB + 1];
    factor_diag(diag_value(M, N, 0), v, D, flag);
}

// Step k's panel, from the factor D of its diagonal block, by substitution:
// L_bk D^T = A_bk for the blocks b > k (to P, N x 32; a vector is a row), D
// (L^-1)_kb = R_kb for b < k and D (L^-1)_kk = I (a vector is a column).  A warp
// takes 8 of a block's 32 vectors, four lanes a vector, lane g its elements g,
// g + 4, ...: a value's updates go out as soon as it is known.  What bounds it is
// the FP64 pipe's rate for one warp, 64 clocks an instruction, on the critical
// path of every step: about 300 instructions (10 us), where a lane per vector took
// 700 (40 us).
__global__ void __launch_bounds__(128) k_panel(double* __restrict__ M, int N, int k, const double* __restrict__ D,
                                               double* __restrict__ P) {
    __shared__ double d[NB][NB + 1], t[NB][NB + 1], rcp[NB];
    const int tid = threadIdx.x, lane = tid & 31, b = blockIdx.x, kb = NB * k, bb = NB * b;
#pragma unroll
    for (int i = tid >> 5; i < NB; i += 4) {
        d[i][lane] = D[i * NB + lane];                   // (the upper triangle is not read)
        if (b > k)
            t[i][lane] = bb + i < N ? M[(size_t)(bb + i) * N + kb + lane] : 0.0;
        else if (b < k)
            t[lane][i] = kb + i < N ? M[(size_t)(kb + i) * N + bb + lane] : 0.0;
        else
            t[lane][i] = i == lane ? 1.0 : 0.0;
    }
    __syncthreads();
    if (tid < NB) rcp[tid] = 1.0 / d[tid][tid];
    __syncthreads();
    const int vec = 8 * (tid >> 5) + (lane >> 2), g = lane & 3;
    double x[NB / 4];
#pragma unroll
    for (int e = 0; e < NB / 4; ++e) x[e] = t[vec][4 * e + g];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
        const int e = q >> 2;
        const double xq = __shfl_sync(0xffffffffu, quotient(x[e], d[q][q], rcp[q]), (lane & ~3) | (q & 3));
        if (g == (q & 3)) x[e] = xq;
        const double u = x[e] - d[4 * e + g][q] * xq;
        if (g > (q & 3)) x[e] = u;
#pragma unroll
        for (int f = e + 1; f < NB / 4; ++f) x[f] -= d[4 * f + g][q] * xq;
    }
#pragma unroll
    for (int e = 0; e < NB / 4; ++e) t[vec][4 * e + g] = x[e];
    __syncthreads();
    for (int i = tid >> 5; i < NB; i += 4) {
        if (b > k) {
            if (bb + i < N) P[(size_t)(bb + i) * NB + lane] = t[i][lane];
        } else if (kb + i < N && bb + lane < N) {
            M[(size_t)(kb + i) * N + bb + lane] = t[lane][i];
        }
    }
}

// Step k's update of the blocks (i, j), k < i, j <= i, one CTA each; the first
// CTA takes block (k + 1, k + 1) and factors it for the next step.
__global__ void __launch_bounds__(NB * NB, 2) k_update(double* __restrict__ M, int N, int k, const double* __restrict__ P,
                                                       double* __restrict__ D, int* __restrict__ flag) {
    __shared__ double l[NB][NB + 1], v[NB][NB + 1];
    const int tx = threadIdx.x, ty = threadIdx.y, kb = NB * k;
    // block number in the triangle's row order, the next diagonal block first
    const int first = (k + 1) * (k + 2) / 2;
    int b = blockIdx.x;
    b = b == 0 ? k + 1 : (b <= k + 1 ? b - 1 : b);
    const int t = first + b;
    int i = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= t) ++i;
    while (i * (i + 1) / 2 > t) --i;
    const int j = t - i * (i + 1) / 2;
    const int row = NB * i + ty, col = NB * j + tx;
    double m = (j != k && row < N && col < N) ? M[(size_t)row * N + col] : 0.0;
    l[ty][tx] = row < N ? P[(size_t)row * NB + tx] : 0.0;
    if (j > k) {
        const int r = NB * j + ty;
        v[tx][ty] = r < N ? P[(size_t)r * NB + tx] : 0.0;
    } else {
        v[ty][tx] = M[(size_t)(kb + ty) * N + col];          // block row k lies below N: i > k has rows
    }
    __syncthreads();
    if (j > k) {
        double s = 0.0;
#pragma unroll 8
        for (int q = 0; q < NB; ++q) s += l[ty][q] * v[q][tx];
        m -= s;
    } else {
#pragma unroll 8
        for (int q = 0; q < NB; ++q) m -= l[ty][q] * v[q][tx];
    }
    if (blockIdx.x == 0) {
        // identity beyond N; the block's lower half mirrored
        if (row >= N || col >= N) m = row == col ? 1.0 : 0.0;
        __syncthreads();
        l[ty][tx] = m;
        __syncthreads();
        if (tx > ty) m = l[tx][ty];
        factor_diag(m, v, D, flag);
    } else if (row < N && col <= row) {
        M[(size_t)row * N + col] = m;
    }
}

// t = L^-1 y for both outputs' columns of y, one warp per row
__global__ void k_alpha_fwd(const double* __restrict__ Xm, const double* __restrict__ y, int N, double* __restrict__ t) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= N) return;
    double s0 = 0.0, s1 = 0.0;
    for (int j = lane; j <= i; j += 32) {
        const double x = Xm[(size_t)i * N + j];
        s0 += x * y[2 * j];
        s1 += x * y[2 * j + 1];
    }
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    if (lane == 0) {
        t[2 * i] = s0;
        t[2 * i + 1] = s1;
    }
}

// alpha = L^-T t in kAlphaParts parts of the rows, 32 columns a CTA
constexpr int kAlphaParts = 8;
__global__ void k_alpha_bwd(const double* __restrict__ Xm, const double* __restrict__ t, int N, double* __restrict__ part) {
    __shared__ double r0[8][33], r1[8][33];
    const int tx = threadIdx.x, ty = threadIdx.y, j = blockIdx.x * 32 + tx;
    const int rows = (N + kAlphaParts - 1) / kAlphaParts;
    const int i0 = max(blockIdx.y * rows, blockIdx.x * 32), i1 = min(N, (blockIdx.y + 1) * rows);
    double s0 = 0.0, s1 = 0.0;
    if (j < N)
        for (int i = i0 + ty; i < i1; i += 8) {
            const double x = Xm[(size_t)i * N + j];          // zero above the diagonal
            s0 += x * t[2 * i];
            s1 += x * t[2 * i + 1];
        }
    r0[ty][tx] = s0;
    r1[ty][tx] = s1;
    __syncthreads();
    if (ty == 0 && j < N) {
        for (int q = 1; q < 8; ++q) {
            s0 += r0[q][tx];
            s1 += r1[q][tx];
        }
        part[((size_t)blockIdx.y * N + j) * 2] = s0;
        part[((size_t)blockIdx.y * N + j) * 2 + 1] = s1;
    }
}
__global__ void k_alpha_sum(const double* __restrict__ part, int N, int o, double* __restrict__ alpha) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    double s = 0.0;
    for (int q = 0; q < kAlphaParts; ++q) s += part[((size_t)q * N + j) * 2 + o];
    alpha[j] = s;
}

// L^-T in the pieces of the query rollout's variance (GpDevice::Wb): block column
// cb holds rows 0 .. 128 (cb + 1) - 1, 128 columns each.  32 x 32 tiles turned in
// shared memory; blockIdx: tile of the points j, of the columns i.
__global__ void __launch_bounds__(256) k_pack_wb(const double* __restrict__ Xm, int N, float* __restrict__ Wb) {
    __shared__ float t[32][33];
    const int tx = threadIdx.x, ty = threadIdx.y, j0 = 32 * blockIdx.x, i0 = 32 * blockIdx.y, cb = i0 / 128;
    if (j0 / 128 > cb) return;
    for (int r = ty; r < 32; r += 8) {
        const int i = i0 + r, j = j0 + tx;
        t[r][tx] = (i < N && j <= i) ? (float)Xm[(size_t)i * N + j] : 0.0f;
    }
    __syncthreads();
    float* out = Wb + (size_t)cb * (cb + 1) / 2 * (128 * 128) + i0 % 128 + tx;
    for (int r = ty; r < 32; r += 8) out[(size_t)(j0 + r) * 128] = t[tx][r];
}

__global__ void k_pack_x(const double* __restrict__ X, int N, double s0, double s1, double s2,
                         double s3, float* __restrict__ Xs) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    Xs[j * 4 + 0] = (float)(X[j * 4 + 0] * s0);
    Xs[j * 4 + 1] = (float)(X[j * 4 + 1] * s1);
    Xs[j * 4 + 2] = (float)(X[j * 4 + 2] * s2);
    Xs[j * 4 + 3] = (float)(X[j * 4 + 3] * s3);
}

__global__ void k_pack_alpha(const double* __restrict__ a0, const double* __restrict__ a1, int N,
                             float* __restrict__ out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    out[j * 2 + 0] = (float)a0[j];
    out[j * 2 + 1] = (float)a1[j];
}

// max |L^-1| over the lower triangle (positive doubles order like their bits)
__global__ void k_absmax(const double* __restrict__ Xm, size_t n, unsigned long long* out) {
    double m = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        m = fmax(m, fabs(Xm[i]));
    atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// Tensor-core tiles of the streaming rollout.  The factor's rows (output
// columns of V) are grouped in pairs of 128-row blocks (NP = ceil(NB / 2)
// pairs of 256 rows; the rows past NpM of an odd NB's last pair are zero) and
// its columns (training points) in stages of 32.  Piece (c, p) holds element
// (i = 256 p + r, j = 32 c + 8 sl + e) of cB L^-1 at
// ((c * NP + p) * 4 + sl) * 2048 + r * 8 + e, so one stage holds the 16 KiB
// pieces of all pairs contiguously, each as four 8-point slabs of 256 rows.
// Formats 0 (FP16) and 1 (BF16): hi = round(v), lo = round(v - hi); format 2
// (BF16, three parts): hi = round(v), mid = round(v - hi), lo = round(v - hi -
// mid), the residuals exact in double.  A GP of a terrain ensemble goes to the
// diagonal block of a stacked factor: its piece (c, p) lands at (c + c_off,
// p + p_off) of a grid NP_out pairs wide (a single GP: 0, 0, its own NP).
__global__ void k_pack_mma(const double* __restrict__ Xm, int N, int NpM, int fmt, double cB, int c_off,
                           int p_off, int NP_out, uint16_t* __restrict__ hi, uint16_t* __restrict__ lo,
                           uint16_t* __restrict__ mid) {
    const size_t idx0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    const int NP = (NpM / 128 + 1) / 2;
    const size_t total = (size_t)(NpM / 32) * NP * 8192;
    if (idx0 >= total) return;
    const size_t piece = idx0 / 8192;
    const int w = (int)(idx0 % 8192);
    const int c = (int)(piece / NP), p = (int)(piece % NP);
    const size_t idx = ((size_t)(c + c_off) * NP_out + (p + p_off)) * 8192 + w;
    const int sl = w / 2048, r = (w / 8) % 256, e = w % 8;
    const int i = 256 * p + r, j = 32 * c + 8 * sl + e;
    double v = 0.0;
    if (i < N && j < N && j <= i) v = cB * Xm[(size_t)i * N + j];
    if (fmt == 0) {
        const __half h = __double2half(v);
        hi[idx] = __half_as_ushort(h);
        lo[idx] = __half_as_ushort(__double2half(v - (double)__half2float(h)));
    } else if (fmt == 1) {
        const __nv_bfloat16 h = __double2bfloat16(v);
        hi[idx] = __bfloat16_as_ushort(h);
        lo[idx] = __bfloat16_as_ushort(__double2bfloat16(v - (double)__bfloat162float(h)));
    } else {
        const __nv_bfloat16 h = __double2bfloat16(v);
        const double r1 = v - (double)__bfloat162float(h);
        const __nv_bfloat16 m = __double2bfloat16(r1);
        hi[idx] = __bfloat16_as_ushort(h);
        mid[idx] = __bfloat16_as_ushort(m);
        lo[idx] = __bfloat16_as_ushort(__double2bfloat16(r1 - (double)__bfloat162float(m)));
    }
}

}  // namespace

// Training inputs and alpha of one GP in pair layout: point j (j < npc; far
// away with alpha 0 past N) at position J0 + j of an array of NpT points (a
// single GP: J0 = 0, NpT = npc; J0 even).
__global__ void k_pack_xa(const float* __restrict__ Xs, const float* __restrict__ alpha, int N, int npc,
                          int J0, int NpT, float* __restrict__ out) {
    const int j0 = blockIdx.x * blockDim.x + threadIdx.x;
    if (j0 >= npc) return;
    const int j = j0;
    float4 x = make_float4(1.0e4f, 1.0e4f, 1.0e4f, 1.0e4f);
    float2 al = make_float2(0.0f, 0.0f);
    if (j < N) {
        x = reinterpret_cast<const float4*>(Xs)[j];
        al = reinterpret_cast<const float2*>(alpha)[j];
    }
    const int J = J0 + j;
    float* xp = out + 8 * (J >> 1) + (J & 1);
    xp[0] = x.x;
    xp[2] = x.y;
    xp[4] = x.z;
    xp[6] = x.w;
    float* ap = out + 4 * NpT + 4 * (J >> 1) + (J & 1);
    ap[0] = al.x;
    ap[2] = al.y;
}

// Scale of the tensor-core operand cB L^-1: the largest power of two with
// cB max|L^-1| <= 2^14 (16-bit range, room for the sums).
int set_cB(GpDevice& g) {
    if (g.cB != 0.0f || g.N == 0) return GPMPPI_OK;
    unsigned long long* d = nullptr;
    GPM_CUDA(cudaMalloc(&d, sizeof(unsigned long long)));
    cudaError_t e = cudaMemset(d, 0, sizeof(unsigned long long));
    if (e == cudaSuccess) {
        k_absmax<<<256, 256>>>(g.Linv64[0], (size_t)g.N * g.N, d);
        e = cudaGetLastError();
    }
    unsigned long long bits = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&bits, d, sizeof(bits), cudaMemcpyDeviceToHost);
    cudaFree(d);
    if (e != cudaSuccess) return cuda_fail(e, "tensor-core factor: absmax");
    double mx = 0.0;
    std::memcpy(&mx, &bits, sizeof(mx));
    g.cB = (float)std::ldexp(1.0, (int)std::floor(std::log2(16384.0 / (mx > 0 ? mx : 1.0))));
    return GPMPPI_OK;
}

// The tiles belong to the GP once all of them are there: after a failure the next call
// starts anew.
int build_mma_tiles(GpDevice& g, int fmt) {
    if (g.mma_hi[fmt] || g.N == 0) return GPMPPI_OK;
    const int N = g.N, NpM = ((N + 127) / 128) * 128;
    const int rc = set_cB(g);
    if (rc) return rc;
    // 32-point stages x pairs of 128-row blocks x 256 rows x 32 points
    const size_t n = (size_t)(NpM / 32) * (size_t)((NpM / 128 + 1) / 2) * 8192;
    uint16_t *hi = nullptr, *lo = nullptr, *mid = nullptr;
    float* xa = g.mma_xa;
    cudaError_t e = cudaMalloc(&hi, n * sizeof(uint16_t));
    if (e == cudaSuccess) e = cudaMalloc(&lo, n * sizeof(uint16_t));
    if (e == cudaSuccess && fmt == 2) e = cudaMalloc(&mid, n * sizeof(uint16_t));
    if (e == cudaSuccess && !xa) e = cudaMalloc(&xa, sizeof(float) * 6 * (size_t)NpM);
    if (e == cudaSuccess) {
        k_pack_mma<<<(unsigned)((n + 255) / 256), 256>>>(g.Linv64[0], N, NpM, fmt, (double)g.cB, 0, 0,
                                                          (NpM / 128 + 1) / 2, hi, lo, mid);
        // the batched rollout's training inputs and alpha in pair layout
        if (!g.mma_xa) k_pack_xa<<<(NpM + 127) / 128, 128>>>(g.Xs[0], g.alpha, N, NpM, 0, NpM, xa);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
    }
    if (e != cudaSuccess) {
        cudaFree(hi);
        cudaFree(lo);
        cudaFree(mid);
        if (!g.mma_xa) cudaFree(xa);
        return cuda_fail(e, "batched rollout: factor tiles");
    }
    g.NpM = NpM;
    g.mma_hi[fmt] = hi;
    g.mma_lo[fmt] = lo;
    if (fmt == 2) g.mma_mid = mid;
    g.mma_xa = xa;
    return GPMPPI_OK;
}

int build_mma_ensemble(GpDevice* const* gs, int M, int fmt, MmaTerrains& tr, uint16_t** hi, uint16_t** lo,
                       uint16_t** mid, float** xa) {
    *hi = *lo = *mid = nullptr;
    *xa = nullptr;
    tr = MmaTerrains{};
    tr.M = M;
    int nb = 0;
    for (int t = 0; t < M; ++t) {
        GpDevice& g = *gs[t];
        int rc = build_mma_tiles(g, fmt);             // the GP's cB (and its own tiles)
        if (rc) return rc;
        // an even number of blocks per GP: no block pair straddles two GPs
        const int nbt = g.N == 0 ? 0 : 2 * ((g.NpM / 128 + 1) / 2);
        tr.blk0[t] = nb;
        nb += nbt;
        const double r = (double)g.sf2[0] / (g.cB > 0.0f ? (double)g.cB : 1.0);
        tr.qscale[t] = (float)(r * r);
        tr.sf2[t] = g.sf2[0];
        tr.w[t] = 1.0f;
        for (int d = 0; d < 4; ++d) tr.zscale[t][d] = g.zscale[0][d];
    }
    tr.blk0[M] = nb;
    if (nb == 0) return GPMPPI_OK;
    const int NpT = nb * 128, NP = nb / 2;
    const size_t n = (size_t)(NpT / 32) * NP * 8192;
    cudaError_t e = cudaMalloc(hi, n * sizeof(uint16_t));
    if (e == cudaSuccess) e = cudaMalloc(lo, n * sizeof(uint16_t));
    if (e == cudaSuccess && fmt == 2) e = cudaMalloc(mid, n * sizeof(uint16_t));
    if (e == cudaSuccess) e = cudaMalloc(xa, sizeof(float) * 6 * (size_t)NpT);
    if (e == cudaSuccess) e = cudaMemset(*hi, 0, n * sizeof(uint16_t));
    if (e == cudaSuccess) e = cudaMemset(*lo, 0, n * sizeof(uint16_t));
    if (e == cudaSuccess && fmt == 2) e = cudaMemset(*mid, 0, n * sizeof(uint16_t));
    for (int t = 0; t < M && e == cudaSuccess; ++t) {
        const GpDevice& g = *gs[t];
        const int nbt = tr.blk0[t + 1] - tr.blk0[t];
        if (nbt == 0) continue;
        const size_t nt = (size_t)(nbt * 4) * (nbt / 2) * 8192;
        k_pack_mma<<<(unsigned)((nt + 255) / 256), 256>>>(g.Linv64[0], g.N, nbt * 128, fmt, (double)g.cB,
                                                           4 * tr.blk0[t], tr.blk0[t] / 2, NP, *hi, *lo, *mid);
        k_pack_xa<<<(nbt * 128 + 127) / 128, 128>>>(g.Xs[0], g.alpha, g.N, nbt * 128, 128 * tr.blk0[t], NpT, *xa);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        cudaFree(*hi);
        cudaFree(*lo);
        cudaFree(*mid);
        cudaFree(*xa);
        *hi = *lo = *mid = nullptr;
        *xa = nullptr;
        return cuda_fail(e, "batched rollout: stacked factor tiles");
    }
    return GPMPPI_OK;
}

// Fit both outputs.  X (N x 4) and Y (N x 2) are host arrays; g.hyper is set.
int gp_fit_device(GpDevice& g, const double* X, const double* Y, int N, cudaStream_t st) {
    g.N = N;
    // columns of the sums of squares and of the adjoint's b: a multiple of 16, at least
    // 64 (the orders of both are part of the results); none at N = 0
    g.Np = (N > 0) ? ((N + 15) / 16) * 16 : 0;
    if (g.Np > 0 && g.Np < 64) g.Np = 64;
    g.npad = ((N + 127) / 128) * 128;
    const size_t nb = (size_t)g.npad / 128;
    const double log2e = 1.4426950408889634;
    for (int o = 0; o < 2; ++o) {
        g.sf2[o] = (float)g.hyper[o].signal_var;
        for (int d = 0; d < 4; ++d)
            g.zscale[o][d] = (float)(std::sqrt(0.5 * log2e) / g.hyper[o].lengthscale[d]);
    }
    const int nout = g.shared ? 1 : 2;
    const size_t nn = (size_t)N * N;
    // one allocation owned by g (freed by the caller on any failure), pieces on
    // 256-byte boundaries: an allocation of its own for each costs as much as
    // the fit of a small training set
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const size_t n1 = N > 0 ? (size_t)N : 1;
    const size_t o_alpha = take(sizeof(float) * 2 * n1);
    const size_t o_a64[2] = {take(sizeof(double) * n1), take(sizeof(double) * n1)};
    size_t o_xs[2], o_l[2], o_xq[2], o_wb[2];
    for (int o = 0; o < nout; ++o) {
        o_xs[o] = take(sizeof(float) * 4 * n1);
        o_l[o] = take(sizeof(double) * nn);
        o_xq[o] = take(sizeof(float) * 6 * (size_t)g.npad);
        o_wb[o] = take(sizeof(float) * nb * (nb + 1) / 2 * (128 * 128));
    }
    GPM_CUDA(cudaMalloc(&g.mem, off));
    char* mem = static_cast<char*>(g.mem);
    g.alpha = reinterpret_cast<float*>(mem + o_alpha);
    for (int o = 0; o < 2; ++o) {
        const int s = o < nout ? o : 0;              // shared hyper-parameters: one factor
        g.alpha64[o] = reinterpret_cast<double*>(mem + o_a64[o]);
        g.Xs[o] = reinterpret_cast<float*>(mem + o_xs[s]);
        g.Linv64[o] = reinterpret_cast<double*>(mem + o_l[s]);
        g.xq[o] = reinterpret_cast<float*>(mem + o_xq[s]);
        g.Wb[o] = reinterpret_cast<float*>(mem + o_wb[s]);
    }
    if (N == 0) return GPMPPI_OK;

    // one scratch allocation: x, y, t, alpha's parts, the panel, a diagonal block, the flag
    const size_t n_y = 2 * (size_t)N, n_part = 2 * (size_t)kAlphaParts * N, n_p = (size_t)NB * N;
    double* scratch = nullptr;
    auto cleanup = [&]() { cudaFree(scratch); };
    auto check = [&](cudaError_t e, const char* what) -> int {
        if (e != cudaSuccess) {
            cleanup();
            return cuda_fail(e, what);
        }
        return GPMPPI_OK;
    };
    int rc;
    if ((rc = check(cudaMalloc(&scratch, sizeof(double) * (4 * n_y + n_part + n_p + NB * NB + 1)), "cudaMalloc scratch")))
        return rc;
    double *dX = scratch, *dY = dX + 2 * n_y, *dt = dY + n_y, *dpart = dt + n_y, *dP = dpart + n_part, *dD = dP + n_p;
    int* dflag = reinterpret_cast<int*>(dD + NB * NB);
    if ((rc = check(cudaMemcpyAsync(dX, X, sizeof(double) * 4 * N, cudaMemcpyHostToDevice, st),
                    "copy X")))
        return rc;
    if ((rc = check(cudaMemcpyAsync(dY, Y, sizeof(double) * 2 * N, cudaMemcpyHostToDevice, st),
                    "copy Y")))
        return rc;
    const int nblk = (N + NB - 1) / NB;
    for (int o = 0; o < nout; ++o) {
        const gpmppi_hyper& h = g.hyper[o];
        if ((rc = check(cudaMemsetAsync(dflag, 0, sizeof(int), st), "memset flag"))) return rc;
        double* M = g.Linv64[o];
        k_build_kxx<<<dim3(nblk, (N + 7) / 8), dim3(32, 8), 0, st>>>(
            dX, N, 1.0 / h.lengthscale[0], 1.0 / h.lengthscale[1], 1.0 / h.lengthscale[2], 1.0 / h.lengthscale[3],
            h.signal_var, h.noise_var, M);
        k_first_diag<<<1, dim3(NB, NB), 0, st>>>(M, N, dD, dflag);
        for (int k = 0; k < nblk; ++k) {
            k_panel<<<nblk, 128, 0, st>>>(M, N, k, dD, dP);
            const int blocks = nblk * (nblk + 1) / 2 - (k + 1) * (k + 2) / 2;
            if (blocks > 0) k_update<<<blocks, dim3(NB, NB), 0, st>>>(M, N, k, dP, dD, dflag);
        }
        if ((rc = check(cudaGetLastError(), "factorisation kernels"))) return rc;
        int hflag = 0;
        if ((rc = check(cudaMemcpyAsync(&hflag, dflag, sizeof(int), cudaMemcpyDeviceToHost, st),
                        "copy flag")))
            return rc;
        if ((rc = check(cudaStreamSynchronize(st), "factorisation sync"))) return rc;
        if (hflag) {
            cleanup();
            return fail(GPMPPI_ERR_NOT_PD, "gp_fit: K_XX + noise_var I is not positive definite");
        }
        const int tb = 128, gb = (N + tb - 1) / tb;
        k_alpha_fwd<<<(N + 7) / 8, 256, 0, st>>>(M, dY, N, dt);
        k_alpha_bwd<<<dim3(nblk, kAlphaParts), dim3(32, 8), 0, st>>>(M, dt, N, dpart);
        k_alpha_sum<<<gb, tb, 0, st>>>(dpart, N, o, g.alpha64[o]);
        if (g.shared) k_alpha_sum<<<gb, tb, 0, st>>>(dpart, N, 1, g.alpha64[1]);
        const double s = std::sqrt(0.5 * log2e);
        k_pack_x<<<gb, tb, 0, st>>>(dX, N, s / h.lengthscale[0], s / h.lengthscale[1],
                                    s / h.lengthscale[2], s / h.lengthscale[3], g.Xs[o]);
        if ((rc = check(cudaGetLastError(), "inverse kernels"))) return rc;
    }
    k_pack_alpha<<<(N + 127) / 128, 128, 0, st>>>(g.alpha64[0], g.alpha64[1], N, g.alpha);
    for (int o = 0; o < nout; ++o) {
        k_pack_xa<<<(g.npad + 127) / 128, 128, 0, st>>>(g.Xs[o], g.alpha, N, g.npad, 0, g.npad, g.xq[o]);
        k_pack_wb<<<dim3((unsigned)(4 * nb), (unsigned)(4 * nb)), dim3(32, 8), 0, st>>>(g.Linv64[o], N, g.Wb[o]);
    }
    if ((rc = check(cudaGetLastError(), "pack alpha"))) return rc;
    if ((rc = check(cudaStreamSynchronize(st), "gp_fit sync"))) return rc;
    cleanup();
    return GPMPPI_OK;
}

}  // namespace gpm
