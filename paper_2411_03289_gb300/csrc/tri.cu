// Triangular products of the GP factor in FP32 on the CUDA cores, and the sums
// of squares over their rows.
//   forward   v_q = L^-1 k*_q   (query rollout, gp_predict, adjoint)
//   backward  b_q = L^-T v_q = K^-1 k*_q   (adjoint)
// An item is 64 queries x one 128-column block, reduced over the training points
// of its triangle in chunks of 32: the factor piece (32 x 128 floats, contiguous)
// and the chunk's points arrive by bulk copies in a ring, the CTA makes the
// kernel values (forward) or transposes the rows of v (backward).  A thread
// holds two columns x 16 queries, so that a step is 16 packed FMAs on four
// broadcast reads; column sets past the diagonal are left out.  Items are very
// uneven (one to N / 32 chunks) and go longest first, three CTAs an SM.
// Every result is one FMA chain over the points in their order, so that it does
// not depend on the split.  The GP variance is what remains of sf2 after nearly
// all of it cancels: its last digits are the rounding of these chains and of the
// sums of squares, whose orders (SumOrder) are part of the results.
// Bound: the FP32 FMA pipe (N (N + 1) / 2 FMAs a query); v is written once
// (4 N bytes a query) and read back once by the sums.
#include "query.cuh"

namespace gpm {
namespace {

using namespace qr;

constexpr int PT = 256;              // threads
constexpr int PQ = 64;               // queries per item
constexpr int CH = 32;               // training points per chunk
constexpr int CB = 128;              // columns per block
constexpr int NST = 3;               // ring stages
constexpr int PIECE = CH * CB * 4;
constexpr int XB = CH * 16;
constexpr int STG = PIECE + XB;
constexpr int OFF_A = NST * STG;                     // 2 x CH x PQ floats: kernel values (rows of v)
constexpr int OFF_BAR = OFF_A + 2 * CH * PQ * 4;
constexpr int SMEM = OFF_BAR + 8 * (NST + 1) + 16;

// acc += a column's factor entries times the 16 queries' values, one chunk
template <bool LO, bool HI>
__device__ __forceinline__ void rows_fma(const float* A, const float* B, uint64_t (&lo)[8], uint64_t (&hi)[8]) {
#pragma unroll 4
    for (int k = 0; k < CH; ++k) {
        uint64_t av[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(A + k * PQ + 4 * i);
            av[2 * i] = a.x;
            av[2 * i + 1] = a.y;
        }
        if (HI) {
            const float b = B[k * CB + 64];
            const uint64_t bb = tc::f2pack(b, b);
#pragma unroll
            for (int i = 0; i < 8; ++i) hi[i] = tc::f2fma(av[i], bb, hi[i]);
        }
        if (LO) {
            const float b = B[k * CB];
            const uint64_t bb = tc::f2pack(b, b);
#pragma unroll
            for (int i = 0; i < 8; ++i) lo[i] = tc::f2fma(av[i], bb, lo[i]);
        }
    }
}

// FUSEZ: a difference z - x is one rounding, fma(z, scale, -x), instead of two
template <bool BACK, bool FUSEZ>
__global__ void __launch_bounds__(PT, 3) k_tri(const TriJob p) {
    extern __shared__ __align__(128) unsigned char psm[];
    float* As = reinterpret_cast<float*>(psm + OFF_A);
    uint64_t* full = reinterpret_cast<uint64_t*>(psm + OFF_BAR);
    uint64_t* never = full + NST;
    int* copies_on = reinterpret_cast<int*>(never + 1);
    const int tid = threadIdx.x, warp = tid >> 5;
    const int nb = (int)gridDim.y, nrow = (p.N + CH - 1) / CH;
    const int cb = BACK ? (int)blockIdx.y : nb - 1 - (int)blockIdx.y;          // longest first
    const int q0 = blockIdx.x * PQ;
    // chunks r0 .. r1 - 1 of the points, and the block's first piece
    const int r0 = BACK ? (CB / CH) * cb : 0;
    const int r1 = BACK ? nrow : min((CB / CH) * (cb + 1), nrow);
    const int nr = r1 - r0;
    const float* fac = p.fac + (BACK ? (size_t)cb * nb - (size_t)cb * (cb - 1) / 2 : (size_t)cb * (cb + 1) / 2) * (CB * CB);

    if (tid == 0) {
        for (int i = 0; i < NST; ++i) tc::mbar_init(full + i, 1);
        tc::mbar_init(never, 1);
        tc::fence_mbar_init();
        // failure-detection hook: a first wait that nothing completes runs out,
        // records the timeout and turns this CTA's copies off, as a copy that
        // never lands would; the kernel then ends normally
        *copies_on = (p.expire_first && !tc::mbar_wait(never, 0u, p.wait_ns, p.err)) ? 0 : 1;
    }
    __syncthreads();
    bool on = *copies_on != 0;
    int fetched = 0;
    auto fetch = [&](int r) {
        unsigned char* dst = psm + (r % NST) * STG;
        uint64_t* bar = full + r % NST;
        ++fetched;
        tc::mbar_expect_tx(bar, BACK ? PIECE : STG);
        bulk_g2s(dst, fac + (size_t)r * (CH * CB), PIECE, bar);
        if (!BACK) bulk_g2s(dst + PIECE, p.xq + (size_t)r * (CH * 4), XB, bar);
    };
    // the factor does not depend on the previous kernel: fetch before it ends
    if (tid == 0 && on)
        for (int r = 0; r < NST && r < nr; ++r) fetch(r);
    grid_wait();

    const int m = tid % PQ, h = tid / PQ;            // query m, points 8 h .. 8 h + 7 of a chunk
    const int qm = min(q0 + m, p.Q - 1);
    uint64_t zz[4], zs[4];
    float4 va, vb;                                   // (backward) the next chunk's 8 values
    const float* vrow = nullptr;
    if (BACK) {
        vrow = p.z + (size_t)qm * p.ldz + CH * r0 + 8 * h;
        va = __ldcg(reinterpret_cast<const float4*>(vrow));
        vb = __ldcg(reinterpret_cast<const float4*>(vrow) + 1);
    } else {
        const float* z = p.z + 4 * (size_t)qm;
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const float v = FUSEZ ? __ldcg(z + d) : __ldcg(z + d) * p.zscale[d];
            zz[d] = tc::f2pack(v, v);
            zs[d] = tc::f2pack(p.zscale[d], p.zscale[d]);
        }
    }
    auto make = [&](int r) {
        if (on) on = tc::mbar_wait(full + r % NST, (uint32_t)(r / NST) & 1u, p.wait_ns, p.err);
        float* dst = As + (r & 1) * (CH * PQ) + h * 8 * PQ + m;
        if (BACK) {
            const float v[8] = {va.x, va.y, va.z, va.w, vb.x, vb.y, vb.z, vb.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) dst[i * PQ] = v[i];
            if (r + 1 < nr) {
                va = __ldcg(reinterpret_cast<const float4*>(vrow + CH * (r + 1)));
                vb = __ldcg(reinterpret_cast<const float4*>(vrow + CH * (r + 1)) + 1);
            }
            return;
        }
        const ulonglong2* x = reinterpret_cast<const ulonglong2*>(psm + (r % NST) * STG + PIECE) + h * 8;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            // k = sf2 2^-(e0 e0 + e1 e1 + e2 e2 + e3 e3), the sum as one chain
            // that starts with the product of e1
            const ulonglong2 a = x[2 * i], b = x[2 * i + 1];
            auto diff = [&](int d, uint64_t y) {
                return FUSEZ ? tc::f2fma(zz[d], zs[d], y ^ 0x8000000080000000ull) : tc::f2sub(zz[d], y);
            };
            const uint64_t d0 = diff(0, a.x), d1 = diff(1, a.y), d2 = diff(2, b.x), d3 = diff(3, b.y);
            uint64_t t = tc::f2mul(d1, d1);
            t = tc::f2fma(d0, d0, t);
            t = tc::f2fma(d2, d2, t);
            t = tc::f2fma(d3, d3, t);
            float t0, t1;
            tc::f2unpack(t, t0, t1);
            dst[2 * i * PQ] = p.sf2 * ex2(-t0);
            dst[(2 * i + 1) * PQ] = p.sf2 * ex2(-t1);
        }
    };

    const int g = tid >> 6, c = tid & 63, wc = warp & 1;     // queries 16 g .., columns c and c + 64
    uint64_t lo[8], hi[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        lo[i] = 0ull;
        hi[i] = 0ull;
    }
    make(0);
    __syncthreads();
    for (int r = 0; r < nr; ++r) {
        if (r + 1 < nr) make(r + 1);
        const float* A = As + (r & 1) * (CH * PQ) + 16 * g;
        const float* B = reinterpret_cast<const float*>(psm + (r % NST) * STG) + c;
        // chunk d of the diagonal block (points 32 d ..): forward, columns below
        // 32 d are zero; backward, columns past 32 d + 31
        const int d = BACK ? r : r - (CB / CH) * cb;
        const bool dolo = BACK ? d >= wc : d <= wc, dohi = BACK ? d >= wc + 2 : d <= wc + 2;
        if (dolo && dohi) rows_fma<true, true>(A, B, lo, hi);
        else if (dolo) rows_fma<true, false>(A, B, lo, hi);
        else if (dohi) rows_fma<false, true>(A, B, lo, hi);
        __syncthreads();
        if (tid == 0 && on && r + NST < nr) {
            tc::fence_proxy_async();                 // the CTA's reads of this stage precede the refill
            fetch(r + NST);
        }
    }
    if (tid == 0 && !on) {                           // copies in flight land before the shared memory is released
        const uint64_t t0 = tc::global_ns();
        for (int r = fetched > NST ? fetched - NST : 0; r < fetched; ++r)
            while (!tc::mbar_try_wait(full + r % NST, (uint32_t)(r / NST) & 1u) && tc::global_ns() - t0 < 200000000ull) {
            }
    }
    const int col = CB * cb + c;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float l[2], u[2];
        tc::f2unpack(lo[i], l[0], l[1]);
        tc::f2unpack(hi[i], u[0], u[1]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int q = q0 + 16 * g + 2 * i + e;
            if (q >= p.Q) continue;
            // row q, or its place among rows padded from rk to rkpad
            const size_t row = p.rk ? (size_t)(q / p.rk) * p.rkpad + q % p.rk : (size_t)q;
            float* o = p.out + row * p.ldo + col;
            if (col < p.ldo) o[0] = l[e];
            if (col + 64 < p.ldo) o[64] = u[e];
        }
    }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// |v_q|^2 of the rows of V, one warp a query
//   kSumPairs  pairs of 8-column groups from both ends of the Np columns (equal
//              triangular work), each pair one chain, the pairs in order
//   kSumLanes  lane l the columns l mod 32, then the shuffle tree
template <int ORDER>
__global__ void __launch_bounds__(256) k_rowsum(const float* __restrict__ V, int ld, int Q, int Np, float* __restrict__ out) {
    const int q = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    grid_wait();
    if (q >= Q) return;
    const float* v = V + (size_t)q * ld;
    float s = 0.0f;
    if (ORDER == kSumPairs) {
        const int np = Np / 16;
        for (int p0 = 0; p0 < np; p0 += 32) {
            const int p = p0 + lane;
            float t = 0.0f;
            if (p < np) {
                float a[8], b[8];
                *reinterpret_cast<float4*>(a) = __ldcg(reinterpret_cast<const float4*>(v + 8 * p));
                *reinterpret_cast<float4*>(a + 4) = __ldcg(reinterpret_cast<const float4*>(v + 8 * p + 4));
                *reinterpret_cast<float4*>(b) = __ldcg(reinterpret_cast<const float4*>(v + Np - 8 * (p + 1)));
                *reinterpret_cast<float4*>(b + 4) = __ldcg(reinterpret_cast<const float4*>(v + Np - 8 * (p + 1) + 4));
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    t = fmaf(a[c], a[c], t);
                    t = fmaf(b[c], b[c], t);
                }
            }
            const int n = min(32, np - p0);
            for (int i = 0; i < n; ++i) s += __shfl_sync(0xffffffffu, t, i);
        }
    } else {
        for (int i = lane; i < Np; i += 32) {
            const float x = __ldcg(v + i);
            s = fmaf(x, x, s);
        }
        s = warp_sum(s);
    }
    if (lane == 0) out[q] = s;
}

// the same, thread i mod 256 of a CTA per query, warps in order
__global__ void __launch_bounds__(256) k_rowsum_block(const float* __restrict__ V, int ld, int N, float* __restrict__ out) {
    __shared__ float red[8];
    const int tid = threadIdx.x;
    grid_wait();
    const float* v = V + (size_t)blockIdx.x * ld;
    float s = 0.0f;
    for (int i = tid; i < N; i += 256) {
        const float x = __ldcg(v + i);
        s = fmaf(x, x, s);
    }
    s = warp_sum(s);
    if ((tid & 31) == 0) red[tid >> 5] = s;
    __syncthreads();
    if (tid == 0) {
        float t = 0.0f;
        for (int i = 0; i < 8; ++i) t += red[i];
        out[blockIdx.x] = t;
    }
}

// L^-1 in the pieces of the backward product: block column cb holds rows
// 128 cb .. npad - 1, 128 columns each, in chunks of 32 rows
__global__ void k_pack_lb(const double* __restrict__ Linv, int N, int nb, float* __restrict__ out) {
    const int cb = blockIdx.y;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (nb - cb) * CB * CB) return;
    const int i = CB * cb + idx / CB, j = CB * cb + idx % CB;
    out[((size_t)cb * nb - (size_t)cb * (cb - 1) / 2) * (CB * CB) + idx] =
        (i < N && j <= i) ? (float)Linv[(size_t)i * N + j] : 0.0f;
}

template <bool BACK>
int launch_tri(const TriJob& j, bool dependent, cudaStream_t st) {
    const dim3 grid((unsigned)((j.Q + PQ - 1) / PQ), (unsigned)((j.N + CB - 1) / CB));
    auto kern = j.fusez ? k_tri<BACK, true> : k_tri<BACK, false>;
    GPM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM));
    GPM_CUDA(launch_ex(kern, grid, PT, SMEM, st, dependent, 1u, j));
    return GPMPPI_OK;
}

}  // namespace

// the forward product of GP g's output o at Q queries (z: Q x 4) into V (Q x npad)
TriJob tri_forward(const GpSet::One& G, const float* z, int Q, float* V) {
    TriJob j = {};
    j.z = z;
    j.fac = G.Wb;
    j.xq = G.xq;
    j.out = V;
    j.ldo = G.npad;
    j.Q = Q;
    j.N = G.N;
    j.sf2 = G.sf2;
    for (int d = 0; d < 4; ++d) j.zscale[d] = G.zscale[d];
    j.wait_ns = 2000000000ull;
    return j;
}

int launch_tri_forward(const TriJob& j, bool dependent, cudaStream_t st) {
    return j.Q > 0 && j.N > 0 ? launch_tri<false>(j, dependent, st) : GPMPPI_OK;
}
int launch_tri_backward(const TriJob& j, bool dependent, cudaStream_t st) {
    return j.Q > 0 && j.N > 0 ? launch_tri<true>(j, dependent, st) : GPMPPI_OK;
}

int launch_rowsum(const float* V, int ld, int Q, int N, SumOrder order, float* out, cudaStream_t st) {
    if (Q <= 0) return GPMPPI_OK;
    int Np = (N + 15) / 16 * 16;
    if (Np > 0 && Np < 64) Np = 64;
    const dim3 grid((unsigned)((Q + 7) / 8));
    if (order == kSumBlock)
        GPM_CUDA(launch_ex(k_rowsum_block, dim3((unsigned)Q), 256, 0, st, true, 1u, V, ld, N, out));
    else if (order == kSumPairs)
        GPM_CUDA(launch_ex(k_rowsum<kSumPairs>, grid, 256, 0, st, true, 1u, V, ld, Q, Np, out));
    else
        GPM_CUDA(launch_ex(k_rowsum<kSumLanes>, grid, 256, 0, st, true, 1u, V, ld, Q, Np, out));
    return GPMPPI_OK;
}

int build_back_pieces(GpDevice& g, cudaStream_t st) {
    if (g.Lb || g.N == 0) return GPMPPI_OK;
    const int nb = g.npad / CB;
    float* out = nullptr;
    GPM_CUDA(cudaMalloc(&out, sizeof(float) * (size_t)nb * (nb + 1) / 2 * (CB * CB)));
    k_pack_lb<<<dim3((unsigned)(nb * CB * CB / 256), (unsigned)nb), 256, 0, st>>>(g.Linv64[0], g.N, nb, out);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaFree(out);
        return cuda_fail(e, "mppi_grad: factor pieces");
    }
    g.Lb = out;
    return GPMPPI_OK;
}

GpSet single_gp_set(const GpDevice& g, int o) {
    GpSet s = {};
    s.M = 1;
    GpSet::One& G = s.gp[0];
    G.xq = g.xq[o];
    G.Wb = g.Wb[o];
    G.Xs = g.Xs[o];
    G.alpha = g.alpha;
    G.N = g.N;
    G.npad = g.npad;
    G.sf2 = g.sf2[o];
    G.w = 1.0f;
    G.qscale = 1.0f;
    for (int d = 0; d < 4; ++d) G.zscale[d] = g.zscale[o][d];
    return s;
}

}  // namespace gpm
