// Triangular products of the GP factor in FP32 on the CUDA cores, and the sums
// of squares over their rows.
//   forward   v_q = L^-1 k*_q   (query rollout, Alg. 1 Step 2, gp_predict, adjoint)
//   backward  b_q = L^-T v_q = K^-1 k*_q   (adjoint)
// An item is 128 queries x one 128-column block, reduced over the training points
// of its triangle in chunks of 32: the factor piece (32 x 128 floats, contiguous)
// and the chunk's points (forward) or its rows of v (backward) arrive by bulk
// copies in a ring.  A thread multiplies an 8-query x 8-column tile in registers
// with packed FMAs (query pairs): 4 shared-memory reads for 32 of them, where 2
// columns x 16 queries needed 12 and the reads, not the FMAs, bounded it.  A warp
// owns 16 columns, leaves out the diagonal's rows that hold none of them, and does
// nothing past N.  Items are very uneven (one to N / 32 chunks) and go longest first, two
// CTAs an SM.  v is kept by tiles of 128 queries, query the fastest index, so that
// it leaves in whole lines, comes back as operands by bulk copies and is summed
// with a thread per query.
// Every result is one FMA chain over the points in their order, so that it does
// not depend on the split.  The GP variance is what remains of sf2 after nearly
// all of it cancels: its last digits are the rounding of these chains and of the
// sums of squares, whose orders (SumOrder) are part of the results.
// Bound: the FP32 FMA pipe (N (N + 1) / 2 FMAs a query; three quarters active), the rest
// the barriers around a chunk; v is written once (4 N bytes a query) and read back once
// by the sums.  204,800 queries, forward: N = 500 0.98 ms (52 TFLOP/s; 1.32 with 2
// columns x 16 queries; 2.5 inside the rollout that carried a sample tile through the
// horizon), N = 1000 3.74 ms; backward, N = 1000: 3.57 ms (57 TFLOP/s).  81,920 queries
// of N = 400: 0.29 ms (0.41 with the columns past N multiplied).  Barriers in shared
// memory that let warps drift a chunk apart: 8 % slower.
#include "query.cuh"

namespace gpm {
namespace {

using namespace qr;

constexpr int PT = 256;              // threads
constexpr int PQ = 128;              // queries per item (kTriTile)
constexpr int CH = 32;               // training points per chunk
constexpr int CB = 128;              // columns per block
constexpr int NST = 3;               // ring stages
constexpr int PIECE = CH * CB * 4;
constexpr int AB = CH * PQ * 4;      // a chunk's operand: kernel values or rows of v
static_assert(PQ == kTriTile, "tile of v");

// shared memory: ring (piece, then points or rows of v), kernel values, barriers
template <bool BACK>
struct TriLayout {
    static constexpr int stage = PIECE + (BACK ? AB : CH * 16);
    static constexpr int a = NST * stage;
    static constexpr int bar = a + (BACK ? 0 : 2 * AB);
    static constexpr int total = bar + 8 * (NST + 1) + 16;
};

// FUSEZ: a difference z - x is one rounding, fma(z, scale, -x), instead of two
template <bool BACK, bool FUSEZ>
__global__ void __launch_bounds__(PT, 2) k_tri(const TriJob p) {
    extern __shared__ __align__(128) unsigned char psm[];
    using L = TriLayout<BACK>;
    float* As = reinterpret_cast<float*>(psm + L::a);
    uint64_t* full = reinterpret_cast<uint64_t*>(psm + L::bar);
    uint64_t* never = full + NST;
    int* copies_on = reinterpret_cast<int*>(never + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nb = (int)gridDim.y, nrow = (p.N + CH - 1) / CH;
    const int cb = BACK ? (int)blockIdx.y : nb - 1 - (int)blockIdx.y;          // longest first
    const int tile = blockIdx.x, q0 = tile * PQ;
    // chunks r0 .. r1 - 1 of the points, and the block's first piece
    const int r0 = BACK ? (CB / CH) * cb : 0;
    const int r1 = BACK ? nrow : min((CB / CH) * (cb + 1), nrow);
    const int nr = r1 - r0;
    const float* fac = p.fac + (BACK ? (size_t)cb * nb - (size_t)cb * (cb - 1) / 2 : (size_t)cb * (cb + 1) / 2) * (CB * CB);
    // rows of v of this tile (backward): npad x 128 floats
    const float* vt = p.z + ((size_t)tile * p.ldz + CH * r0) * PQ;

    if (tid == 0) {
        for (int i = 0; i < NST; ++i) tc::mbar_init(full + i, 1);
        tc::mbar_init(never, 1);
        tc::fence_mbar_init();
        // failure-detection hook: a first wait that nothing completes runs out,
        // records the timeout and turns this CTA's copies off, as a copy that
        // never lands would; the kernel then ends normally.  Once one CTA has recorded
        // it the others need not wait: a rollout has thousands of them.
        const bool known = p.expire_first && (*(volatile unsigned int*)p.err & 1u);
        *copies_on = (known || (p.expire_first && !tc::mbar_wait(never, 0u, p.wait_ns, p.err))) ? 0 : 1;
    }
    __syncthreads();
    bool on = *copies_on != 0;
    int fetched = 0;
    auto fetch = [&](int r) {
        unsigned char* dst = psm + (r % NST) * L::stage;
        uint64_t* bar = full + r % NST;
        ++fetched;
        tc::mbar_expect_tx(bar, L::stage);
        bulk_g2s(dst, fac + (size_t)r * (CH * CB), PIECE, bar);
        if (BACK) bulk_g2s(dst + PIECE, vt + (size_t)r * (CH * PQ), AB, bar);
        else bulk_g2s(dst + PIECE, p.xq + (size_t)r * (CH * 4), CH * 16, bar);
    };
    // the factor and the points do not depend on the previous kernel (v does)
    if (BACK) grid_wait();
    if (tid == 0 && on)
        for (int r = 0; r < NST && r < nr; ++r) fetch(r);
    if (!BACK) grid_wait();

    const int m = tid % PQ, h = tid / PQ;            // kernel values: query m, points 16 h .. 16 h + 15 of a chunk
    uint64_t zz[4], zs[4];
    if (!BACK) {
        const float* z = p.z + 4 * (size_t)min(q0 + m, p.Q - 1);
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const float v = FUSEZ ? __ldcg(z + d) : __ldcg(z + d) * p.zscale[d];
            zz[d] = tc::f2pack(v, v);
            zs[d] = tc::f2pack(p.zscale[d], p.zscale[d]);
        }
    }
    auto arrived = [&](int r) {
        if (on) on = tc::mbar_wait(full + r % NST, (uint32_t)(r / NST) & 1u, p.wait_ns, p.err);
    };
    auto make = [&](int r) {
        arrived(r);
        const ulonglong2* x = reinterpret_cast<const ulonglong2*>(psm + (r % NST) * L::stage + PIECE) + h * 16;
        float* dst = As + (r & 1) * (CH * PQ) + h * 16 * PQ + m;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
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

    // The warp's columns: 16 w for warps 0-3 and from the other end for 4-7, so that
    // the two warps of every scheduler share the diagonal's work evenly; none past N.
    const int w0 = 16 * (warp < 4 ? warp : 11 - warp);
    // first row (backward) or last row (forward) of the block's first 128 that it needs
    const int edge = CB * cb + w0 >= (BACK ? p.ldo : p.N) ? (BACK ? 1 << 20 : -(1 << 20)) : BACK ? w0 : w0 + 16;
    const int lq = lane & 15, c0 = w0 + 8 * (lane >> 4);
    uint64_t acc[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[i][c] = 0ull;
    if (!BACK) {
        make(0);
        __syncthreads();
    }
    for (int r = 0; r < nr; ++r) {
        // kernel values of the next chunk: one of a scheduler's two warps before its
        // products, the other after, so that they overlap
        if (BACK) arrived(r);
        else if (warp < 4 && r + 1 < nr) make(r + 1);
        const unsigned char* stage = psm + (r % NST) * L::stage;
        const float* A = BACK ? reinterpret_cast<const float*>(stage + PIECE) : As + (r & 1) * (CH * PQ);
        const float* B = reinterpret_cast<const float*>(stage) + c0;
        // rows of the diagonal block that hold none of this warp's columns: forward
        // those past its last column, backward those before its first
        const int d = BACK ? CH * r : CH * (r - (CB / CH) * cb);
        const int k0 = BACK ? min(CH, max(0, edge - d)) : 0;
        const int k1 = BACK ? CH : min(CH, edge - d);
        // 16 points of loads and FMAs in flight (4 points: 1.05 against 0.98 ms at N = 500)
#pragma unroll 16
        for (int k = k0; k < k1; ++k) {
            uint64_t av[4];
            const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(A + k * PQ + 4 * lq);
            const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(A + k * PQ + 64 + 4 * lq);
            av[0] = a0.x; av[1] = a0.y; av[2] = a1.x; av[3] = a1.y;
            const float4 b0 = *reinterpret_cast<const float4*>(B + k * CB);
            const float4 b1 = *reinterpret_cast<const float4*>(B + k * CB + 4);
            const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint64_t bb = tc::f2pack(b[c], b[c]);
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i][c] = tc::f2fma(av[i], bb, acc[i][c]);
            }
        }
        if (!BACK && warp >= 4 && r + 1 < nr) make(r + 1);
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
    float o[8][8];                                   // query, column
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 8; ++c) tc::f2unpack(acc[i][c], o[2 * i][c], o[2 * i + 1][c]);
    if (!BACK) {
        float* v = p.out + ((size_t)tile * p.ldo + CB * cb + c0) * PQ + 4 * lq;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            *reinterpret_cast<float4*>(v + c * PQ) = make_float4(o[0][c], o[1][c], o[2][c], o[3][c]);
            *reinterpret_cast<float4*>(v + c * PQ + 64) = make_float4(o[4][c], o[5][c], o[6][c], o[7][c]);
        }
    } else {
        // row q, at its place among rows padded from rk to rkpad; 8 columns at a
        // time (ldo is a multiple of 16)
        const int col = CB * cb + c0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int q = q0 + (i >> 2) * 64 + 4 * lq + (i & 3);
            if (q >= p.Q || col >= p.ldo) continue;
            float* b = p.out + ((size_t)(q / p.rk) * p.rkpad + q % p.rk) * p.ldo + col;
            *reinterpret_cast<float4*>(b) = make_float4(o[i][0], o[i][1], o[i][2], o[i][3]);
            *reinterpret_cast<float4*>(b + 4) = make_float4(o[i][4], o[i][5], o[i][6], o[i][7]);
        }
    }
}

// |v_q|^2, one thread a query
//   kSumPairs  pairs of 8-column groups from both ends of the Np columns (equal
//              triangular work), each pair one chain, the pairs in order
//   kSumLanes  32 chains over the columns l mod 32, added as a tree
template <int ORDER>
__global__ void __launch_bounds__(PQ) k_rowsum(const float* __restrict__ V, int ld, int Q, int Np, float* __restrict__ out) {
    grid_wait();
    const float* v = V + (size_t)blockIdx.x * ld * PQ + threadIdx.x;
    float s = 0.0f;
    if (ORDER == kSumPairs) {
        for (int p = 0; p < Np / 16; ++p) {
            float a[8], b[8], t = 0.0f;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                a[c] = __ldcg(v + (size_t)(8 * p + c) * PQ);
                b[c] = __ldcg(v + (size_t)(Np - 8 * (p + 1) + c) * PQ);
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                t = fmaf(a[c], a[c], t);
                t = fmaf(b[c], b[c], t);
            }
            s += t;
        }
    } else {
        s = lane_squares<32>(v, PQ, 0, Np);
    }
    const int q = blockIdx.x * PQ + threadIdx.x;
    if (q < Q) out[q] = s;
}

// max(0, sf2 - |v_q|^2): 256 chains over the columns mod 256, eight threads a query for
// the trees of their warps, which are added in order
__global__ void __launch_bounds__(8 * PQ) k_block_variance(const float* __restrict__ V, int ld, int Q, int N, float sf2,
                                                           float* __restrict__ out) {
    __shared__ float red[8][PQ];
    const int w = threadIdx.x / PQ, l = threadIdx.x % PQ;
    grid_wait();
    red[w][l] = lane_squares<256>(V + (size_t)blockIdx.x * ld * PQ + l, PQ, 32 * w, N);
    __syncthreads();
    const int q = blockIdx.x * PQ + l;
    if (w > 0 || q >= Q) return;
    float s = 0.0f;
    for (int i = 0; i < 8; ++i) s += red[i][l];
    out[q] = fmaxf(0.0f, sf2 - s);
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
    const int smem = TriLayout<BACK>::total;
    GPM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    GPM_CUDA(launch_ex(kern, grid, PT, smem, st, dependent, j));
    return GPMPPI_OK;
}

}  // namespace

// the forward product of a GP at Q queries (z: Q x 4) into V (tiles of 128 queries x npad)
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
    auto kern = order == kSumPairs ? k_rowsum<kSumPairs> : k_rowsum<kSumLanes>;
    GPM_CUDA(launch_ex(kern, dim3((unsigned)((Q + PQ - 1) / PQ)), PQ, 0, st, true, V, ld, Q, Np, out));
    return GPMPPI_OK;
}

int launch_block_variance(const float* V, int ld, int Q, int N, float sf2, float* out, cudaStream_t st) {
    if (Q <= 0) return GPMPPI_OK;
    GPM_CUDA(launch_ex(k_block_variance, dim3((unsigned)((Q + PQ - 1) / PQ)), 8 * PQ, 0, st, true, V, ld, Q, N, sf2, out));
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
