// GP variance of many queries in FP32 on the CUDA cores: q = |L^-1 k*|^2 for
// all queries of a rollout (or of gp_predict), a triangular matrix product
// K* L^-T with the squares summed in the epilogue.
//
// A CTA takes TQ queries and the 128-column blocks of L^-T in turn.  The
// reduction runs over chunks of 32 training points: the factor piece (32 x 128
// floats, contiguous in GpDevice::Wb) and the chunk's inputs arrive by bulk
// copies in a ring of stages, the CTA makes the 32 kernel values of its
// queries, and each thread multiplies an 8-query x 8-column tile in registers
// with packed FMAs (query pairs).  Warp w owns columns 16 w .. 16 w + 15 of a
// block: in the block's last 128 rows, the diagonal, it stops where its columns
// end, which leaves the issue slots to the other warps.
// The blocks are dealt to the CTAs of a cluster along y where the queries alone
// do not fill the chip; rank 0 adds the ranks' partial sums in rank order.
// Bound: the FP32 FMA pipe (N (N + 1) / 2 FMAs per query; the kernel values add
// 8 pipe slots for every 128 columns, the diagonal blocks 6 % at N = 500), active
// 71 % of the time; the rest are the chunk barriers with two CTAs per SM.
// Measured: 1.11 ms for 204800 queries at N = 500 and 122 ms for 1638400 at
// N = 2048 (46 and 56 TFLOP/s of the 80 the pipe reaches), against 2.87 and
// 265 ms of the kernel that carried a sample tile's whole recurrence in a CTA.
// 32-point chunks instead of 16: 1 % faster.
#include "query.cuh"

namespace gpm {
namespace {

using namespace qr;

constexpr int VT = 256;              // threads
constexpr int CH = 32;               // training points per chunk
constexpr int CB = 128;              // columns per block
constexpr int NST = 3;               // ring stages
constexpr int PIECE = CH * CB * 4;   // bytes of a factor piece
constexpr int XB = CH * 16;          // bytes of a chunk's inputs
constexpr int STG = PIECE + XB;

template <int TQ>
struct VLayout {
    static constexpr int a = NST * STG;                     // 2 x CH x TQ floats: kernel values
    static constexpr int red = a + 2 * CH * TQ * 4;         // 8 x TQ floats: the warps' sums
    static constexpr int rank = red + 8 * TQ * 4;           // TQ floats: this CTA's sums (read by rank 0)
    static constexpr int mean = rank + TQ * 4;              // 8 x TQ float2: mean partials
    static constexpr int bars = mean + 8 * TQ * 8;
    static constexpr int total = bars + 8 * (NST + 1) + 16;
};

// The chunks of one CTA: blocks cb(0), cb(1), ... of the split, each from row
// chunk 0 to its diagonal (or the last chunk that holds training points).
struct ChunkIt {
    int nb, nsplit, split, nrow;     // column blocks, splits, this split, row chunks of the training set
    int i, cb, r, nr;                // position: block number, block, row chunk, its row chunks
    __device__ ChunkIt(int nb_, int nsplit_, int split_, int nrow_)
        : nb(nb_), nsplit(nsplit_), split(split_), nrow(nrow_), i(0), r(0) {
        seek();
    }
    // longest blocks first, dealt back and forth over the splits
    __device__ void seek() {
        const int j = i * nsplit + ((i & 1) ? nsplit - 1 - split : split);
        cb = nb - 1 - j;
        nr = cb >= 0 ? min((CB / CH) * (cb + 1), nrow) : 0;
    }
    __device__ bool valid() const { return cb >= 0; }
    __device__ bool last_of_block() const { return r == nr - 1; }
    __device__ void next() {
        if (++r == nr) {
            r = 0;
            ++i;
            seek();
        }
    }
    // float offset of the piece in Wb: block cb starts after 128 x 128 floats
    // for each of the cb (cb + 1) / 2 full pieces of the blocks before it
    __device__ size_t piece() const { return (size_t)cb * (cb + 1) / 2 * (CB * CB) + (size_t)r * (CH * CB); }
};

// Bounded wait for a phase (as every wait of this library): on expiry records
// the error; the caller then goes on without waiting.
__device__ __forceinline__ bool bounded(uint64_t* bar, uint32_t parity, unsigned long long ns, unsigned int* err) {
    if (tc::mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = tc::global_ns();
    while (!tc::mbar_try_wait(bar, parity)) {
        if (tc::global_ns() - t0 > ns) {
            if (err) atomicOr(err, 1u);
            return false;
        }
    }
    return true;
}

template <int TQ, bool MEAN>
__global__ void __launch_bounds__(VT, 2) k_var_fp32(const GpSet gs, const VarJob job) {
    extern __shared__ __align__(128) unsigned char vsm[];
    using L = VLayout<TQ>;
    constexpr int NP = TQ / 32;                   // query pairs per thread
    constexpr int PT = CH * TQ / VT;              // kernel values per thread and chunk
    float* As = reinterpret_cast<float*>(vsm + L::a);
    float* red = reinterpret_cast<float*>(vsm + L::red);
    float* rk = reinterpret_cast<float*>(vsm + L::rank);
    uint64_t* full = reinterpret_cast<uint64_t*>(vsm + L::bars);
    uint64_t* never = full + NST;
    int* copies_on = reinterpret_cast<int*>(never + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const GpSet::One& G = gs.gp[blockIdx.z];
    const int nsplit = gridDim.y, split = blockIdx.y;
    const int q0 = blockIdx.x * TQ;
    const int nb = G.npad / CB, nrow = (G.N + CH - 1) / CH;

    if (tid == 0) {
        for (int i = 0; i < NST; ++i) tc::mbar_init(full + i, 1);
        tc::mbar_init(never, 1);
        tc::fence_mbar_init();
        // failure-detection hook: a first wait that nothing completes runs out,
        // records the timeout and turns this CTA's copies off, as a copy that
        // never lands would; the kernel then ends normally
        *copies_on = (job.expire_first && !bounded(never, 0u, job.wait_ns, job.err)) ? 0 : 1;
    }
    __syncthreads();
    bool on = *copies_on != 0;

    // factor and inputs do not depend on the previous kernel: fetch before it ends
    ChunkIt ld(nb, nsplit, split, nrow);          // next chunk to fetch (thread 0)
    int ld_st = 0;
    uint32_t fetched = 0;
    auto fetch = [&]() {
        if (!ld.valid()) return;
        ++fetched;
        unsigned char* dst = vsm + ld_st * STG;
        tc::mbar_expect_tx(full + ld_st, STG);
        bulk_g2s(dst, G.Wb + ld.piece(), PIECE, full + ld_st);
        bulk_g2s(dst + PIECE, G.xq + (size_t)ld.r * (CH * 4), XB, full + ld_st);
        ld_st = ld_st == NST - 1 ? 0 : ld_st + 1;
        ld.next();
    };
    if (tid == 0 && on)
        for (int i = 0; i < NST; ++i) fetch();
    grid_wait();

    // the query this thread makes kernel values for (a spare one repeats the last)
    const int m = tid % TQ, h = tid / TQ;
    uint64_t zz[4];
    {
        const float* z = job.z + 4 * (size_t)min(q0 + m, job.Q - 1);
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const float v = __ldcg(z + d) * G.zscale[d];
            zz[d] = tc::f2pack(v, v);
        }
    }
    float mv = 0.0f, mw = 0.0f, cv = 0.0f, cw = 0.0f;
    // kernel values of the chunk in stage st into buffer buf: points h PT .. of
    // the chunk, value k of query m at [k TQ + m]
    auto make = [&](int st, int buf, int r, bool with_mean) {
        const ulonglong2* x = reinterpret_cast<const ulonglong2*>(vsm + st * STG + PIECE) + h * PT;
        float* dst = As + buf * (CH * TQ) + h * PT * TQ + m;
        uint64_t pv = 0ull, pw = 0ull;
#pragma unroll
        for (int p = 0; p < PT / 2; ++p) {
            float k0, k1;
            kernel_pair(zz, x[2 * p], x[2 * p + 1], k0, k1);
            dst[(2 * p) * TQ] = k0;
            dst[(2 * p + 1) * TQ] = k1;
            if (MEAN) {
                if (with_mean) {
                    const ulonglong2 al = __ldg(reinterpret_cast<const ulonglong2*>(G.xq + 4 * (size_t)G.npad) +
                                                (r * CH + h * PT) / 2 + p);
                    const uint64_t kk = tc::f2pack(k0, k1);
                    pv = tc::f2fma(kk, al.x, pv);
                    pw = tc::f2fma(kk, al.y, pw);
                }
            }
        }
        if (MEAN) {
            if (with_mean) {
                float x0, x1;
                tc::f2unpack(pv, x0, x1);
                kahan_add(mv, cv, x0 + x1);
                tc::f2unpack(pw, x0, x1);
                kahan_add(mw, cw, x0 + x1);
            }
        }
    };

    const int lq = lane & 15, c0 = 16 * warp + 8 * (lane >> 4);
    uint64_t acc[NP][8], qs[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        qs[i] = 0ull;
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[i][c] = 0ull;
    }

    ChunkIt mk(nb, nsplit, split, nrow);          // next chunk to make kernel values for
    int mk_st = 0, st = 0, buf = 0;
    uint32_t mk_ph = 0;
    auto make_next = [&]() {
        if (on) on = bounded(full + mk_st, mk_ph, job.wait_ns, job.err);
        make(mk_st, buf, mk.r, MEAN && mk.cb == nb - 1);
        if (++mk_st == NST) {
            mk_st = 0;
            mk_ph ^= 1u;
        }
        mk.next();
    };
    if (mk.valid()) make_next();
    __syncthreads();
    for (ChunkIt it(nb, nsplit, split, nrow); it.valid(); it.next()) {
        const float* Ac = As + buf * (CH * TQ);
        buf ^= 1;
        if (mk.valid()) make_next();
        // rows past this warp's last column are zero
        const int rows = min(CH, CB * it.cb + 16 * warp + 16 - CH * it.r);      // <= 0, 16 or 32
        {
            const float* Bc = reinterpret_cast<const float*>(vsm + st * STG) + c0;
#pragma unroll 4
            for (int k = 0; k < rows; ++k) {
                uint64_t av[NP];
                if constexpr (TQ == 128) {
                    const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(Ac + k * TQ + 4 * lq);
                    const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(Ac + k * TQ + 64 + 4 * lq);
                    av[0] = a0.x; av[1] = a0.y; av[2] = a1.x; av[3] = a1.y;
                } else {
                    av[0] = *reinterpret_cast<const uint64_t*>(Ac + k * TQ + 2 * lq);
                }
                const float4 b0 = *reinterpret_cast<const float4*>(Bc + k * CB);
                const float4 b1 = *reinterpret_cast<const float4*>(Bc + k * CB + 4);
                const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint64_t bb = tc::f2pack(b[c], b[c]);
#pragma unroll
                    for (int i = 0; i < NP; ++i) acc[i][c] = tc::f2fma(av[i], bb, acc[i][c]);
                }
            }
        }
        if (it.last_of_block()) {
#pragma unroll
            for (int i = 0; i < NP; ++i)
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    qs[i] = tc::f2fma(acc[i][c], acc[i][c], qs[i]);
                    acc[i][c] = 0ull;
                }
        }
        __syncthreads();
        if (tid == 0 && on && ld.valid()) {
            tc::fence_proxy_async();              // the CTA's reads of this stage precede the refill
            fetch();
        }
        st = st == NST - 1 ? 0 : st + 1;
    }

    // sum over the two column halves of a warp, the warps, the ranks
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        float x, y;
        tc::f2unpack(qs[i], x, y);
        x += __shfl_xor_sync(0xffffffffu, x, 16);
        y += __shfl_xor_sync(0xffffffffu, y, 16);
        const int q = TQ == 128 ? (i >> 1) * 64 + 4 * lq + 2 * (i & 1) : 2 * lq;
        if (lane < 16) *reinterpret_cast<float2*>(red + warp * TQ + q) = make_float2(x, y);
    }
    if (MEAN) reinterpret_cast<float2*>(vsm + L::mean)[h * TQ + m] = make_float2(mv + cv, mw + cw);
    __syncthreads();
    float sum = 0.0f;
    if (tid < TQ) {
#pragma unroll
        for (int w = 0; w < 8; ++w) sum += red[w * TQ + tid];
        rk[tid] = sum;
    }
    if (nsplit > 1) {
        // rank 0 reads the other ranks' sums through the cluster's shared memory
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (split == 0 && tid < TQ) {
            const uint32_t mine = tc::smem_addr(rk + tid);
            for (int r = 1; r < nsplit; ++r) {
                uint32_t theirs;
                float v;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(theirs) : "r"(mine), "r"(r));
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(theirs) : "memory");
                sum += v;
            }
        }
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    if (split == 0 && tid < TQ && q0 + tid < job.Q) {
        const size_t q = (size_t)(q0 + tid);
        if (MEAN) {
            const float2* mp = reinterpret_cast<const float2*>(vsm + L::mean);
            float2 ms = mp[tid];
#pragma unroll
            for (int i = 1; i < VT / TQ; ++i) {
                ms.x += mp[i * TQ + tid].x;
                ms.y += mp[i * TQ + tid].y;
            }
            const float v = fmaxf(0.0f, G.sf2 - G.qscale * sum);
            if (job.out != 1) {
                job.mean[2 * q] = G.sf2 * ms.x;
                job.var[2 * q] = v;
            }
            if (job.out != 0) {
                job.mean[2 * q + 1] = G.sf2 * ms.y;
                job.var[2 * q + 1] = v;
            }
        } else {
            job.q[(size_t)blockIdx.z * job.Q + q] = sum;
        }
    }
    // copies may still be in flight after a wait ran out: give them a bounded
    // time to land before the shared memory is released
    if (tid == 0 && !on) {
        const uint64_t t0 = tc::global_ns();
        for (uint32_t f = fetched > (uint32_t)NST ? fetched - NST : 0u; f < fetched; ++f)
            while (!tc::mbar_try_wait(full + f % NST, (f / NST) & 1u) && tc::global_ns() - t0 < 200000000ull) {
            }
    }
}

template <int TQ, bool MEAN>
int launch_t(const GpSet& gs, const VarJob& j, int nsplit, bool dependent, cudaStream_t st) {
    auto kern = k_var_fp32<TQ, MEAN>;
    const int smem = VLayout<TQ>::total;
    GPM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    const dim3 grid((unsigned)((j.Q + TQ - 1) / TQ), (unsigned)nsplit, (unsigned)gs.M);
    GPM_CUDA(launch_ex(kern, grid, VT, smem, st, dependent, (unsigned)nsplit, gs, j));
    return GPMPPI_OK;
}

}  // namespace

GpSet single_gp_set(const GpDevice& g, int o) {
    GpSet s = {};
    s.M = 1;
    GpSet::One& G = s.gp[0];
    G.xq = g.xq[o];
    G.Wb = g.Wb[o];
    G.N = g.N;
    G.npad = g.npad;
    G.sf2 = g.sf2[o];
    G.w = 1.0f;
    G.qscale = g.sf2[o] * g.sf2[o];
    for (int d = 0; d < 4; ++d) G.zscale[d] = g.zscale[o][d];
    return s;
}

int launch_var_fp32(const GpSet& gs, const VarJob& j, bool dependent, cudaStream_t st) {
    if (j.Q <= 0) return GPMPPI_OK;
    int nb = 1;
    for (int t = 0; t < gs.M; ++t) nb = gs.gp[t].npad / CB > nb ? gs.gp[t].npad / CB : nb;
    // 128-query tiles where they (with their column blocks dealt to clusters of
    // up to eight) give every SM two CTAs, else 32-query tiles; as many splits as
    // bring about ten waves, so that the last, partly filled one costs little
    const int split_max = nb < 8 ? nb : 8;
    const long long t128 = (long long)(j.Q + 127) / 128 * gs.M;
    const bool wide = t128 * split_max >= 304;
    const long long tiles = wide ? t128 : (long long)(j.Q + 31) / 32 * gs.M;
    int nsplit = 1;
    while (nsplit < split_max && tiles * nsplit < (wide ? 3040 : 608)) nsplit *= 2;
    if (nsplit > split_max) nsplit = split_max;
    if (j.mean) return wide ? launch_t<128, true>(gs, j, nsplit, dependent, st) : launch_t<32, true>(gs, j, nsplit, dependent, st);
    return wide ? launch_t<128, false>(gs, j, nsplit, dependent, st) : launch_t<32, false>(gs, j, nsplit, dependent, st);
}

}  // namespace gpm
