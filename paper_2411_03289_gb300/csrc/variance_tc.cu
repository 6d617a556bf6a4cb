// GP variance of many queries on the tensor cores: q = |V_m|^2 with V = K* B^T,
// B = cB L^-1 (cB a power of two per GP), for all queries of a rollout at once.
//
// Operands are split into 16-bit parts (hi + lo in FP16 or BF16: three products
// hi.hi, hi.lo, lo.hi; hi + mid + lo in BF16: six), accumulated in FP32 in
// tensor memory.  hi.hi has its own column set and the small products a second
// one, added when the squares are summed: the tensor core rounds its
// accumulator at every MMA, so the large sum sees one addition per 16 points.
//
// A pair of CTAs (cluster of two, one pair per SM pair, persistent) takes 256
// queries, 128 in each CTA, and the factor's columns in passes of 256.  The MMAs
// are cta_group::2, M = 256 x N <= 256 x K = 16: each CTA stages its own 128
// kernel rows (A) and half of the factor piece (B), so each SM takes in half of
// the factor's bytes and shared memory feeds A and B at half its bandwidth.
// Columns above the diagonal are cut off by 64s (MMAs of N = 256, 192, 128, 64
// over a pass's last 256 points).
//   warps 0-15   kernel rows, eight warps a stage in turn: a thread makes 8 points
//                for two or four queries, so that a training point read from
//                shared memory serves 64 or 128 of them a warp
//   warps 16-19  squares: 64 columns as soon as their last MMA is done (the
//                diagonal ends 0-63 192 points before 192-255), so that only the
//                last quarter of a pass is read with the tensor pipe idle
//   warp 20      rank 0 issues the MMAs of both CTAs; rank 1 tells it when its
//                factor piece of a stage is in place
//   warp 21      factor pieces and training points by bulk copies
//   warp 22      makes a stage's rows visible to the tensor core and tells rank 0
//                (in the warps that make the rows it cost 6 %)
// What bounds it: the tensor pipe (three or six split products of the
// triangle) at large N: K = 16384, T = 100, N = 2048 in FP16 11.0 ms, the measured BF16
// peak of issued products (15.9 ms with 32-point stages and the stage's item divided
// out by the loader each time; the step took 18.4 ms as one kernel over the horizon).
// Up to N = 512 the roles' hand-offs per stage, the tensor pipe 65 % active: 123 us at
// K = 4096, T = 50, N = 500 (the whole rollout as one kernel: 303 us).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "query.cuh"

namespace gpm {
namespace {

using namespace qr;

constexpr int QM = 128;              // queries per CTA
constexpr int PASS = 256;            // factor columns per pass
constexpr int QUART = 64;            // columns per step of the diagonal
constexpr int EPI_WARP = 16, MMA_WARP = 20, LOAD_WARP = 21;
constexpr int NT = 736;              // threads
constexpr int XR = 8;                // ring of the stages' training points
// training points per stage: 64 where the rings then hold three stages, which
// halves every role's hand-offs per point
__host__ __device__ constexpr int stage_points(int parts) { return parts == 2 ? 64 : 32; }
constexpr uint32_t LO_COL = 256;     // TMEM column of the small products' set
constexpr uint64_t kWaitNs = 2000000000ull;

template <int PARTS>
struct TcLayout {
    static constexpr int kc = stage_points(PARTS);
    static constexpr int na = PARTS == 2 ? 3 : 4, nb = PARTS == 2 ? 3 : 4;
    static constexpr int a_part = QM * kc * 2;                    // kernel rows, one part
    static constexpr int b_part = (PASS / 2) * kc * 2;            // factor piece (this CTA's half), one part
    static constexpr int a_stage = PARTS * a_part, b_stage = PARTS * b_part;
    static constexpr int b = na * a_stage;
    static constexpr int x = b + nb * b_stage;
    static constexpr int bars = x + XR * kc * 16;
    // a_raw, a_full [na], b_full, done [nb], x_full [XR], q_done [4], t_free
    static constexpr int tslot = bars + 8 * (2 * na + 2 * nb + XR + 5);
    static constexpr int abort_flag = tslot + 4;
    static constexpr int total = (abort_flag + 4 + 15) / 16 * 16;
};

// ---- the passes of one GP of N points ---------------------------------------
// pass p: columns 256 p .. 256 p + hi - 1, stages 0 .. pass_stages - 1; stage c
// multiplies columns lo(c) .. hi - 1 (those below hold no point of the stage)
__host__ __device__ inline int pass_count(int N) { return (N + PASS - 1) / PASS; }
__host__ __device__ inline int pass_stages(int N, int p, int kc) {
    const int n = (N + kc - 1) / kc, full = PASS / kc * (p + 1);
    return full < n ? full : n;
}
__host__ __device__ inline int pass_hi(int N, int p) {
    const int n = (N - PASS * p + QUART - 1) / QUART * QUART;
    return n < PASS ? n : PASS;
}
__host__ __device__ inline int stage_lo(int p, int c, int kc) {
    const int d = kc * c - PASS * p;
    return d > 0 ? QUART * (d / QUART) : 0;
}
// position of (pass p, stage 0) in the packed factor, in columns x points (only
// the last pass is narrower, and nothing follows it)
__host__ __device__ inline size_t pass_base(int p) { return (size_t)32768 * p * (p - 1) + (size_t)40960 * p; }

// The passes a split of a GP takes: dealt back and forth, largest first; without a
// split and with the batched rollout's sums (BSUM) in their order.
template <bool BSUM>
__host__ __device__ inline int split_pass(int np, int nsplit, int split, int i) {
    if (BSUM && nsplit == 1) return i < np ? i : -1;
    return np - 1 - (i * nsplit + ((i & 1) ? nsplit - 1 - split : split));
}

// the three-part split of a pair: hi, mid, lo (each residual exact)
__device__ __forceinline__ void split3(float a, float b, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    float ra, rb, sa, sb;
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    tc::split_resid<1>(hi, a, b, ra, rb);
    const __nv_bfloat162 m = __floats2bfloat162_rn(ra, rb);
    mid = *reinterpret_cast<const uint32_t*>(&m);
    tc::split_resid<1>(mid, ra, rb, sa, sb);
    const __nv_bfloat162 l = __floats2bfloat162_rn(sa, sb);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

// the two-part split of a pair
template <int FMT>
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
    float ra, rb;
    if (FMT == 0) {
        const __half2 h = __floats2half2_rn(a, b);
        hi = *reinterpret_cast<const uint32_t*>(&h);
        tc::split_resid<0>(hi, a, b, ra, rb);
        const __half2 l = __floats2half2_rn(ra, rb);
        lo = *reinterpret_cast<const uint32_t*>(&l);
    } else {
        const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        hi = *reinterpret_cast<const uint32_t*>(&h);
        tc::split_resid<1>(hi, a, b, ra, rb);
        const __nv_bfloat162 l = __floats2bfloat162_rn(ra, rb);
        lo = *reinterpret_cast<const uint32_t*>(&l);
    }
}

__device__ __forceinline__ uint32_t mapa(const void* p, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(tc::smem_addr(p)), "r"(rank));
    return r;
}
// Arrive on a barrier of either CTA.  What it announces is operands of the async
// proxy (behind a proxy fence, or bulk copies that have landed) or reads that are
// done, so the arrival needs no cluster-scope release: with one it took 900 clocks.
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Every wait gives up after kWaitNs, or once any role of the pair has.
struct Waits {
    volatile int* flag;
    uint32_t peer_flag;
    unsigned int* err;
    __device__ bool poll(uint64_t* bar, uint32_t parity) const {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(tc::smem_addr(bar)), "r"(parity)
            : "memory");
        return ok != 0;
    }
    __device__ bool operator()(uint64_t* bar, uint32_t parity) const {
        if (poll(bar, parity)) return true;
        const uint64_t t0 = tc::global_ns();
        while (!poll(bar, parity)) {
            if (*flag) return false;
            if (tc::global_ns() - t0 > kWaitNs) {
                *flag = 1;
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_flag), "r"(1) : "memory");
                if (err) atomicOr(err, 1u);
                return false;
            }
        }
        return true;
    }
};

// commit: arrives on the barrier at this offset in both CTAs of the pair once
// the MMAs issued so far are done
__device__ __forceinline__ void commit2_elect(uint64_t* bar) {
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}" ::"r"(
            tc::smem_addr(bar)),
        "h"((uint16_t)3)
        : "memory");
}

// Two K-steps of the two-part split: A_hi B_hi into d, A_hi B_lo and
// A_lo B_hi into d + LO_COL; the second K-step's operands sa and sb further on.
// The first product of each set accumulates only if acc != 0.
__device__ __forceinline__ void stage_split2(uint32_t d, uint64_t ah, uint64_t al, uint64_t bh, uint64_t bl,
                                             uint64_t sa, uint64_t sb, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred e, p0, p1;\n\t"
        ".reg .b32 dl;\n\t.reg .b64 ah1, al1, bh1, bl1;\n\t"
        "add.u32 dl, %0, 256;\n\t"
        "add.u64 ah1, %1, %5;\n\tadd.u64 al1, %2, %5;\n\tadd.u64 bh1, %3, %6;\n\tadd.u64 bl1, %4, %6;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p0, %8, 0;\n\t"
        "setp.ne.b32 p1, 1, 0;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %3, %7, p0;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [dl], %1, %4, %7, p0;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [dl], %2, %3, %7, p1;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], ah1, bh1, %7, p1;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [dl], ah1, bl1, %7, p1;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [dl], al1, bh1, %7, p1;\n\t}" ::"r"(d),
        "l"(ah), "l"(al), "l"(bh), "l"(bl), "l"(sa), "l"(sb), "r"(idesc), "r"(acc)
        : "memory");
}

// One K-step of the three-part split: A_hi B_hi into d; A_hi B_mid, A_mid B_hi,
// A_hi B_lo, A_lo B_hi, A_mid B_mid into d + LO_COL.
__device__ __forceinline__ void step_split3(uint32_t d, uint64_t ah, uint64_t am, uint64_t al, uint64_t bh,
                                            uint64_t bm, uint64_t bl, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred e, p0, p1;\n\t.reg .b32 dl;\n\t"
        "add.u32 dl, %0, 256;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p0, %8, 0;\n\t"
        "setp.ne.b32 p1, 1, 0;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %4, %7, p0;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [dl], %1, %5, %7, p0;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [dl], %2, %4, %7, p1;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [dl], %1, %6, %7, p1;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [dl], %3, %4, %7, p1;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [dl], %2, %5, %7, p1;\n\t}" ::"r"(d),
        "l"(ah), "l"(am), "l"(al), "l"(bh), "l"(bm), "l"(bl), "r"(idesc), "r"(acc)
        : "memory");
}

// FMT: 0 = FP16 hi/lo, 1 = BF16 hi/lo, 2 = BF16 hi/mid/lo.  BSUM: the squares in the
// order of the batched rollout (rollout_mma.cu), where the two halves of a pass's
// columns are summed apart, 32 columns at a time in four chains, pass after pass.
// The MMAs of a column are the same products in the same order there and here, so
// that q is the same bits (what is cut off here are products with zero).  With a
// split the 32-column sums go out, and the stage costs add them.  11.3 ms at
// K = 16384, T = 100, N = 2048, FP16, as in the other order (4 % more with chains
// packed across registers that are not loaded as pairs).
template <int FMT, bool BSUM>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NT, 1) k_var_tc(const GpSet gs, const VarTcJob job) {
    extern __shared__ __align__(1024) unsigned char tsm[];
    constexpr int PARTS = FMT == 2 ? 3 : 2;
    using L = TcLayout<PARTS>;
    constexpr int NA = L::na, NBP = L::nb, KC = L::kc;
    uint64_t* a_raw = reinterpret_cast<uint64_t*>(tsm + L::bars);
    uint64_t* a_full = a_raw + NA;
    uint64_t* b_full = a_full + NA;
    uint64_t* done = b_full + NBP;             // the MMAs of a stage, by its piece's slot
    uint64_t* x_full = done + NBP;
    uint64_t* q_done = x_full + XR;
    uint64_t* t_free = q_done + 4;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(tsm + L::tslot);
    volatile int* flag = reinterpret_cast<volatile int*>(tsm + L::abort_flag);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = blockIdx.x & 1u;
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int ntiles = (job.Q + 2 * QM - 1) / (2 * QM);
    const int nitems = ntiles * gs.M * job.nsplit;

    if (tid == 0) {
        for (int i = 0; i < NA; ++i) {
            tc::mbar_init(a_raw + i, 8);
            tc::mbar_init(a_full + i, 2);                                // rank 0's: either CTA's rows
        }
        for (int i = 0; i < NBP; ++i) {
            tc::mbar_init(b_full + i, rank == 0 ? 2 : 1);                // rank 0's: the peer's piece too
            tc::mbar_init(done + i, 1);
        }
        for (int i = 0; i < XR; ++i) tc::mbar_init(x_full + i, 1);
        for (int i = 0; i < 4; ++i) tc::mbar_init(q_done + i, 1);
        tc::mbar_init(t_free, 8);
        *flag = 0;
        tc::fence_mbar_init();
    }
    if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(tc::smem_addr(tslot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc::fence_before_sync();
    __syncthreads();
    cluster_sync();                            // barriers and columns of both CTAs are ready
    tc::fence_after_sync();
    const uint32_t taddr = *tslot;
    const Waits wait = {flag, mapa((const void*)flag, rank ^ 1u), job.err};

    // Every role goes through the same items (tile, GP, split), passes and stages.
    uint32_t n = 0;                            // stages so far
    int sa = 0, sb = 0;                        // ring positions and the parities of their current use
    uint32_t pa = 0, pb = 0;
    auto advance = [&]() {
        ++n;
        if (++sa == NA) {
            sa = 0;
            pa ^= 1u;
        }
        if (++sb == NBP) {
            sb = 0;
            pb ^= 1u;
        }
    };
    bool ok = true;

    if (warp < EPI_WARP) {
        // ---------------- kernel rows --------------------------------------------
        constexpr int SLABS = KC / 8, NQ = SLABS / 2;       // slabs of 8 points; queries per thread
        const int slab = warp % SLABS, m0 = 32 * NQ * ((warp & 7) / SLABS) + lane;
        const uint32_t turn = (uint32_t)(warp >> 3);        // the stages this warp takes: n = turn (mod 2)
        grid_wait();
        const float4* zp = reinterpret_cast<const float4*>(job.z);
        auto query = [&](int item, int m) {
            const int q = (item % ntiles) * (2 * QM) + (int)rank * QM + m;
            return __ldcg(zp + min(q, job.Q - 1));          // spare rows repeat the last query
        };
        float4 zn[NQ];
#pragma unroll
        for (int r = 0; r < NQ; ++r) zn[r] = pair < nitems ? query(pair, m0 + 32 * r) : make_float4(0, 0, 0, 0);
        for (int item = pair; item < nitems && ok; item += npairs) {
            const int ts = item / ntiles;
            const GpSet::One& G = gs.gp[ts / job.nsplit];
            const int split = ts % job.nsplit, np = pass_count(G.N);
            float z[NQ][4];
#pragma unroll
            for (int r = 0; r < NQ; ++r) {
                z[r][0] = zn[r].x * G.zscale[0];
                z[r][1] = zn[r].y * G.zscale[1];
                z[r][2] = zn[r].z * G.zscale[2];
                z[r][3] = zn[r].w * G.zscale[3];
                // the next tile's queries, in flight meanwhile
                if (item + npairs < nitems) zn[r] = query(item + npairs, m0 + 32 * r);
            }
            for (int i = 0, p; ok && (p = split_pass<BSUM>(np, job.nsplit, split, i)) >= 0; ++i) {
                const int ns = pass_stages(G.N, p, KC);
                for (int c = 0; c < ns; ++c) {
                    if ((n & 1u) != turn) {
                        advance();
                        continue;
                    }
                    const bool got = wait(x_full + n % XR, (n / XR) & 1u);
                    const ulonglong2* x = reinterpret_cast<const ulonglong2*>(tsm + L::x + (n % XR) * (KC * 16)) + 8 * slab;
                    // two queries at a time share the points' registers; the first two are
                    // made before the slot is free
                    uint32_t hi_[2][4], lo_[2][4], mid_[2][PARTS == 3 ? 4 : 1];
                    bool room = true;
#pragma unroll
                    for (int r0 = 0; r0 < NQ; r0 += 2) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const ulonglong2 xa = x[2 * q], xb = x[2 * q + 1];
#pragma unroll
                            for (int r = 0; r < 2; ++r) {
                                uint64_t zz[4];
#pragma unroll
                                for (int d = 0; d < 4; ++d) zz[d] = tc::f2pack(z[r0 + r][d], z[r0 + r][d]);
                                float k0, k1;
                                kernel_pair(zz, xa, xb, k0, k1);
                                if constexpr (PARTS == 3) split3(k0, k1, hi_[r][q], mid_[r][q], lo_[r][q]);
                                else split2<FMT>(k0, k1, hi_[r][q], lo_[r][q]);
                            }
                        }
                        if (r0 == 0) {
                            // A warp takes every second stage, so that with a ring of three its
                            // waits on a slot all have one parity.  The phase before is over all
                            // the same: two stages ago it saw the commit of stage n - NA - 2, and
                            // the slot's last use, stage n - NA - NBP, was committed before that.
                            static_assert(NBP >= 2, "the slot's last use is older than the last commit seen");
                            room = n < (uint32_t)NA || wait(done + (n - NA) % NBP, ((n - NA) / NBP) & 1u);
                            ok = __all_sync(0xffffffffu, got && room);
                            if (!ok) break;
                        }
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            unsigned char* dst = tsm + sa * L::a_stage + slab * (QM * 16) + (m0 + 32 * (r0 + r)) * 16;
                            *reinterpret_cast<uint4*>(dst) = make_uint4(hi_[r][0], hi_[r][1], hi_[r][2], hi_[r][3]);
                            if constexpr (PARTS == 3)
                                *reinterpret_cast<uint4*>(dst + L::a_part) =
                                    make_uint4(mid_[r][0], mid_[r][1], mid_[r][2], mid_[r][3]);
                            *reinterpret_cast<uint4*>(dst + (PARTS - 1) * L::a_part) =
                                make_uint4(lo_[r][0], lo_[r][1], lo_[r][2], lo_[r][3]);
                        }
                    }
                    if (!ok) break;
                    __syncwarp();
                    if (lane == 0) arrive(a_raw + sa);
                    advance();
                }
            }
        }
    } else if (warp < MMA_WARP) {
        // ---------------- sums of squares ----------------------------------------
        const int e = warp - EPI_WARP;                      // TMEM lanes 32 e .. 32 e + 31
        const uint32_t row = taddr + ((uint32_t)(32 * e) << 16);
        const uint32_t t_free0 = mapa(t_free, 0u);
        uint32_t qph = 0;                                   // bit j: parity of q_done[j]'s next phase
        for (int item = pair; item < nitems && ok; item += npairs) {
            const int ts = item / ntiles, tile = item % ntiles;
            const GpSet::One& G = gs.gp[ts / job.nsplit];
            const int split = ts % job.nsplit, np = pass_count(G.N);
            const int q = tile * (2 * QM) + (int)rank * QM + 32 * e + lane;
            float sum = 0.0f, half2 = 0.0f;
            for (int i = 0, p; ok && (p = split_pass<BSUM>(np, job.nsplit, split, i)) >= 0; ++i) {
                const int nq = pass_hi(G.N, p) / QUART;
                for (int j = 0; j < nq; ++j) {
                    ok = __all_sync(0xffffffffu, wait(q_done + j, (qph >> j) & 1u));
                    if (!ok) break;
                    qph ^= 1u << j;
                    tc::fence_after_sync();
                    if constexpr (BSUM) {
                        const bool second = j >= (job.even ? 2 : (nq + 1) / 2);
#pragma unroll
                        for (int cc = 0; cc < QUART; cc += 32) {
                            float g[4];
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                float v[16], w[16];
                                const uint32_t col = row + (uint32_t)(QUART * j + cc + 16 * h);
                                tc::tmem_ld16x2(col, col + LO_COL, v, w);
                                // pairs of neighbouring columns (a register pair as loaded)
                                // are added, each chain's squares one by one
                                float x[16], s0 = 0.0f, s1 = 0.0f;
#pragma unroll
                                for (int k = 0; k < 16; k += 2)
                                    tc::f2unpack(tc::f2add(tc::f2pack(v[k], v[k + 1]), tc::f2pack(w[k], w[k + 1])), x[k], x[k + 1]);
#pragma unroll
                                for (int k = 0; k < 8; ++k) {
                                    s0 = fmaf(x[k], x[k], s0);
                                    s1 = fmaf(x[8 + k], x[8 + k], s1);
                                }
                                g[2 * h] = s0;
                                g[2 * h + 1] = s1;
                            }
                            const float s32 = (g[0] + g[1]) + (g[2] + g[3]);
                            if (job.nparts > 1) {
                                if (q < job.Q)
                                    job.q[((size_t)(ts / job.nsplit) * job.nparts + 8 * p + 2 * j + cc / 32) * job.Q + q] = s32;
                            } else if (second) {
                                half2 += s32;
                            } else {
                                sum += s32;
                            }
                        }
                        continue;
                    }
#pragma unroll
                    for (int cc = 0; cc < QUART; cc += 16) {
                        float v[16], w[16];
                        const uint32_t col = row + (uint32_t)(QUART * j + cc);
                        tc::tmem_ld16x2(col, col + LO_COL, v, w);
                        uint64_t s0 = 0ull, s1 = 0ull;
#pragma unroll
                        for (int k = 0; k < 16; k += 4) {
                            const uint64_t x0 = tc::f2add(tc::f2pack(v[k], v[k + 1]), tc::f2pack(w[k], w[k + 1]));
                            const uint64_t x1 = tc::f2add(tc::f2pack(v[k + 2], v[k + 3]), tc::f2pack(w[k + 2], w[k + 3]));
                            s0 = tc::f2fma(x0, x0, s0);
                            s1 = tc::f2fma(x1, x1, s1);
                        }
                        float a0, a1, b0, b1;
                        tc::f2unpack(s0, a0, a1);
                        tc::f2unpack(s1, b0, b1);
                        sum += (a0 + a1) + (b0 + b1);
                    }
                }
                if (!ok) break;
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) arrive_cluster(t_free0);
            }
            if (BSUM && job.nparts > 1) continue;
            if (ok && q < job.Q) job.q[(size_t)ts * job.Q + q] = BSUM ? sum + half2 : sum;
        }
    } else if (warp == MMA_WARP && rank == 0) {
        // ---------------- MMA issuer -----------------------------------------------
        constexpr int TYPE = FMT == 0 ? 0 : 1;
        const uint32_t idesc0 = tc::idesc_f16(TYPE, 2 * QM, 0);
        const uint64_t dA0 = tc::smem_desc(tc::smem_addr(tsm), QM * 16, 128);
        uint32_t passes = 0;
        for (int item = pair; item < nitems && ok; item += npairs) {
            const int ts = item / ntiles;
            const int N = gs.gp[ts / job.nsplit].N;
            const int split = ts % job.nsplit, np = pass_count(N);
            for (int i = 0, p; ok && (p = split_pass<BSUM>(np, job.nsplit, split, i)) >= 0; ++i, ++passes) {
                const int ns = pass_stages(N, p, KC), hi = pass_hi(N, p);
                if (passes > 0) {
                    // both CTAs have read the last pass
                    if (!(ok = __all_sync(0xffffffffu, wait(t_free, (passes - 1) & 1u)))) break;
                    tc::fence_after_sync();
                }
                for (int c = 0; c < ns; ++c) {
                    bool go = wait(b_full + sb, pb);
                    go = go && wait(a_full + sa, pa);
                    if (!(ok = __all_sync(0xffffffffu, go))) break;
                    tc::fence_after_sync();
                    const int lo = stage_lo(p, c, KC), cols = hi - lo, h = cols / 2;
                    const uint64_t ah = dA0 + (uint64_t)((sa * L::a_stage) >> 4);
                    const uint64_t bh = tc::smem_desc(tc::smem_addr(tsm) + (uint32_t)(L::b + sb * L::b_stage), (uint32_t)h * 16u, 128);
                    const uint64_t bstep = (uint64_t)(KC * h * 2 / 16);  // one part of the piece
                    const uint32_t idesc = idesc0 | ((uint32_t)(cols >> 3) << 17);
                    const uint64_t a1 = (uint64_t)(L::a_part >> 4);
                    const uint64_t ka = (uint64_t)((2 * QM * 16) >> 4), kb = (uint64_t)(2 * h);
                    if constexpr (PARTS == 2) {
#pragma unroll
                        for (int j = 0; j < KC / 16; j += 2)
                            stage_split2(taddr + (uint32_t)lo, ah + j * ka, ah + a1 + j * ka, bh + j * kb, bh + bstep + j * kb,
                                         ka, kb, idesc, c + j > 0 ? 1u : 0u);
                    } else {
#pragma unroll
                        for (int j = 0; j < KC / 16; ++j)
                            step_split3(taddr + (uint32_t)lo, ah + j * ka, ah + a1 + j * ka, ah + 2 * a1 + j * ka,
                                        bh + j * kb, bh + bstep + j * kb, bh + 2 * bstep + j * kb, idesc,
                                        c + j > 0 ? 1u : 0u);
                    }
                    commit2_elect(done + sb);
                    // columns 64 j .. 64 j + 63 are complete after their diagonal's last stage
                    const int d = KC * c - PASS * p;
                    if (d >= 0 && ((d + KC) % QUART == 0 || c == ns - 1)) commit2_elect(q_done + d / QUART);
                    advance();
                }
            }
        }
        // MMAs in flight land before the pair's shared memory is released
        if (!ok) {
            const uint64_t t0 = tc::global_ns();
            for (uint32_t i = n >= (uint32_t)NBP ? n - NBP : 0u; i < n; ++i)
                while (!tc::mbar_try_wait(done + i % NBP, (i / NBP) & 1u) && tc::global_ns() - t0 < 200000000ull) {
                }
        }
    } else if (warp == MMA_WARP) {
        // ---------------- rank 1: its factor piece of a stage is in place -----------
        if (lane == 0) {
            const uint32_t peer0 = mapa(b_full, 0u);
            for (int item = pair; item < nitems && ok; item += npairs) {
                const int ts = item / ntiles;
                const int N = gs.gp[ts / job.nsplit].N;
                const int split = ts % job.nsplit, np = pass_count(N);
                for (int i = 0, p; ok && (p = split_pass<BSUM>(np, job.nsplit, split, i)) >= 0; ++i) {
                    const int ns = pass_stages(N, p, KC);
                    for (int c = 0; c < ns; ++c) {
                        if (!(ok = wait(b_full + sb, pb))) break;
                        arrive_cluster(peer0 + 8u * (uint32_t)sb);
                        advance();
                    }
                }
            }
        }
    } else if (warp > LOAD_WARP) {
        // ---------------- rows to the tensor core ------------------------------------
        if (lane == 0) {
            const uint32_t a_full0 = mapa(a_full, 0u);
            for (int item = pair; item < nitems && ok; item += npairs) {
                const int ts = item / ntiles;
                const int N = gs.gp[ts / job.nsplit].N;
                const int split = ts % job.nsplit, np = pass_count(N);
                for (int i = 0, p; ok && (p = split_pass<BSUM>(np, job.nsplit, split, i)) >= 0; ++i) {
                    const int ns = pass_stages(N, p, KC);
                    for (int c = 0; c < ns; ++c) {
                        if (!(ok = wait(a_raw + sa, pa))) break;
                        tc::fence_proxy_async();
                        arrive_cluster(a_full0 + 8u * (uint32_t)sa);
                        advance();
                    }
                }
            }
        }
    } else if (lane == 0) {
        // ---------------- factor pieces and training points -------------------------
        // The points of a stage are fetched up to XR stages ahead: their slot is
        // free once the MMAs XR stages earlier are done.
        int xi = pair, xpi = 0;                             // item and number of its next pass
        int xc = 0, xns = 0;                                // stage and stages of the pass being fetched
        const float* xsrc = nullptr;
        uint32_t xn = 0;
        auto next_x_pass = [&]() {
            xc = xns = 0;
            while (xi < nitems && xns == 0) {
                const int ts = xi / ntiles;
                const GpSet::One& G = gs.gp[ts / job.nsplit];
                const int p = split_pass<BSUM>(pass_count(G.N), job.nsplit, ts % job.nsplit, xpi);
                if (p >= 0) {
                    xns = pass_stages(G.N, p, KC);
                    xsrc = G.xq;
                    ++xpi;
                } else {
                    xpi = 0;
                    xi += npairs;
                }
            }
        };
        auto fetch_x = [&]() {
            if (xns == 0) return;
            uint64_t* bar = x_full + xn % XR;
            tc::mbar_expect_tx(bar, KC * 16);
            bulk_g2s(tsm + L::x + (xn % XR) * (KC * 16), xsrc + (size_t)xc * (KC * 4), KC * 16, bar);
            ++xn;
            if (++xc == xns) next_x_pass();
        };
        next_x_pass();
        for (int i = 0; i < XR; ++i) fetch_x();
        for (int item = pair; item < nitems && ok; item += npairs) {
            const int ts = item / ntiles;
            const GpSet::One& G = gs.gp[ts / job.nsplit];
            const int split = ts % job.nsplit, np = pass_count(G.N);
            for (int i = 0, p; ok && (p = split_pass<BSUM>(np, job.nsplit, split, i)) >= 0; ++i) {
                const int ns = pass_stages(G.N, p, KC), hi = pass_hi(G.N, p);
                const unsigned char* src = reinterpret_cast<const unsigned char*>(G.Bt) + pass_base(p) * (2 * PARTS);
                for (int c = 0; c < ns; ++c) {
                    if (n >= (uint32_t)NBP) {
                        if (!(ok = wait(done + sb, pb ^ 1u))) break;
                        fetch_x();
                    }
                    const int cols = hi - stage_lo(p, c, KC);
                    const uint32_t bytes = (uint32_t)(KC * PARTS * cols);      // this CTA's half of the columns
                    tc::mbar_expect_tx(b_full + sb, bytes);
                    bulk_g2s(tsm + L::b + sb * L::b_stage, src + rank * bytes, bytes, b_full + sb);
                    src += 2 * bytes;
                    advance();
                }
            }
        }
        // copies in flight land before the shared memory is released
        if (!ok || *flag) {
            const uint64_t t0 = tc::global_ns();
            for (uint32_t i = n >= (uint32_t)NBP ? n - NBP : 0u; i < n; ++i)
                while (!tc::mbar_try_wait(b_full + i % NBP, (i / NBP) & 1u) && tc::global_ns() - t0 < 200000000ull) {
                }
            for (uint32_t i = xn >= (uint32_t)XR ? xn - XR : 0u; i < xn; ++i)
                while (!tc::mbar_try_wait(x_full + i % XR, (i / XR) & 1u) && tc::global_ns() - t0 < 200000000ull) {
                }
        }
    }
    __syncwarp();
    tc::fence_before_sync();
    __syncthreads();
    cluster_sync();                            // neither CTA leaves while the other still uses it
    if (warp == MMA_WARP)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(taddr) : "memory");
}

// cB L^-1 in the pieces of the passes: (pass, stage) holds, for each CTA of the
// pair, its half of the stage's columns: the parts (hi, lo or hi, mid, lo) one
// after the other, each as slabs of 8 points x (columns / 2) rows.
__global__ void k_pack_tc(const double* __restrict__ Xm, int N, int fmt, double cB, uint16_t* __restrict__ out) {
    const int parts = fmt == 2 ? 3 : 2, kc = stage_points(parts);
    const int p = blockIdx.y, c = blockIdx.x;
    if (c >= pass_stages(N, p, kc)) return;
    const int hi = pass_hi(N, p), lo = stage_lo(p, c, kc), cols = hi - lo, h = cols / 2;
    size_t off = pass_base(p);
    for (int i = 0; i < c; ++i) off += (size_t)(hi - stage_lo(p, i, kc)) * kc;
    uint16_t* dst = out + off * parts;
    for (int idx = threadIdx.x; idx < cols * kc; idx += blockDim.x) {
        const int e = idx % 8, row = (idx / 8) % h, sl = (idx / (8 * h)) % (kc / 8), r = idx / (kc * h);
        const int i = PASS * p + lo + r * h + row, j = kc * c + 8 * sl + e;
        const double v = (i < N && j <= i) ? cB * Xm[(size_t)i * N + j] : 0.0;
        uint16_t* o = dst + r * (parts * h * kc) + sl * (h * 8) + row * 8 + e;
        if (fmt == 0) {
            const __half a = __double2half(v);
            o[0] = __half_as_ushort(a);
            o[h * kc] = __half_as_ushort(__double2half(v - (double)__half2float(a)));
        } else {
            double rest = v;
            for (int q = 0; q < parts; ++q) {              // each residual exact in double
                const __nv_bfloat16 a = __double2bfloat16(rest);
                o[q * h * kc] = __bfloat16_as_ushort(a);
                rest -= (double)__bfloat162float(a);
            }
        }
    }
}

}  // namespace

int build_tc_pieces(GpDevice& g, int fmt) {
    if (g.Bt[fmt] || g.N == 0) return GPMPPI_OK;
    const int rc = set_cB(g);
    if (rc) return rc;
    const int N = g.N, np = pass_count(N), p = np - 1;
    const int parts = fmt == 2 ? 3 : 2, kc = stage_points(parts);
    size_t n = pass_base(p);                     // columns x points
    for (int c = 0; c < pass_stages(N, p, kc); ++c) n += (size_t)(pass_hi(N, p) - stage_lo(p, c, kc)) * kc;
    uint16_t* Bt = nullptr;
    GPM_CUDA(cudaMalloc(&Bt, n * (size_t)(2 * parts)));
    k_pack_tc<<<dim3((unsigned)(PASS / kc * np), (unsigned)np), 256>>>(g.Linv64[0], N, fmt, (double)g.cB, Bt);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        cudaFree(Bt);
        return cuda_fail(e, "tensor-core factor pieces");
    }
    g.Bt[fmt] = Bt;
    return GPMPPI_OK;
}

// Splits of a GP's passes over the pairs of CTAs: the count that gives the least
// estimated time, waves x the longest split (in stages of 256 columns; about
// two stages more for an item's start and end).
int var_tc_splits(const GpSet& gs, int Q, int nsm) {
    const long long tiles = (long long)(Q + 2 * QM - 1) / (2 * QM) * gs.M;
    const int pairs = nsm / 2;
    int best = 1;
    double least = 0.0;
    for (int s = 1; s <= kMaxVarSplits; ++s) {
        int longest = 0;
        for (int t = 0; t < gs.M; ++t) {
            const int np = pass_count(gs.gp[t].N);
            for (int j = 0; j < s; ++j) {
                int w = 0;
                for (int i = 0, p; (p = split_pass<false>(np, s, j, i)) >= 0; ++i) w += 8 * p + 6;
                longest = w > longest ? w : longest;
            }
        }
        const double cost = (double)((tiles * s + pairs - 1) / pairs) * (longest + 2);
        if (s == 1 || cost < least) {
            least = cost;
            best = s;
        }
    }
    return best;
}

int launch_var_tc(const GpSet& gs, const VarTcJob& j, int fmt, int nsm, bool dependent, cudaStream_t st) {
    if (j.Q <= 0) return GPMPPI_OK;
    const long long items = (long long)((j.Q + 2 * QM - 1) / (2 * QM)) * gs.M * j.nsplit;
    const int pairs = (int)(items < nsm / 2 ? items : nsm / 2);
    auto kern = fmt == 2   ? k_var_tc<2, true>
                : j.rps > 0 ? (fmt == 0 ? k_var_tc<0, true> : k_var_tc<1, true>)
                            : (fmt == 0 ? k_var_tc<0, false> : k_var_tc<1, false>);
    const int smem = fmt == 2 ? TcLayout<3>::total : TcLayout<2>::total;
    GPM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    GPM_CUDA(launch_ex(kern, dim3((unsigned)(2 * pairs)), NT, smem, st, dependent, gs, j));
    return GPMPPI_OK;
}

}  // namespace gpm
