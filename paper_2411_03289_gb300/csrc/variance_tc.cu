// GP variance of many queries on the tensor cores: q = |V_m|^2 with V = K* B^T,
// B = cB L^-1 (cB a power of two per GP), for all queries of a rollout at once.
//
// Operands are split into 16-bit parts (hi + lo in FP16 or BF16: three products
// hi.hi, hi.lo, lo.hi; hi + mid + lo in BF16: six), accumulated in FP32 in
// tensor memory.  The tensor core rounds its accumulator at every MMA, so that what
// shares a column set and in which order is part of the result (VarSums): with the
// small products in a set of their own, added when the squares are summed, the large
// sum sees one addition per 16 points.
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
// Up to N = 512 the roles' hand-offs per stage, the tensor pipe 65 % active, and the
// stages that come twice for the slices' orders (15 entries instead of 12): 159 us at
// K = 4096, T = 50, N = 500, 125 us with one order for all columns, which an input in
// six moved beyond rounding at K = 16000, T = 100 (the whole rollout as one kernel:
// 303 us).
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
// pass p: columns 256 p .. 256 p + hi - 1, in 64-column quarters; entry c of a pass
// multiplies one stage of points with some of them (those that hold none of its points
// are left out).  In the order of the points (kSumsTwo, kSumsOne) entry c is stage c
// and the quarters lo(c) / 64 on.  kSumsShares gives every quarter the order that it
// had when a cluster of CTAs held the factor and each CTA took its stages as its share
// of the mean came first: of 257 to 512 points quarter 5 in the order 0 3 4 5 1 2, 6 in
// 0 6 1 .. 5, 7 in 0 7 1 .. 6, of 129 to 256 points quarter 3 in 0 3 1 2, the others
// ascending.  A pass is a common sequence of its quarters' orders, in which some stages
// come twice (11 entries instead of 8 for the last pass of 512 points).
__host__ __device__ inline int pass_count(int N) { return (N + PASS - 1) / PASS; }
__host__ __device__ inline int pass_hi(int N, int p) {
    const int n = (N - PASS * p + QUART - 1) / QUART * QUART;
    return n < PASS ? n : PASS;
}
__host__ __device__ inline int stage_lo(int p, int c, int kc) {
    const int d = kc * c - PASS * p;
    return d > 0 ? QUART * (d / QUART) : 0;
}

// kSumsShares: entry c of a pass in hexadecimal digit c (of two words of eight)
struct Digits {
    unsigned int lo, hi;
    __host__ __device__ int operator[](int c) const { return (int)((c < 8 ? lo >> 4 * c : hi >> 4 * (c - 8)) & 15u); }
};
struct Shares {
    int n;
    Digits stage;           // its stage
    Digits quarters;        // the quarters it multiplies
    Digits done;            // those that are complete after it
    unsigned int order;     // the quarters as they become complete
};
__host__ __device__ inline Shares shares_of(int N, int p) {
    const int h = pass_hi(N, p) / QUART;
    if (p == 1) {
        if (h == 1) return {5, {0x43210u, 0u}, {0x11111u, 0u}, {0x10000u, 0u}, 0x0u};
        if (h == 2) return {8, {0x21543210u, 0u}, {0x22233113u, 0u}, {0x20010000u, 0u}, 0x10u};
        if (h == 3) return {9, {0x15432160u, 0x2u}, {0x26775547u, 0x2u}, {0x04100000u, 0x2u}, 0x120u};
        return {11, {0x54321670u, 0x216u}, {0xEFFDD48Fu, 0x228u}, {0x41000000u, 0x208u}, 0x1320u};
    }
    if (h == 4 && N <= PASS) return {4, {0x2130u, 0u}, {0xCE8Fu, 0u}, {0xC201u, 0u}, 0x3210u};
    const unsigned int all = (1u << h) - 1u;
    return {h, {0x3210u, 0u}, {0x8CEFu & all * 0x1111u, 0u}, {0x8421u, 0u}, 0x3210u};
}
// the bits set in a digit
__host__ __device__ inline int quarter_count(int q) { return (q & 1) + (q >> 1 & 1) + (q >> 2 & 1) + (q >> 3); }

template <int SUMS>
__host__ __device__ inline int pass_stages(int N, int p, int kc) {
    if (SUMS == kSumsShares) return shares_of(N, p).n;
    const int n = (N + kc - 1) / kc, full = PASS / kc * (p + 1);
    return full < n ? full : n;
}
// columns of entry c
template <int SUMS>
__host__ __device__ inline int stage_cols(int N, int p, int c, int kc) {
    if (SUMS == kSumsShares) return QUART * quarter_count(shares_of(N, p).quarters[c]);
    return pass_hi(N, p) - stage_lo(p, c, kc);
}
template <int SUMS>
__host__ __device__ inline int stage_id(int N, int p, int c) {
    return SUMS == kSumsShares ? shares_of(N, p).stage[c] : c;
}
// position of (pass p, stage 0) in the packed factor, in columns x points (only
// the last pass is narrower, and nothing follows it)
__host__ __device__ inline size_t pass_base(int p) { return (size_t)32768 * p * (p - 1) + (size_t)40960 * p; }

// The passes a split of a GP takes: dealt back and forth, largest first; without a
// split in their order.
__host__ __device__ inline int split_pass(int np, int nsplit, int split, int i) {
    if (nsplit == 1) return i < np ? i : -1;
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

// Two K-steps of the two-part split: A_hi B_hi into d, A_hi B_lo into d + hl and
// A_lo B_hi into d + lh; the second K-step's operands sa and sb further on.  The first
// product accumulates only if acc != 0, the second only if acc_hl != 0.
__device__ __forceinline__ void stage_split2(uint32_t d, uint32_t hl, uint32_t lh, uint64_t ah, uint64_t al, uint64_t bh,
                                             uint64_t bl, uint64_t sa, uint64_t sb, uint32_t idesc, uint32_t acc,
                                             uint32_t acc_hl) {
    asm volatile(
        "{\n\t.reg .pred e, p0, p1, p2;\n\t"
        ".reg .b32 d2, d3;\n\t.reg .b64 ah1, al1, bh1, bl1;\n\t"
        "add.u32 d2, %0, %9;\n\tadd.u32 d3, %0, %10;\n\t"
        "add.u64 ah1, %1, %5;\n\tadd.u64 al1, %2, %5;\n\tadd.u64 bh1, %3, %6;\n\tadd.u64 bl1, %4, %6;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p0, %8, 0;\n\t"
        "setp.ne.b32 p2, %11, 0;\n\t"
        "setp.ne.b32 p1, 1, 0;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %3, %7, p0;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [d2], %1, %4, %7, p2;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [d3], %2, %3, %7, p1;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], ah1, bh1, %7, p1;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [d2], ah1, bl1, %7, p1;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [d3], al1, bh1, %7, p1;\n\t}" ::"r"(d),
        "l"(ah), "l"(al), "l"(bh), "l"(bl), "l"(sa), "l"(sb), "r"(idesc), "r"(acc), "r"(hl), "r"(lh), "r"(acc_hl)
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

// FMT: 0 = FP16 hi/lo, 1 = BF16 hi/lo, 2 = BF16 hi/mid/lo.  SUMS: which products share
// a column set, the order of a column's MMAs and of the squares.
//   kSumsTwo     hi.hi apart; the two halves of a pass's columns summed apart, 32
//                columns at a time in four chains, pass after pass
//   kSumsOne     all in one set; the halves of 512 columns, 64 at a time in four chains
//   kSumsShares  hi.lo apart; 64 columns at a time in eight chains, the outermost of
//                the slices first
// The products of a column are the same in the same order as in the batched rollout
// (kSumsShares: as in the cluster of CTAs that had the rollout), so that q is the same
// bits; what is cut off here are products with zero.  With a split the sums of 32 or 64
// columns go out, and k_var_parts adds them.  11.3 ms at K = 16384, T = 100, N =
// 2048, FP16, as with the squares in any order (4 % more with chains packed across
// registers that are not loaded as pairs).
template <int FMT, int SUMS>
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
            for (int i = 0, p; ok && (p = split_pass(np, job.nsplit, split, i)) >= 0; ++i) {
                const int ns = pass_stages<SUMS>(G.N, p, KC);
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
            float sum = 0.0f, half2 = 0.0f, slice[SUMS == kSumsShares ? 8 : 1] = {};
            for (int i = 0, p; ok && (p = split_pass(np, job.nsplit, split, i)) >= 0; ++i) {
                const int nq = pass_hi(G.N, p) / QUART;
                // of the 128-column blocks of a pass of 256 (kSumsOne: 512) columns, those
                // whose halves are summed apart: the first half ends after so many quarters
                int edge = job.even ? 2 : (nq + 1) / 2;
                if (SUMS == kSumsOne) {
                    const int left = (G.N - 2 * PASS * (p / 2) + QUART - 1) / QUART;      // quarters of the 512
                    edge = left >= 8 ? 4 : job.even ? 2 * ((left + 3) / 4) : (left + 1) / 2;
                    edge -= 4 * (p & 1);
                }
                unsigned int order = 0x3210u;
                if constexpr (SUMS == kSumsShares) order = shares_of(G.N, p).order;
                for (int jj = 0; jj < nq; ++jj) {
                    const int j = (int)(order >> 4 * jj & 15u);
                    ok = __all_sync(0xffffffffu, wait(q_done + j, (qph >> j) & 1u));
                    if (!ok) break;
                    qph ^= 1u << j;
                    tc::fence_after_sync();
                    const uint32_t col0 = row + (uint32_t)(QUART * j);
                    float* part = job.q + ((size_t)(ts / job.nsplit) * job.nparts) * job.Q + q;    // with a split
                    auto add = [&](float g, int at) {
                        if (job.nparts > 1) {
                            if (q < job.Q) part[(size_t)at * job.Q] = g;
                        } else if (j >= edge) {
                            half2 += g;
                        } else {
                            sum += g;
                        }
                    };
                    if constexpr (SUMS == kSumsTwo) {
#pragma unroll
                        for (int cc = 0; cc < QUART; cc += 32) {
                            float g[4];
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                float v[16], w[16];
                                tc::tmem_ld16x2(col0 + cc + 16 * h, col0 + cc + 16 * h + LO_COL, v, w);
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
                            add((g[0] + g[1]) + (g[2] + g[3]), 8 * p + 2 * j + cc / 32);
                        }
                    } else if constexpr (SUMS == kSumsOne) {
                        float g[4];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            float v[16], w[16], s0 = 0.0f, s1 = 0.0f;
                            tc::tmem_ld16x2(col0 + 32 * h, col0 + 32 * h + 16, v, w);
#pragma unroll
                            for (int k = 0; k < 16; ++k) {
                                s0 = fmaf(v[k], v[k], s0);
                                s1 = fmaf(w[k], w[k], s1);
                            }
                            g[2 * h] = s0;
                            g[2 * h + 1] = s1;
                        }
                        add((g[0] + g[1]) + (g[2] + g[3]), 4 * p + j);
                    } else {
                        uint64_t s[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                        for (int cc = 0; cc < QUART; cc += 16) {
                            float v[16], w[16];
                            tc::tmem_ld16x2(col0 + cc, col0 + cc + LO_COL, v, w);
#pragma unroll
                            for (int k = 0; k < 16; k += 2) {
                                const uint64_t x = tc::f2add(tc::f2pack(v[k], v[k + 1]), tc::f2pack(w[k], w[k + 1]));
                                s[k / 2 % 4] = tc::f2fma(x, x, s[k / 2 % 4]);
                            }
                        }
                        float g[8];
#pragma unroll
                        for (int k = 0; k < 4; ++k) tc::f2unpack(s[k], g[2 * k], g[2 * k + 1]);
                        const float g64 = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7]));
                        if (job.nparts > 1) {
                            add(g64, 4 * p + j);
                        } else {
#pragma unroll
                            for (int k = 0; k < 8; ++k) slice[k] = k == 4 * p + j ? g64 : slice[k];
                        }
                    }
                }
                if (!ok) break;
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) arrive_cluster(t_free0);
            }
            if (!ok || job.nparts > 1 || q >= job.Q) continue;
            if constexpr (SUMS == kSumsShares) {
                const int last = G.N <= 128 ? 1 : G.N <= 256 ? 3 : 7;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (2 * r >= last) break;
                    sum += slice[r];
                    sum += last == 1 ? slice[1 - r] : last == 3 ? slice[3 - r > 0 ? 3 - r : 0] : slice[7 - r];
                }
            }
            job.q[(size_t)ts * job.Q + q] = sum + half2;
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
            for (int i = 0, p; ok && (p = split_pass(np, job.nsplit, split, i)) >= 0; ++i, ++passes) {
                const int ns = pass_stages<SUMS>(N, p, KC), hi = pass_hi(N, p);
                Shares sh = {};
                if constexpr (SUMS == kSumsShares) sh = shares_of(N, p);
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
                    const uint64_t ah = dA0 + (uint64_t)((sa * L::a_stage) >> 4);
                    const uint64_t a1 = (uint64_t)(L::a_part >> 4), ka = (uint64_t)((2 * QM * 16) >> 4);
                    // the entry's columns, in one run of quarters or (kSumsShares) two
                    int lo = stage_lo(p, c, KC), cols = hi - lo, left = 0;
                    if constexpr (SUMS == kSumsShares) {
                        left = sh.quarters[c];
                        lo = QUART * (__ffs(left) - 1);
                        cols = QUART * (__ffs(~(left >> lo / QUART)) - 1);
                        left &= -1 << (lo + cols) / QUART;
                    }
                    uint32_t bs = (uint32_t)(L::b + sb * L::b_stage);
                    while (true) {
                        const int h = cols / 2;
                        const uint64_t bh = tc::smem_desc(tc::smem_addr(tsm) + bs, (uint32_t)h * 16u, 128);
                        const uint64_t bstep = (uint64_t)(KC * h * 2 / 16);  // one part of the piece
                        const uint64_t kb = (uint64_t)(2 * h);
                        const uint32_t idesc = idesc0 | ((uint32_t)(cols >> 3) << 17);
                        if constexpr (PARTS == 2) {
                            constexpr uint32_t HL = SUMS == kSumsOne ? 0u : LO_COL, LH = SUMS == kSumsTwo ? LO_COL : 0u;
#pragma unroll
                            for (int j = 0; j < KC / 16; j += 2)
                                stage_split2(taddr + (uint32_t)lo, HL, LH, ah + j * ka, ah + a1 + j * ka, bh + j * kb,
                                             bh + bstep + j * kb, ka, kb, idesc, c + j > 0 ? 1u : 0u,
                                             SUMS == kSumsOne || c + j > 0 ? 1u : 0u);
                        } else {
#pragma unroll
                            for (int j = 0; j < KC / 16; ++j)
                                step_split3(taddr + (uint32_t)lo, ah + j * ka, ah + a1 + j * ka, ah + 2 * a1 + j * ka,
                                            bh + j * kb, bh + bstep + j * kb, bh + 2 * bstep + j * kb, idesc,
                                            c + j > 0 ? 1u : 0u);
                        }
                        if (SUMS != kSumsShares || left == 0) break;
                        bs += (uint32_t)(KC * PARTS * cols);      // this CTA's half of the first run
                        lo = QUART * (__ffs(left) - 1);
                        cols = QUART * (__ffs(~(left >> lo / QUART)) - 1);
                        left = 0;
                    }
                    commit2_elect(done + sb);
                    // quarters are complete after their last entry
                    if constexpr (SUMS == kSumsShares) {
                        const int over = sh.done[c];
                        for (int j = 0; j < 4; ++j)
                            if (over >> j & 1) commit2_elect(q_done + j);
                    } else {
                        const int d = KC * c - PASS * p;
                        if (d >= 0 && ((d + KC) % QUART == 0 || c == ns - 1)) commit2_elect(q_done + d / QUART);
                    }
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
                for (int i = 0, p; ok && (p = split_pass(np, job.nsplit, split, i)) >= 0; ++i) {
                    const int ns = pass_stages<SUMS>(N, p, KC);
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
                for (int i = 0, p; ok && (p = split_pass(np, job.nsplit, split, i)) >= 0; ++i) {
                    const int ns = pass_stages<SUMS>(N, p, KC);
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
        int xc = 0, xns = 0, xp = 0, xN = 0;                // entry and entries of the pass being fetched, its pass and GP
        const float* xsrc = nullptr;
        uint32_t xn = 0;
        auto next_x_pass = [&]() {
            xc = xns = 0;
            while (xi < nitems && xns == 0) {
                const int ts = xi / ntiles;
                const GpSet::One& G = gs.gp[ts / job.nsplit];
                const int p = split_pass(pass_count(G.N), job.nsplit, ts % job.nsplit, xpi);
                if (p >= 0) {
                    xns = pass_stages<SUMS>(G.N, p, KC);
                    xsrc = G.xq;
                    xp = p;
                    xN = G.N;
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
            bulk_g2s(tsm + L::x + (xn % XR) * (KC * 16), xsrc + (size_t)stage_id<SUMS>(xN, xp, xc) * (KC * 4), KC * 16, bar);
            ++xn;
            if (++xc == xns) next_x_pass();
        };
        next_x_pass();
        for (int i = 0; i < XR; ++i) fetch_x();
        for (int item = pair; item < nitems && ok; item += npairs) {
            const int ts = item / ntiles;
            const GpSet::One& G = gs.gp[ts / job.nsplit];
            const int split = ts % job.nsplit, np = pass_count(G.N);
            for (int i = 0, p; ok && (p = split_pass(np, job.nsplit, split, i)) >= 0; ++i) {
                const int ns = pass_stages<SUMS>(G.N, p, KC);
                const unsigned char* src = reinterpret_cast<const unsigned char*>(G.Bt) + pass_base(p) * (2 * PARTS);
                for (int c = 0; c < ns; ++c) {
                    if (n >= (uint32_t)NBP) {
                        if (!(ok = wait(done + sb, pb ^ 1u))) break;
                        fetch_x();
                    }
                    // this CTA's half of the columns
                    const uint32_t bytes = (uint32_t)(KC * PARTS * stage_cols<SUMS>(G.N, p, c, KC));
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

// |V_m|^2 of a query from its parts (stride Q): a part for every 32 columns (kSumsTwo)
// or 64, added in the order of one CTA pair.
__device__ float parts_sum(int sums, int even, const float* qp, size_t Q, int N) {
    float h0 = 0.0f, h1 = 0.0f;
    const int ns = (N + 63) / 64;
    if (sums == kSumsShares) {
        const int last = N <= 128 ? 1 : N <= 256 ? 3 : 7;
        for (int r = 0; 2 * r < last; ++r) {
            if (r < ns) h0 += qp[(size_t)r * Q];
            if (last - r < ns) h0 += qp[(size_t)(last - r) * Q];
        }
        return h0;
    }
    // eight parts at a time: a pass of 256 columns in 32s or of 512 in 64s, its halves
    // (of the 128-column blocks that it has) apart
    const bool two = sums == kSumsTwo;
    for (int n = two ? 2 * ns : ns; n > 0; n -= 8, qp += 8 * Q) {
        int h = 4;
        if (two) h = even || n >= 8 ? 4 : (n + 2) / 4 * 2;
        else if (n < 8) h = even ? 2 * ((n + 3) / 4) : (n + 1) / 2;
        float g[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) g[j] = j < n ? qp[j * Q] : 0.0f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (j < n && j < h) h0 += g[j];
            if (j < n && j >= h) h1 += g[j];
        }
    }
    return h0 + h1;
}

// after a split: the first part of every query and GP becomes its sum.  A launch of its
// own: in the stage costs' loads the parts' loop cost 15 to 70 us.
__global__ void __launch_bounds__(256) k_var_parts(const GpSet gs, const VarTcJob job) {
    grid_wait();
    const int q = blockIdx.x * 256 + threadIdx.x;
    if (q >= job.Q) return;
    float* p = job.q + (size_t)blockIdx.y * job.nparts * job.Q + q;
    *p = parts_sum(job.sums, job.even, p, (size_t)job.Q, gs.gp[blockIdx.y].N);
}

// cB L^-1 in the pieces of the passes: (pass, entry) holds, for each CTA of the
// pair, its half of every run of the entry's columns, a run's parts (hi, lo or hi, mid,
// lo) one after the other, each as slabs of 8 points x (columns / 2) rows.
template <int SUMS>
__global__ void k_pack_tc(const double* __restrict__ Xm, int N, int fmt, double cB, uint16_t* __restrict__ out) {
    const int parts = fmt == 2 ? 3 : 2, kc = stage_points(parts);
    const int p = blockIdx.y, c = blockIdx.x;
    if (c >= pass_stages<SUMS>(N, p, kc)) return;
    const int cols = stage_cols<SUMS>(N, p, c, kc), st = stage_id<SUMS>(N, p, c);
    // the runs of quarters: start and columns of the first, start of the second
    int lo = stage_lo(p, c, kc), n0 = cols, lo1 = 0;
    if (SUMS == kSumsShares) {
        const int q = shares_of(N, p).quarters[c];
        lo = QUART * (__ffs(q) - 1);
        n0 = QUART * (__ffs(~(q >> lo / QUART)) - 1);
        const int rest = q & (-1 << (lo + n0) / QUART);
        lo1 = rest ? QUART * (__ffs(rest) - 1) : 0;
    }
    size_t off = pass_base(p);
    for (int i = 0; i < c; ++i) off += (size_t)stage_cols<SUMS>(N, p, i, kc) * kc;
    for (int idx = threadIdx.x; idx < cols * kc; idx += blockDim.x) {
        const int r = idx / (kc * cols / 2);
        int in = idx % (kc * cols / 2);
        uint16_t* dst = out + off * parts + (size_t)r * (parts * kc * cols / 2);
        const bool second = in >= kc * n0 / 2;
        if (second) {
            in -= kc * n0 / 2;
            dst += parts * kc * n0 / 2;
        }
        const int h = (second ? cols - n0 : n0) / 2;
        const int e = in % 8, row = (in / 8) % h, sl = in / (8 * h);
        const int i = PASS * p + (second ? lo1 : lo) + r * h + row, j = kc * st + 8 * sl + e;
        const double v = (i < N && j <= i) ? cB * Xm[(size_t)i * N + j] : 0.0;
        uint16_t* o = dst + sl * (h * 8) + row * 8 + e;
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

int build_tc_pieces(GpDevice& g, int fmt, bool shares) {
    uint16_t*& made = shares ? g.Bs[fmt] : g.Bt[fmt];
    if (made || g.N == 0) return GPMPPI_OK;
    const int rc = set_cB(g);
    if (rc) return rc;
    const int N = g.N, np = pass_count(N), p = np - 1;
    const int parts = fmt == 2 ? 3 : 2, kc = stage_points(parts);
    // columns x points: the same for either order
    size_t n = pass_base(p);
    for (int c = 0; c < pass_stages<kSumsTwo>(N, p, kc); ++c) n += (size_t)stage_cols<kSumsTwo>(N, p, c, kc) * kc;
    uint16_t* Bt = nullptr;
    GPM_CUDA(cudaMalloc(&Bt, n * (size_t)(2 * parts)));
    const dim3 grid((unsigned)(shares ? 11 : PASS / kc * np), (unsigned)np);
    auto kern = shares ? k_pack_tc<kSumsShares> : k_pack_tc<kSumsTwo>;
    kern<<<grid, 256>>>(g.Linv64[0], N, fmt, (double)g.cB, Bt);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        cudaFree(Bt);
        return cuda_fail(e, "tensor-core factor pieces");
    }
    made = Bt;
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
                for (int i = 0, p; (p = split_pass(np, s, j, i)) >= 0; ++i) w += 8 * p + 6;
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
    auto kern = fmt == 2               ? k_var_tc<2, kSumsTwo>
                : j.sums == kSumsTwo ? (fmt == 0 ? k_var_tc<0, kSumsTwo> : k_var_tc<1, kSumsTwo>)
                : j.sums == kSumsOne ? (fmt == 0 ? k_var_tc<0, kSumsOne> : k_var_tc<1, kSumsOne>)
                                     : (fmt == 0 ? k_var_tc<0, kSumsShares> : k_var_tc<1, kSumsShares>);
    const int smem = fmt == 2 ? TcLayout<3>::total : TcLayout<2>::total;
    GPM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    GPM_CUDA(launch_ex(kern, dim3((unsigned)(2 * pairs)), NT, smem, st, dependent, gs, j));
    if (j.nparts > 1)
        GPM_CUDA(launch_ex(k_var_parts, dim3((unsigned)((j.Q + 255) / 256), (unsigned)gs.M), 256, 0, st, true, gs, j));
    return GPMPPI_OK;
}

}  // namespace gpm
