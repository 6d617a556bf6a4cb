// The GP posterior at M queries (gp_predict), FP32: the triangular product of
// tri.cu and its row sums (or, without scratch, one CTA a query), and the means
// with one CTA a query.
#include <mutex>

#include "query.cuh"

namespace gpm {
namespace {

struct PredArgs {
    const float* Z;          // queries, M x 4
    const float* Xs;         // GpDevice::Xs, alpha
    const float* alpha;
    const float* Wb;         // GpDevice::Wb
    const float* V;          // tiles of kTriTile queries, npad columns each
    float* mean;
    float* var;
    int M, N, npad;
    float sf2;
    float zscale[4];
    int out;                 // the output, or -1 for both (shared hyper-parameters)
};

// Stream-ordered scratch of gp_predict: one memory pool per device, for every
// stream and thread.  It keeps up to kPoolKeep bytes between calls (mapping the
// 80 MB of 20000 queries at N = 1000 anew costs more than the call) while GP
// handles exist, and is given back with the last of them.
constexpr uint64_t kPoolKeep = 256ull << 20;
constexpr int kMaxDevices = 64;
std::mutex g_pool_mu;
cudaMemPool_t g_pool[kMaxDevices] = {};
int g_pool_users[kMaxDevices] = {};

int scratch_pool(int device, cudaMemPool_t* out) {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    if (!g_pool[device]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = device;
        GPM_CUDA(cudaMemPoolCreate(&g_pool[device], &props));
        uint64_t keep = kPoolKeep;
        GPM_CUDA(cudaMemPoolSetAttribute(g_pool[device], cudaMemPoolAttrReleaseThreshold, &keep));
    }
    *out = g_pool[device];
    return GPMPPI_OK;
}

constexpr int ST = 128;

__device__ float block_sum(float v, float* red) {
    // deterministic: fixed shuffle tree, then warp partials summed in order
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    float s = 0.0f;
    for (int i = 0; i < ST / 32; ++i) s += red[i];
    return s;
}

// the means, one CTA a query
__global__ void __launch_bounds__(ST) k_pred_mean(const PredArgs p) {
    __shared__ float red[ST / 32];
    const int q = blockIdx.x;
    float zq[4];
    for (int d = 0; d < 4; ++d) zq[d] = p.Z[q * (size_t)4 + d] * p.zscale[d];
    const int o0 = p.out < 0 ? 0 : p.out, o1 = p.out < 0 ? 1 : p.out;
    float m0 = 0.0f, m1 = 0.0f;
    for (int j = threadIdx.x; j < p.N; j += ST) {
        const float4 x = reinterpret_cast<const float4*>(p.Xs)[j];
        const float e0 = zq[0] - x.x, e1 = zq[1] - x.y, e2 = zq[2] - x.z, e3 = zq[3] - x.w;
        const float k = p.sf2 * exp2f(-(e0 * e0 + e1 * e1 + e2 * e2 + e3 * e3));
        m0 += k * p.alpha[2 * j + o0];
        m1 += k * p.alpha[2 * j + o1];
    }
    m0 = block_sum(m0, red);
    m1 = block_sum(m1, red);
    if (threadIdx.x == 0) {
        p.mean[2 * (size_t)q + o0] = m0;
        p.mean[2 * (size_t)q + o1] = m1;
    }
}

// the variances from the rows of v: the squares as 128 threads of a CTA would sum
// them, four threads a query for the four warps' trees, added in order
__global__ void __launch_bounds__(4 * kTriTile) k_pred_var(const PredArgs p) {
    __shared__ float red[4][kTriTile];
    const int w = threadIdx.x / kTriTile, l = threadIdx.x % kTriTile;
    qr::grid_wait();
    red[w][l] = qr::lane_squares<128>(p.V + (size_t)blockIdx.x * p.npad * kTriTile + l, kTriTile, 32 * w, p.N);
    __syncthreads();
    const int q = blockIdx.x * kTriTile + l;
    if (w > 0 || q >= p.M) return;
    float qf = 0.0f;
    for (int i = 0; i < 4; ++i) qf += red[i][l];
    const float s = fmaxf(0.0f, p.sf2 - qf);
    if (p.out != 1) p.var[2 * (size_t)q] = s;
    if (p.out != 0) p.var[2 * (size_t)q + 1] = s;
}

// The variances without scratch, one CTA a query: the same sums in the same order (v
// one chain over the points, the squares as above), every query reading the whole
// factor.  In all, 20000 queries at N = 1000: 1.83 ms, 0.44 by way of V; 200: 152
// against 111 us; 200 at N = 300: 25 against 36.  For calls under stream capture,
// where scratch would be an allocation node, with which a graph may neither be
// instantiated twice at a time nor be a child of another, and for a device without
// room for 128 rows.
__global__ void __launch_bounds__(ST) k_pred_direct(const PredArgs p) {
    extern __shared__ float ks[];                    // N floats
    __shared__ float red[ST / 32];
    const float* z = p.Z + 4 * (size_t)blockIdx.x;
    for (int j = threadIdx.x; j < p.N; j += ST) {
        const float4 x = reinterpret_cast<const float4*>(p.Xs)[j];
        const float e0 = fmaf(z[0], p.zscale[0], -x.x), e1 = fmaf(z[1], p.zscale[1], -x.y);
        const float e2 = fmaf(z[2], p.zscale[2], -x.z), e3 = fmaf(z[3], p.zscale[3], -x.w);
        ks[j] = p.sf2 * qr::ex2(-fmaf(e3, e3, fmaf(e2, e2, fmaf(e0, e0, e1 * e1))));
    }
    __syncthreads();
    float qf = 0.0f;
    for (int i = threadIdx.x; i < p.N; i += ST) {
        const int cb = i / 128;
        const float* w = p.Wb + (size_t)cb * (cb + 1) / 2 * (128 * 128) + i % 128;
        float v = 0.0f;
        for (int j = 0; j <= i; ++j) v = fmaf(ks[j], w[j * 128], v);
        qf = fmaf(v, v, qf);
    }
    qf = block_sum(qf, red);
    const float s = fmaxf(0.0f, p.sf2 - qf);
    if (threadIdx.x == 0 && p.out != 1) p.var[2 * (size_t)blockIdx.x] = s;
    if (threadIdx.x == 0 && p.out != 0) p.var[2 * (size_t)blockIdx.x + 1] = s;
}

}  // namespace

// a GP handle more or less on the device
void scratch_user(int device, int change) {
    if (device < 0 || device >= kMaxDevices) return;
    std::lock_guard<std::mutex> lock(g_pool_mu);
    g_pool_users[device] += change;
    if (g_pool_users[device] == 0 && g_pool[device]) cudaMemPoolTrimTo(g_pool[device], 0);
}

int launch_gp_predict(const GpDevice& g, const float* Z, int M, float* mean, float* var, cudaStream_t st) {
    if (M == 0) return GPMPPI_OK;
    // V in stream-ordered scratch (calls from several threads or streams share
    // nothing), at most what the pool keeps: more queries go in pieces, smaller ones on
    // a full device
    size_t piece = g.npad ? kPoolKeep / 4 / g.npad / kTriTile * kTriTile : (size_t)M;
    if (piece > (size_t)M) piece = (size_t)M;
    float* V = nullptr;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    GPM_CUDA(cudaStreamIsCapturing(st, &cap));
    if (g.npad && cap == cudaStreamCaptureStatusNone) {
        cudaMemPool_t pool = nullptr;
        if (g.device < 0 || g.device >= kMaxDevices) return fail(GPMPPI_ERR_UNSUPPORTED, "gp_predict: device number");
        const int rc0 = scratch_pool(g.device, &pool);
        if (rc0) return rc0;
        cudaError_t e;
        while ((e = cudaMallocFromPoolAsync(
                    (void**)&V, sizeof(float) * ((piece + kTriTile - 1) / kTriTile * kTriTile) * g.npad, pool, st)) ==
                   cudaErrorMemoryAllocation &&
               piece > kTriTile) {
            cudaGetLastError();
            piece = (piece / 2 + kTriTile - 1) / kTriTile * kTriTile;
        }
        if (e != cudaSuccess && e != cudaErrorMemoryAllocation) return cuda_fail(e, "gp_predict: scratch");
        if (e != cudaSuccess) {
            cudaGetLastError();
            V = nullptr;
        }
    }
    if (!V) piece = (size_t)M;
    int rc = GPMPPI_OK;
    for (int o = 0; o < (g.shared ? 1 : 2) && rc == GPMPPI_OK; ++o)
        for (size_t q0 = 0; q0 < (size_t)M && rc == GPMPPI_OK; q0 += piece) {
            PredArgs p;
            p.Z = Z + 4 * q0;
            p.Xs = g.Xs[o];
            p.alpha = g.alpha;
            p.Wb = g.Wb[o];
            p.V = V;
            p.mean = mean + 2 * q0;
            p.var = var + 2 * q0;
            p.M = (int)((size_t)M - q0 < piece ? (size_t)M - q0 : piece);
            p.N = g.N;
            p.npad = g.npad;
            p.sf2 = g.sf2[o];
            for (int d = 0; d < 4; ++d) p.zscale[d] = g.zscale[o][d];
            p.out = g.shared ? -1 : o;
            cudaError_t e;
            if (V) {
                TriJob j = tri_forward(single_gp_set(g, o).gp[0], p.Z, p.M, V);
                j.fusez = 1;
                rc = launch_tri_forward(j, false, st);
                if (rc) break;
                e = launch_ex(k_pred_var, dim3((unsigned)((p.M + kTriTile - 1) / kTriTile)), 4 * kTriTile, 0, st, true, p);
            } else {
                k_pred_direct<<<p.M, ST, sizeof(float) * (g.N > 0 ? g.N : 1), st>>>(p);
                e = cudaGetLastError();
            }
            if (e == cudaSuccess) {
                k_pred_mean<<<p.M, ST, 0, st>>>(p);
                e = cudaGetLastError();
            }
            if (e != cudaSuccess) rc = cuda_fail(e, "gp_predict");
        }
    if (V) {
        const cudaError_t e = cudaFreeAsync(V, st);
        if (e != cudaSuccess && rc == GPMPPI_OK) rc = cuda_fail(e, "gp_predict: scratch");
    }
    return rc;
}

}  // namespace gpm
