// K1: pooled block scores.
//   pool_kernel   : one warp per (Q|K, image, head, 64-token block); 128-bit coalesced loads,
//                   fp64 accumulation, mean over the valid tokens of the block.
//                   HBM-bound: reads Q and K exactly once.
//   scores_kernel : S[i][j] = Qbar[i,:] . Kbar[j,:] in fp64 (fp64 mma.sync fragments), rounded once to fp32.
#include "scoring.cuh"

using namespace scoring;

namespace {

// One warp per (Q|K, image, head, 64-token block).  No shared memory.  The batches of eight loads are not unrolled into
// one another: that keeps the kernel under 85 registers, six thread blocks per SM (measured 29 against 40 us on the
// FLUX 1024^2 shapes, where 125 registers left four).
template <int D>
__global__ void __launch_bounds__(128, 6) pool_kernel(const uint16_t* q, const uint16_t* k,
                                                   TensorGeom g, ImgList imgs, double* __restrict__ pooled,
                                                   const DevPlan* plan, int n_cap) {
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int blk = blockIdx.x * 4 + warp, h = blockIdx.y;
    grid_dependency_wait();                           // first kernel of a call: what comes before it may still be running
    if (blk >= g.nb) return;
    const int which = blockIdx.z / n_cap;             // 0 = Q, 1 = K
    const int p = blockIdx.z - which * n_cap;
    if (plan && p >= __ldcg(&plan->sparse.n)) return;  // device-resident plan: fewer images than the grid covers
    const int batch = plan ? __ldcg(&plan->sparse.batch[p]) : imgs.batch[p];
    const uint16_t* base = (which ? k : q) + (long long)batch * g.stride_b + (long long)(g.h0 + h) * g.stride_h + (long long)(blk * 64) * g.stride_n;
    double* out = pooled + ((((long long)which * n_cap + p) * g.H + h) * g.nb + blk) * D;
    // the next kernel's start: not before the loads are through (steps of 17 to 25 us: 1 to 2 %)
    pool_block<D>(base, g.stride_n, min(64, g.N - blk * 64), out, lane, [] { grid_dependency_launch(); });
}

// 32 x 32 tile of S per thread block, eight warps; a warp owns two fragments of 8 x 8 outputs side by side.  The two
// operands (32 block means each) are copied to shared memory as a whole, the first half of the channels as one group of
// asynchronous copies and the second as another: a thread block has little else to do than to wait for them, and one
// round trip is what that costs (chunks of 32 channels through registers cost one each: 28.6 -> 24 us at 264 blocks).
// Rows are padded to D + 4 doubles: the fragment loads then touch every bank pair twice, the minimum for 32 eight-byte
// lanes.  Every output accumulates its products in ascending order of the four-channel groups.
template <int D>
__global__ void __launch_bounds__(256) scores_kernel(const double* pooled, TensorGeom g, int n_img,
                                                     float* __restrict__ scores, const DevPlan* plan) {
    constexpr int T = 32, LDS = D + 4;
    extern __shared__ __align__(16) double tiles[];
    double* sq = tiles;
    double* sk = tiles + T * LDS;
    const int ph = blockIdx.z;                       // p * H + h
    // The block means come from the kernel before, which may still be running when this one starts: wait for its end,
    // and read them past the L1, whose lines no such wait is known to refresh.
    grid_dependency_wait();
    grid_dependency_launch();
    if (plan && ph >= __ldcg(&plan->sparse.n) * g.H) return;
    const int i0 = blockIdx.y * T, j0 = blockIdx.x * T;
    const double* pq = pooled + ((long long)ph * g.nb + i0) * D;
    const double* pk = pooled + (((long long)n_img * g.H + ph) * g.nb + j0) * D;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
#pragma unroll
        for (int x = 0; x < T * D / 4 / 256; ++x) {
            const int e = threadIdx.x + 256 * x, r = e / (D / 4), c = half * (D / 2) + 2 * (e % (D / 4));
            const bool vq = i0 + r < g.nb, vk = j0 + r < g.nb;
            copy16_async(sq + r * LDS + c, vq ? pq + r * D + c : pooled, vq);
            copy16_async(sk + r * LDS + c, vk ? pk + r * D + c : pooled, vk);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, gr = lane >> 2, c = lane & 3;
    const int ri = (warp >> 1) * 8, cj = (warp & 1) * 16;                // the warp's corner inside the tile
    const double* aq = sq + (ri + gr) * LDS + c;
    const double* bk = sk + (cj + gr) * LDS + c;
    double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        if (half == 0) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
#pragma unroll 8
        for (int d = half * (D / 2); d < (half + 1) * (D / 2); d += 4) {
            const double a = aq[d];
            dmma_8x8x4(acc[0][0], acc[0][1], a, bk[d]);
            dmma_8x8x4(acc[1][0], acc[1][1], a, bk[8 * LDS + d]);
        }
    }
    float* so = scores + (long long)ph * g.nb * g.nb;
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int i = i0 + ri + gr, j = j0 + cj + 8 * b + 2 * c + e;
            if (i < g.nb && j < g.nb) so[(long long)i * g.nb + j] = (float)acc[b][e];
        }
}

constexpr int scores_smem_bytes(int D) { return 2 * 32 * (D + 4) * (int)sizeof(double); }

}  // namespace

cudaError_t launch_block_pool(const void* q, const void* k, const TensorGeom& g, const ImgList& imgs,
                              double* pooled, cudaStream_t s, const DevPlan* plan, int n_cap) {
    if (!plan) n_cap = imgs.n;
    dim3 grid((g.nb + 3) / 4, g.H, 2 * n_cap);
    // Small inputs ask for the shared-memory split that the attention kernel needs, so that the SMs need not be drained and
    // split anew between the kernels of the step; that takes the loads' L1 away, which costs large inputs more (17 MB:
    // 47.3 -> 44.3 us a step; 27 MB: 265.0 -> 265.8, 54 MB: 204.3 -> 205.8, 208 MB: 999 -> 1003).
    const long long bytes = 4ll * n_cap * g.H * g.N * g.D;
    const int carveout = bytes <= (20ll << 20) ? (int)cudaSharedmemCarveoutMaxShared : -1;
    return launch_kernel_carveout(g.D == 128 ? pool_kernel<128> : pool_kernel<64>, grid, dim3(128), 0, s, carveout,
                                  static_cast<const uint16_t*>(q), static_cast<const uint16_t*>(k), g, imgs, pooled, plan,
                                  n_cap);
}

cudaError_t launch_block_scores(const double* pooled, const TensorGeom& g, int n_img, float* scores,
                                cudaStream_t s, const DevPlan* plan) {
    // with a plan n_img is the capacity.  32 x 32 tiles at every length: against 64 x 64 tiles they waste less of
    // the ragged edge and fill the SMs more evenly (30 against 35 us at 264 blocks, where 64 x 64 pads 264 to 320)
    const dim3 grid((g.nb + 31) / 32, (g.nb + 31) / 32, n_img * g.H);
    return launch_kernel(g.D == 128 ? scores_kernel<128> : scores_kernel<64>, grid, dim3(256), scores_smem_bytes(g.D), s,
                         pooled, g, n_img, scores, plan);
}

cudaError_t scoring_static_init() {
    const cudaError_t e = cudaFuncSetAttribute(scores_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, scores_smem_bytes(128));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(scores_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, scores_smem_bytes(64));
}

// ---------------------------------------------------------------------------------------------
// rapid3_block_scores_static: the scoring pass for callers that may not allocate device memory.
//
// The block means (the only scratch of this pass) live in the file-scope array below instead of
// a cudaMalloc'ed workspace.  The array is part of the loaded module: every GPU that loads the
// library holds RAPID3_STATIC_SCRATCH_DOUBLES * 8 bytes (16 MiB) until the process exits.
// In host code the array's name is only a stand-in for the symbol, not a device address, so the
// address is looked up once per device with cudaGetSymbolAddress (with that device current) and
// that pointer is what the kernels get.
#include <mutex>

#define RAPID3_STATIC_SCRATCH_DOUBLES (1ll << 21)   // 16 MiB of fp64 block means
static __device__ __align__(256) double g_static_pool_scratch[RAPID3_STATIC_SCRATCH_DOUBLES];

namespace {

constexpr int RAPID3_STATIC_MAX_DEVICES = 64;

std::mutex g_static_mu;
double* g_static_ptr[RAPID3_STATIC_MAX_DEVICES] = {};

// Device address of the scratch array on the current device (looked up on first use per device).
int static_scratch(double** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= RAPID3_STATIC_MAX_DEVICES) return RAPID3_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_pool_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return RAPID3_ERR_CUDA;
        }
        g_static_ptr[dev] = static_cast<double*>(p);
    }
    *out = g_static_ptr[dev];
    return RAPID3_OK;
}

}  // namespace

extern "C" int rapid3_block_scores_static(const rapid3_shape* s, const void* q, const void* k,
                                          const int32_t* img_idx_host, int n_img, float* scores, void* stream) {
    if (!s || !q || !k || !scores) return RAPID3_ERR_INVALID_ARG;
    if (s->block != RAPID3_BLOCK || (s->D != 64 && s->D != 128)) return RAPID3_ERR_UNSUPPORTED;
    if (s->B_max < 1 || s->B_max > RAPID3_MAX_IMG || s->H < 1 || s->H > 65535) return RAPID3_ERR_INVALID_ARG;
    if ((long long)s->B_max * s->H > 65535) return RAPID3_ERR_UNSUPPORTED;     // (image, head) pairs index a grid dimension
    if (s->n_text < 0 || s->n_image < 0) return RAPID3_ERR_INVALID_ARG;
    const long long N = (long long)s->n_text + s->n_image;
    if (N < 1) return RAPID3_ERR_INVALID_ARG;
    if (N > 64ll * RAPID3_MAX_NB) return RAPID3_ERR_UNSUPPORTED;
    if (s->stride_n < s->D || s->stride_h < 1 || s->stride_b < 1) return RAPID3_ERR_INVALID_ARG;
    if ((s->stride_n % 8) || (s->stride_h % 8) || (s->stride_b % 8)) return RAPID3_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(q) % 16) || (reinterpret_cast<uintptr_t>(k) % 16)) return RAPID3_ERR_INVALID_ARG;
    if (n_img < 1 || n_img > s->B_max) return RAPID3_ERR_INVALID_ARG;

    TensorGeom g;
    g.H = s->H;
    g.D = s->D;
    g.N = (int)N;
    g.nb = (int)((N + 63) / 64);
    g.n_text_blocks = (s->n_text + 63) / 64;
    g.h0 = 0;
    g.pair_stride = 1;
    g.stride_b = s->stride_b;
    g.stride_h = s->stride_h;
    g.stride_n = s->stride_n;
    // block means of Q and K for the listed images must fit the fixed array
    const long long need = 2ll * n_img * g.H * g.nb * g.D;
    if (need > RAPID3_STATIC_SCRATCH_DOUBLES) return RAPID3_ERR_WORKSPACE;

    ImgList l;
    l.n = n_img;
    for (int p = 0; p < n_img; ++p) {
        const int b = img_idx_host ? img_idx_host[p] : p;
        if (b < 0 || b >= s->B_max) return RAPID3_ERR_INVALID_ARG;
        l.batch[p] = b;
        l.slot[p] = p;
        l.k_free[p] = 0;
    }
    double* scratch = nullptr;
    const int r = static_scratch(&scratch);
    if (r != RAPID3_OK) return r;
    if (scoring_static_init() != cudaSuccess) {
        cudaGetLastError();
        return RAPID3_ERR_CUDA;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // every element of the used part of the scratch is written by the pooling kernel before the
    // scoring kernel reads it, so nothing has to be cleared between calls
    if (launch_block_pool(q, k, g, l, scratch, st) != cudaSuccess) return RAPID3_ERR_CUDA;
    if (launch_block_scores(scratch, g, n_img, scores, st) != cudaSuccess) return RAPID3_ERR_CUDA;
    return RAPID3_OK;
}

extern "C" int64_t rapid3_static_scratch_bytes(void) { return RAPID3_STATIC_SCRATCH_DOUBLES * (int64_t)sizeof(double); }
