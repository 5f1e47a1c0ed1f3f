// K2: per (image, head, query-block row) forced + top-k block selection.
// One warp per row, the row's scores in registers as order-preserving 32-bit keys (IPL of them a lane, key block
// 32 x + lane in register x).  The k-th largest free candidate is found by a radix search over the key bits, two at a
// time from the highest bit in which two candidates differ: the candidates at or above each of the three trial
// prefixes are counted in ten-bit fields of one word (there are at most 1023), which one warp-wide addition combines.
// The search ends early when exactly k candidates are at or above the prefix.  A free candidate is kept when its key is
// above that threshold, or equal to it and among the first (lowest block index) of the equal ones still needed -- the
// order "score descending, index ascending".  The bitmask is assembled with warp ballots and the ascending kept list
// with ballot prefix counts, so the row is written in one pass.
// Bound by the latency of that chain: a warp has a row to itself and every row's warp is resident.  Keys in shared
// memory and histograms of eight bits a round, which this replaces, took 7.3 us for two images of 24 heads x 70 rows
// (now 4.8), 9.5 us for three of 72 (6.4) and 17.7 us for one of 264 (13.6).
#include "scoring.cuh"

using namespace scoring;

namespace {

constexpr int WARPS = 4;

// HK = NoHeadKeep: one keep count per image.  HK = HeadKeep: one per (image, head), passed by value.
// HK = RowKeep: one per row, read from device memory.
// ORDER: the quads' classes in the attention's order come out too (see QuadOrder); imgs.slot then holds an image's place among the
// sparse ones in the attention's list.
template <typename HK, int IPL, bool ORDER>
__global__ void __launch_bounds__(WARPS * 32) select_kernel(const float* scores, TensorGeom g,
                                                            ImgList imgs, uint32_t* __restrict__ bitmask32,
                                                            int32_t* __restrict__ kept_idx,
                                                            int32_t* __restrict__ kept_cnt, int words32,
                                                            const DevPlan* plan, const QuadOrder order, const HK hk) {
    __shared__ uint32_t kept[ORDER ? WARPS : 1][ORDER ? IPL : 1];        // the thread block's rows: the four query blocks of a quad
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int nb = g.nb;
    const int ph = blockIdx.y, p = ph / g.H;            // p * H + h
    const int i = quad_block(g, blockIdx.x, warp);
    const int row = ph * nb + i;                        // at most 65535 x 1024
    grid_dependency_wait();                             // the scores come from the kernel before, which may still be running
    grid_dependency_launch();
    if (plan && p >= __ldcg(&plan->sparse.n)) return;
    if (i < nb) {
        // free candidates kept in this row: one count per image, or per (image, head) when the policy
        // sets a ratio for every head
        int k;
        if constexpr (HK::mode == 1) k = hk.k[ph];
        else if constexpr (HK::mode == 2) k = __ldcg(hk.k + row);
        else k = plan ? __ldcg(&plan->sparse.k_free[p]) : imgs.k_free[p];
        const float* src = scores + (long long)row * nb;
        select_row<IPL>([&](int j) { return __ldcg(src + j); },          // past the L1: see the wait above
                        i, nb, g.n_text_blocks, k, lane, bitmask32 + (long long)row * words32, words32, kept_idx + (long long)row * nb,
                        kept_cnt + row, [&](int x, uint32_t bits) { if constexpr (ORDER) kept[warp][x] = bits; });
    } else if (ORDER && lane < IPL) {
        kept[ORDER ? warp : 0][ORDER ? lane : 0] = 0u;
    }
    if constexpr (ORDER) {
        __syncthreads();
        if (warp > 0) return;
        const int n_sparse = plan ? __ldcg(&plan->sparse.n) : imgs.n, place = plan ? plan_place(plan, p, lane) : imgs.slot[p];
        uint32_t m[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) m[a] = 32 * lane < nb ? kept[a][lane] : 0u;
        order_quad(order, g, plan ? __ldcg(&plan->n_dense) : order.n_dense, n_sparse, place, ph % g.H, blockIdx.x, m, lane);
    }
}

constexpr int MASS_WARPS = 2;

template <int IPL>
__global__ void __launch_bounds__(MASS_WARPS * 32) mass_count_kernel(const float* scores, TensorGeom g, MassShare share,
                                                                     float scale, int32_t* __restrict__ row_keep) {
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int nb = g.nb;
    const int ph = blockIdx.y, p = ph / g.H, i = blockIdx.x * MASS_WARPS + warp;
    const int row = ph * nb + i;
    grid_dependency_wait();                                // for the scores
    grid_dependency_launch();
    if (i >= nb) return;
    const float* src = scores + (long long)row * nb;
    const int k = mass_row<IPL>([&](int j) { return __ldcg(src + j); }, i, nb, g.n_text_blocks, share.tau[p], scale, lane);
    if (lane == 0) row_keep[row] = k;
}

template <typename HK>
cudaError_t launch_select(const float* scores, const TensorGeom& g, const ImgList& imgs, uint64_t* bitmask, int32_t* kept_idx,
                          int32_t* kept_cnt, cudaStream_t s, const DevPlan* plan, int n_img, const QuadOrder& order, const HK& hk) {
    const dim3 grid((g.nb + WARPS - 1) / WARPS, n_img * g.H);
    return with_ipl(g.nb, [&](auto ipl) {
        return launch_kernel(order.cls ? select_kernel<HK, decltype(ipl)::value, true> : select_kernel<HK, decltype(ipl)::value, false>, grid, dim3(WARPS * 32), 0, s, scores, g, imgs,
                             reinterpret_cast<uint32_t*>(bitmask), kept_idx, kept_cnt, 2 * ((g.nb + 63) / 64), plan, order, hk);
    });
}

}  // namespace

cudaError_t launch_select_mask_mass(const float* scores, const TensorGeom& g, const ImgList& imgs,
                                    const MassShare& share, float scale, int32_t* row_keep, uint64_t* bitmask,
                                    int32_t* kept_idx, int32_t* kept_cnt, cudaStream_t s, const QuadOrder& order) {
    const cudaError_t e = with_ipl(g.nb, [&](auto ipl) {
        return launch_kernel(mass_count_kernel<decltype(ipl)::value>, dim3((g.nb + MASS_WARPS - 1) / MASS_WARPS, imgs.n * g.H),
                             dim3(MASS_WARPS * 32), 0, s, scores, g, share, scale, row_keep);
    });
    if (e != cudaSuccess) return e;
    RowKeep rk;
    rk.k = row_keep;
    return launch_select(scores, g, imgs, bitmask, kept_idx, kept_cnt, s, nullptr, imgs.n, order, rk);
}

cudaError_t launch_select_mask(const float* scores, const TensorGeom& g, const ImgList& imgs, uint64_t* bitmask,
                               int32_t* kept_idx, int32_t* kept_cnt, cudaStream_t s, const DevPlan* plan, int n_cap,
                               const QuadOrder& order) {
    return launch_select(scores, g, imgs, bitmask, kept_idx, kept_cnt, s, plan, plan ? n_cap : imgs.n, order, NoHeadKeep());
}

cudaError_t launch_select_mask_heads(const float* scores, const TensorGeom& g, const ImgList& imgs, const HeadKeep& hk,
                                     uint64_t* bitmask, int32_t* kept_idx, int32_t* kept_cnt, cudaStream_t s, const QuadOrder& order) {
    return launch_select(scores, g, imgs, bitmask, kept_idx, kept_cnt, s, nullptr, imgs.n, order, hk);
}


// ---------------------------------------------------------------------------------------------
// Plan of a gated step from device-resident policy actions: the gate and compaction the host
// entry point does on the CPU, for callers whose sampled actions never leave the GPU.
namespace {

// A thread an image: it counts the images in front of its own in both lists.  Bound by the round trip of the loads.
__global__ void __launch_bounds__(RAPID3_MAX_IMG) plan_kernel(const int32_t* action, const float* ratio, int B, int n_free_img,
                                                              DevPlan* __restrict__ plan, int* __restrict__ status) {
    __shared__ float of[RAPID3_MAX_IMG];              // an attending image's ratio, 0 for the others
    const int b = threadIdx.x;
    grid_dependency_wait();                           // first kernel of a call
    grid_dependency_launch();
    float r = 0.f;
    if (b < B) {
        const int a = __ldcg(action + b);
        const float want = __ldcg(ratio + b);
        const bool known = a == RAPID3_ACT_SKIP || a == RAPID3_ACT_REUSE || a == RAPID3_ACT_ATTEND;
        const bool valid = want > 0.f && want <= 1.f;
        // an unknown action is treated as a skip, an image with a ratio outside (0, 1] is not processed
        if (!known || (a == RAPID3_ACT_ATTEND && !valid)) atomicExch(status, RAPID3_ERR_INVALID_ARG);
        if (a == RAPID3_ACT_ATTEND && valid) r = want;
    }
    of[b] = r;
    __syncthreads();
    int n_all = 0, n_sparse = 0, pos = 0, slot = 0;   // sparse images in batch order; all by descending ratio, equal ones in batch order
    for (int o = 0; o < B; ++o) {
        const float x = of[o];
        const bool sparse = x > 0.f && x < 1.f;
        n_all += x > 0.f;
        n_sparse += sparse;
        slot += sparse && o < b;
        pos += x > r || (x == r && o < b);
    }
    if (r > 0.f) {
        if (r < 1.f) {
            const double x = ceil((double)r * (double)n_free_img - 1e-6);
            plan->sparse.batch[slot] = b;
            plan->sparse.slot[slot] = slot;
            plan->sparse.k_free[slot] = (int)(x < 0.0 ? 0.0 : (x > (double)n_free_img ? (double)n_free_img : x));
        }
        plan->all.batch[pos] = b;
        plan->all.slot[pos] = r < 1.f ? slot : -1;
    }
    if (b == 0) {
        plan->sparse.n = n_sparse;
        plan->all.n = n_all;
        plan->n_dense = n_all - n_sparse;
    }
}

}  // namespace

cudaError_t launch_plan(const int32_t* action_dev, const float* ratio_dev, int B, const TensorGeom& g, DevPlan* plan,
                        int* status, cudaStream_t s) {
    const int n_free_img = g.nb - g.n_text_blocks - 1;
    return launch_kernel(plan_kernel, dim3(1), dim3(RAPID3_MAX_IMG), 0, s, action_dev, ratio_dev, B, n_free_img > 0 ? n_free_img : 0,
                         plan, status);
}
