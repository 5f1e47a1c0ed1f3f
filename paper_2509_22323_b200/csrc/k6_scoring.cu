// K6: the whole scoring pass of an (image, head) pair by one cluster of thread blocks: block means of Q and K, scores, selection.
//
// Three kernels one after the other (k1, k2) each spread over the GPU, wait for one another's last thread block and keep every
// SM from the attention, of which much needs no mask: quads of dense images and of text rows.  Here a pair belongs to a
// cluster of 1 to 6 thread blocks, which meet once, between the means and the scores; the attention kernel starts beside
// them (programmatic dependent launch) on the SMs that they leave free and works on what needs no mask until they are through.
// The cluster size is the launch's choice (scoring_cluster below): few SMs where there is other work for the rest, all of
// them where there is not.
//   means   a warp per 64-token block, as pool_kernel; they go to the workspace, where the cluster's blocks find them in the L2
//   scores  a thread block owns whole quads of query blocks; their means and those of K, 48 key blocks at a time through two
//           buffers, come to shared memory by asynchronous copies; fp64 mma.sync as in scores_kernel, in the same order
//   select  a warp per row, from shared memory
// Bound by the loads of Q and K (24 warps with eight 16-byte loads a lane in flight) and behind them by the chain of the
// three steps.
#include <algorithm>

#include "ptx.cuh"
#include "scoring.cuh"

using namespace scoring;

namespace {

constexpr int WARPS = 24, KSTAGES = 2, KCOLS = 48;
constexpr int SMEM_MAX = 225 * 1024;
constexpr int SCORING_FROM = 222;

// Which rule gives a row's count: one per image, one per (image, head), the cumulative mass.
struct MassRule {
    static constexpr int mode = 3;
    MassShare share;
    float scale;
};
struct ScoreArgs {
    const uint16_t* q;
    const uint16_t* k;
    TensorGeom g;
    ImgList imgs;                  // sparse images; slot: place among them in the attention's list
    double* pooled;                // [2][imgs.n][H][nb][D]
    float* scores;
    uint32_t* bitmask32;
    int32_t* kept_idx;
    int32_t* kept_cnt;
    int words32;
    QuadOrder order;
    int cluster;                   // thread blocks of a cluster
    int rows;                      // of S that are in shared memory at a time
    bool pool;                     // false: the means are there
    int n_cap;                     // images that the means have room for
    const DevPlan* plan;           // rows_kernel: the images from device memory
};

template <int D, int IPL>
constexpr int row_bytes() { return (D + 4) * 8 + (32 * IPL + 4) * 4 + IPL * 4; }
template <int D>
constexpr int ring_bytes() { return KSTAGES * KCOLS * (D + 4) * 8; }

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int D, int IPL, typename HK>
__global__ void __launch_bounds__(WARPS * 32, 1) scoring_kernel(const __grid_constant__ ScoreArgs a, const __grid_constant__ HK hk) {
    constexpr int LDS = D + 4, LDN = 32 * IPL + 4;
    extern __shared__ __align__(16) double smem[];
    const int rows = a.rows;
    double* sq = smem;                                   // [rows][LDS]
    double* sk = sq + rows * LDS;                        // [KSTAGES][KCOLS][LDS]
    float* ss = reinterpret_cast<float*>(sk + KSTAGES * KCOLS * LDS);    // [rows][LDN]
    uint32_t* kept = reinterpret_cast<uint32_t*>(ss + rows * LDN);       // [rows][IPL]
    const TensorGeom& g = a.g;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int nb = g.nb, nq = (nb + 3) >> 2, H = g.H;
    grid_dependency_wait();
    grid_dependency_launch();
    const int rank = a.cluster > 1 ? (int)cluster_rank() : 0;
    const int quads = (nq + a.cluster - 1) / a.cluster, q_first = rank * quads, q_end = min(nq, q_first + quads);   // this thread block's
    // row r of a panel that begins at quad q0 is this query block
    auto row_block = [&](int q0, int r) { return q0 + (r >> 2) < q_end ? quad_block(g, q0 + (r >> 2), r & 3) : nb; };

    const int ph = blockIdx.x / a.cluster;             // the grid is a cluster for each (image, head)
    const int p = ph / H, h = ph - p * H;
    const double* mean_q = a.pooled + (long long)ph * nb * D;
    const double* mean_k = a.pooled + ((long long)a.imgs.n * H + ph) * nb * D;
    if (a.pool) {
        const int batch = a.imgs.batch[p];
        const long long at = (long long)batch * g.stride_b + (long long)(g.h0 + h) * g.stride_h;
        for (int u = rank * WARPS + warp; u < 2 * nb; u += a.cluster * WARPS) {
            const int which = u >= nb, blk = u - which * nb;
            pool_block<D>((which ? a.k : a.q) + at + (long long)(64 * blk) * g.stride_n, g.stride_n, min(64, g.N - 64 * blk),
                          const_cast<double*>(which ? mean_k : mean_q) + (long long)blk * D, lane, [] {});
        }
        if (a.cluster > 1) cluster_sync();
        else __syncthreads();
    }
    for (int q0 = q_first; q0 < q_end; q0 += rows >> 2) {
        auto load_k = [&](int ch) {                  // one group of copies, empty past the end
            if (KCOLS * ch < nb) {
                double* dst = sk + (ch % KSTAGES) * (KCOLS * LDS);
                for (int e = threadIdx.x; e < KCOLS * (D / 2); e += WARPS * 32) {
                    const int r = e / (D / 2), c = 2 * (e % (D / 2)), j = KCOLS * ch + r;
                    copy16_async(dst + r * LDS + c, j < nb ? mean_k + (long long)j * D + c : a.pooled, j < nb);
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        for (int e = threadIdx.x; e < rows * (D / 2); e += WARPS * 32) {
            const int r = e / (D / 2), c = 2 * (e % (D / 2)), i = row_block(q0, r);
            copy16_async(sq + r * LDS + c, i < nb ? mean_q + (long long)i * D + c : a.pooled, i < nb);
        }
#pragma unroll
        for (int ch = 0; ch < KSTAGES; ++ch) load_k(ch);
        const int gr = lane >> 2, c4 = lane & 3;
        for (int ch = 0; KCOLS * ch < nb; ++ch) {
            asm volatile("cp.async.wait_group %0;" ::"n"(KSTAGES - 1) : "memory");
            __syncthreads();
            // two fragments of 8 x 8 side by side a warp
            const int pairs = (min(nb - KCOLS * ch, KCOLS) + 15) >> 4;
            for (int f = warp; f < (rows >> 3) * pairs; f += WARPS) {
                const int ri = (f / pairs) * 8, cj = (f % pairs) * 16;
                const double* aq = sq + (ri + gr) * LDS + c4;
                const double* bk = sk + (ch % KSTAGES) * (KCOLS * LDS) + (cj + gr) * LDS + c4;
                double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll 8
                for (int d = 0; d < D; d += 4) {
                    const double x = aq[d];
                    dmma_8x8x4(acc[0][0], acc[0][1], x, bk[d]);
                    dmma_8x8x4(acc[1][0], acc[1][1], x, bk[8 * LDS + d]);
                }
                float* o = ss + (ri + gr) * LDN + KCOLS * ch + cj + 2 * c4;
                *reinterpret_cast<float2*>(o) = make_float2((float)acc[0][0], (float)acc[0][1]);
                *reinterpret_cast<float2*>(o + 8) = make_float2((float)acc[1][0], (float)acc[1][1]);
            }
            __syncthreads();
            load_k(ch + KSTAGES);
        }
        for (int r = warp; r < rows; r += WARPS) {
            const int i = row_block(q0, r);
            const float* src = ss + r * LDN;
            const long long row = (long long)ph * nb + i;
            if (i < nb) {
                for (int j = lane; j < nb; j += 32) a.scores[row * nb + j] = src[j];
                auto score = [&](int j) { return src[j]; };
                int k;
                if constexpr (HK::mode == MassRule::mode) k = mass_row<IPL>(score, i, nb, g.n_text_blocks, hk.share.tau[p], hk.scale, lane);
                else if constexpr (HK::mode == HeadKeep::mode) k = hk.k[ph];
                else k = a.imgs.k_free[p];
                select_row<IPL>(score, i, nb, g.n_text_blocks, k, lane, a.bitmask32 + row * a.words32, a.words32, a.kept_idx + row * nb,
                                a.kept_cnt + row, [&](int x, uint32_t bits) { kept[r * IPL + x] = bits; });
            } else if (lane < IPL) {
                kept[r * IPL + lane] = 0u;
            }
        }
        __syncthreads();
        if (a.order.cls) {
            for (int x = warp; x < rows >> 2 && q0 + x < q_end; x += WARPS) {
                uint32_t m[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) m[b] = 32 * lane < nb ? kept[(4 * x + b) * IPL + lane] : 0u;
                order_quad(a.order, g, a.order.n_dense, a.imgs.n, a.imgs.slot[p], h, q0 + x, m, lane);
            }
            __syncthreads();
        }
    }
}

// Scores and selection from means that are there, for launches of few quads, where a kernel of its own for each is mostly a launch and a round
// trip: a thread block has the rows of two quads of a pair, all key blocks.  The rows' means come to shared memory; those of K go straight
// from the L2 to the fragments of the one warp that needs them (a warp has eight key blocks; the four lanes of a row take 32 bytes), all loads
// of a fragment at once.  The products run in the order of scores_kernel, the rows of S stay in shared memory for the selection, a row a warp.
// Bound by that chain (10 us of 20 to 30 before, by pooling, scores and selection): whole steps, us, scores and selection apart / in one: 90
// quads by cumulative mass 28.5 / 25.9, 96 of 9 blocks 25.1 / 23.1, 160 of 19 36.4 / 34.2, 192 of 21 at D = 128 48.9 / 46.0; 26 drawn at random
// of 75 to 148 quads 4.0 % faster in the mean, 26 of 149 to 221 3.0 %.
constexpr int ROWS = 8;
template <int D, int IPL, int ROW_WARPS, typename HK>
__global__ void __launch_bounds__(ROW_WARPS * 32) rows_kernel(const __grid_constant__ ScoreArgs a, const __grid_constant__ HK hk) {
    constexpr int LDS = D + 4, LDN = 32 * IPL + 4;
    __shared__ __align__(16) double sq[ROWS * LDS];
    __shared__ __align__(8) float ss[ROWS * LDN];        // stored two at a time
    static_assert(LDN % 2 == 0, "a row's pairs lie on 8 bytes");
    __shared__ uint32_t kept[ROWS][IPL];
    const TensorGeom& g = a.g;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int nb = g.nb, nq = (nb + 3) >> 2, H = g.H, q0 = blockIdx.x * (ROWS / 4);
    const int ph = blockIdx.y, p = ph / H;
    grid_dependency_wait();
    grid_dependency_launch();
    if (a.plan && p >= __ldcg(&a.plan->sparse.n)) return;
    auto row_block = [&](int r) { return q0 + (r >> 2) < nq ? quad_block(g, q0 + (r >> 2), r & 3) : nb; };
    const double* mean_q = a.pooled + (long long)ph * nb * D;
    const double* mean_k = a.pooled + ((long long)a.n_cap * H + ph) * nb * D;
#pragma unroll
    for (int e = threadIdx.x; e < ROWS * (D / 2); e += ROW_WARPS * 32) {
        const int r = e / (D / 2), c = 2 * (e % (D / 2)), i = row_block(r);
        copy16_async(reinterpret_cast<double*>(sq) + r * LDS + c, i < nb ? mean_q + (long long)i * D + c : a.pooled, i < nb);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int gr = lane >> 2, c4 = lane & 3;
    const double* aq = sq + gr * LDS + c4;
    bool there = false;                                  // the rows' means
    for (int cj = 8 * warp; cj < nb; cj += 8 * ROW_WARPS) {
        const double* bk = mean_k + (long long)min(cj + gr, nb - 1) * D + c4;      // key blocks past the end: any, nothing reads their scores
        double acc[2] = {0.0, 0.0};
        double b[D / 4];
#pragma unroll
        for (int x = 0; x < D / 4; ++x) b[x] = __ldcg(bk + 4 * x);
        if (!there) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            ptx::bar_sync(1, ROW_WARPS * 32);
            there = true;
        }
#pragma unroll
        for (int x = 0; x < D / 4; ++x) dmma_8x8x4(acc[0], acc[1], aq[4 * x], b[x]);
        *reinterpret_cast<float2*>(ss + gr * LDN + cj + 2 * c4) = make_float2((float)acc[0], (float)acc[1]);
    }
    if (!there) {                                        // a warp without key blocks
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        ptx::bar_sync(1, ROW_WARPS * 32);
    }
    __syncthreads();
    if (warp < ROWS) {
        const int r = warp, i = row_block(r);
        const float* src = ss + r * LDN;
        const long long row = (long long)ph * nb + i;
        if (i < nb) {
            for (int j = lane; j < nb; j += 32) a.scores[row * nb + j] = src[j];
            auto score = [&](int j) { return src[j]; };
            int k;
            if constexpr (HK::mode == MassRule::mode) k = mass_row<IPL>(score, i, nb, g.n_text_blocks, hk.share.tau[p], hk.scale, lane);
            else if constexpr (HK::mode == HeadKeep::mode) k = hk.k[ph];
            else k = a.plan ? __ldcg(&a.plan->sparse.k_free[p]) : a.imgs.k_free[p];
            select_row<IPL>(score, i, nb, g.n_text_blocks, k, lane, a.bitmask32 + row * a.words32, a.words32, a.kept_idx + row * nb,
                            a.kept_cnt + row, [&](int x, uint32_t bits) { kept[r][x] = bits; });
        } else if (lane < IPL) {
            kept[r][lane] = 0u;
        }
    }
    if (!a.order.cls) return;
    __syncthreads();
    if (warp < ROWS / 4 && q0 + warp < nq) {
        uint32_t m[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) m[b] = 32 * lane < nb ? kept[4 * warp + b][lane] : 0u;
        const int n_sparse = a.plan ? __ldcg(&a.plan->sparse.n) : a.imgs.n, place = a.plan ? plan_place(a.plan, p, lane) : a.imgs.slot[p];
        order_quad(a.order, g, a.plan ? __ldcg(&a.plan->n_dense) : a.order.n_dense, n_sparse, place, ph % H, q0 + warp, m, lane);
    }
}

template <typename HK>
cudaError_t launch_rows_of(const ScoreArgs& a, const HK& hk, cudaStream_t s) {
    const dim3 grid(((a.g.nb + 3) / 4 + ROWS / 4 - 1) / (ROWS / 4), a.n_cap * a.g.H);
    const auto go = [&](auto kernel, int warps) { return launch_kernel(kernel, grid, dim3(warps * 32), 0, s, a, hk); };
    if (a.g.nb <= 64) return go(a.g.D == 128 ? rows_kernel<128, 2, 8, HK> : rows_kernel<64, 2, 8, HK>, 8);
    if (a.g.nb <= 96) return go(a.g.D == 128 ? rows_kernel<128, 3, 12, HK> : rows_kernel<64, 3, 12, HK>, 12);
    return go(a.g.D == 128 ? rows_kernel<128, 4, 16, HK> : rows_kernel<64, 4, 16, HK>, 16);
}

template <int D, typename HK, typename F>
cudaError_t with_kernel(int nb, F&& f) {
    if (nb <= 96) return f(scoring_kernel<D, 3, HK>, row_bytes<D, 3>(), ring_bytes<D>());
    return f(scoring_kernel<D, 6, HK>, row_bytes<D, 6>(), ring_bytes<D>());
}

template <typename HK>
cudaError_t launch(ScoreArgs& a, const HK& hk, int pairs, cudaStream_t s) {
    auto go = [&](auto kernel, int row, int ring) {
        const int nq = (a.g.nb + 3) / 4, own = 4 * ((nq + a.cluster - 1) / a.cluster);
        a.rows = std::min((own + 7) / 8 * 8, (SMEM_MAX - ring) / row / 8 * 8);
        const int smem = ring + a.rows * row;
        return launch_kernel_cluster(kernel, dim3(pairs * a.cluster), dim3(WARPS * 32), smem, s, a.cluster, a, hk);
    };
    return a.g.D == 128 ? with_kernel<128, HK>(a.g.nb, go) : with_kernel<64, HK>(a.g.nb, go);
}

}  // namespace

cudaError_t scoring_cluster_static_init() {
    cudaError_t e = cudaSuccess;
    const auto set = [&](auto kernel, int, int) {
        return e = e != cudaSuccess ? e : cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
    };
    for (int nb : {96, 192}) {
        with_kernel<128, NoHeadKeep>(nb, set);
        with_kernel<128, HeadKeep>(nb, set);
        with_kernel<128, MassRule>(nb, set);
        with_kernel<64, NoHeadKeep>(nb, set);
        with_kernel<64, HeadKeep>(nb, set);
        with_kernel<64, MassRule>(nb, set);
    }
    return e;
}

// Thread blocks of a cluster for that many (image, head) pairs, or 0 for the three kernels, which spread over the GPU what a few
// pairs cannot.  The least SM time decides: what the pass takes of its own SMs, and what the others wait for it after the attention
// that needs no mask (heavy_us of SM time).  The times in us: a thread block alone 21 for a MB of Q and K, the scores at half
// of the fp64 tensor rate, 3.3 or 5 for every 24 rows (5 more by cumulative mass); the three kernels 7 (one more by mass 2.5) and
// 4.5 TB/s.  One thread block a pair, the longest of all, only beside much other work, and only so a second wave of them; of clusters
// (45 of three fit at a time) no second wave; rows of more than 192 blocks gain nothing (24 pairs of 264: 1114 us a step, this way 1109 to 1140).  Launches of
// fewer quads than SCORING_FROM wait for the first masks, not for SMs (96 quads of 15 blocks 23.7 / 28.0, 192 of 29 35.3 / 37.1).
// Steps, us, three kernels / clusters: two images of 24 heads, 1357 tokens, D = 64 43.4 / 41.5 (of two); 864 quads with per-head
// ratios 189.3 / 184.9 (two), by mass 343 / 337 (two), a dense and a sparse image at D = 64 258.7 / 254.2 (one); one image from
// raw projections 202.3 / 195.5 (two to four).
// Beside few pairs and no dense image only text rows need no mask.  Worked on early they shorten a launch whose last round of SMs is
// nearly full; in any other that round has room for them, and the clusters only keep the first masks back: one image by top-k,
// ratio 0.25, 16 heads x 57 blocks (240 quads, 1.62 rounds) 67.1 / 76.8, 24 x 57 (2.43) 95.8 / 101.6, 24 x 108 (4.38) 270 / 288,
// D = 64 24 x 106 168 / 174; but 24 x 72 (2.92) 147.5 / 131.0, 16 x 72 (1.95) 98.3 / 91.8, D = 64 24 x 72 97.3 / 91.4.
constexpr int FEW_PAIRS = 24;
constexpr int FULL_ROUND = 104;    // quads
int scoring_cluster(const TensorGeom& g, int images, int pairs, bool pool, bool mass, double heavy_us) {
    const int nq = (g.nb + 3) / 4;
    const int quads = images * g.H * nq;
    if (g.nb > 192 || pairs < 16 || quads < SCORING_FROM) return 0;
    if (!mass && pairs <= FEW_PAIRS && images * g.H == pairs && (quads - 1) % SM_COUNT + 1 < FULL_ROUND) return 0;
    const double mb = pool ? 256e-6 * g.nb * g.D : 0.0;                  // of Q and K, a pair
    int best = 0;
    double least = 0.95 * SM_COUNT * (7.0 + pairs * (mb / 4.5 + 1.5e-5 * g.nb * g.nb) + (mass ? 2.5 + 2e-5 * pairs * g.nb * g.nb : 0.0));
    for (int c = 1; c <= 6 && c <= nq && (c == 1 || pairs * c <= 100); ++c) {
        const int own = 4 * ((nq + c - 1) / c);
        const double us = 3.0 + (c > 1 ? 1.5 : 0.0) + 21.0 * mb / c + own * g.nb * g.D / (32 * 1900.0) +
                          (own + WARPS - 1) / WARPS * ((g.nb <= 96 ? 3.3 : 5.0) + (mass ? 5.0 : 0.0));
        const int sms = std::min(pairs * c, SM_COUNT);
        if (c == 1 && heavy_us < 2.5 * SM_COUNT * us) continue;
        const double cost = (us * sms + std::max(0.0, us * (SM_COUNT - sms) - heavy_us)) * ((pairs * c + SM_COUNT - 1) / SM_COUNT);
        if (cost < least) {
            best = c;
            least = cost;
        }
    }
    return best;
}

static ScoreArgs score_args(const void* q, const void* k, const TensorGeom& g, const ImgList& imgs, double* pooled, float* scores, uint64_t* bitmask,
                            int32_t* kept_idx, int32_t* kept_cnt, const QuadOrder& order) {
    ScoreArgs a;
    a.q = static_cast<const uint16_t*>(q);
    a.k = static_cast<const uint16_t*>(k);
    a.g = g;
    a.imgs = imgs;
    a.pooled = pooled;
    a.scores = scores;
    a.bitmask32 = reinterpret_cast<uint32_t*>(bitmask);
    a.kept_idx = kept_idx;
    a.kept_cnt = kept_cnt;
    a.words32 = 2 * ((g.nb + 63) / 64);
    a.order = order;
    a.cluster = a.rows = 0;
    a.pool = false;
    a.n_cap = imgs.n;
    a.plan = nullptr;
    return a;
}

// Calls f with what says how a row's count is found.
template <typename F>
static cudaError_t with_rule(const HeadKeep* heads, const MassShare* share, float mass_scale, F&& f) {
    if (share) {
        MassRule m;
        m.share = *share;
        m.scale = mass_scale;
        return f(m);
    }
    return heads ? f(*heads) : f(NoHeadKeep());
}

cudaError_t launch_scoring(const void* q, const void* k, const TensorGeom& g, const ImgList& imgs, double* pooled, float* scores,
                           uint64_t* bitmask, int32_t* kept_idx, int32_t* kept_cnt, int cluster, bool pool, const HeadKeep* heads,
                           const MassShare* share, float mass_scale, cudaStream_t s, const QuadOrder& order) {
    ScoreArgs a = score_args(q, k, g, imgs, pooled, scores, bitmask, kept_idx, kept_cnt, order);
    a.cluster = cluster;
    a.pool = pool;
    return with_rule(heads, share, mass_scale, [&](const auto& rule) { return launch(a, rule, imgs.n * g.H, s); });
}

cudaError_t launch_rows(const TensorGeom& g, const ImgList& imgs, double* pooled, float* scores, uint64_t* bitmask, int32_t* kept_idx,
                        int32_t* kept_cnt, const HeadKeep* heads, const MassShare* share, float mass_scale, cudaStream_t s,
                        const QuadOrder& order, const DevPlan* plan, int n_cap) {
    ScoreArgs a = score_args(nullptr, nullptr, g, imgs, pooled, scores, bitmask, kept_idx, kept_cnt, order);
    a.plan = plan;
    if (plan) a.n_cap = n_cap;
    return with_rule(heads, share, mass_scale, [&](const auto& rule) { return launch_rows_of(a, rule, s); });
}

// Up to 128 key blocks a thread block's warps have one fragment each; longer rows of few pairs lose (2 heads of 129 to 150 blocks at D = 128
// +1.7 %).  From SCORING_FROM quads on it would gain little (1.4 % where there are no clusters).  Launches of up to half as many quads as
// SMs would gain 5 %: this line is no measured one, rapid3.h promises the launches of such steps one by one (rapid3_launch_count).
bool scoring_rows(const TensorGeom& g, int images) {
    const int quads = images * g.H * ((g.nb + 3) / 4);
    return 2 * quads > SM_COUNT && quads < SCORING_FROM && g.nb <= 128;
}
