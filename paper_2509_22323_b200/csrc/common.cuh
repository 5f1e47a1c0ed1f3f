// Shared declarations of the rapid3 CUDA library: launch-argument structs and the internal
// launcher prototypes.  Host API in api.cu; kernels in k1_scores.cu to k6_scoring.cu.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "rapid3.h"

#define RAPID3_BLOCK 64
#define RAPID3_MAX_IMG 64     // images per launch (lists travel as kernel arguments)
#define RAPID3_MAX_NB 1024    // key blocks per sequence (65536 tokens)

constexpr int SM_COUNT = 148; // of a B200

// Per-launch image list.  batch[p]: index into the B dimension of Q/K/V/O.
// slot[p]: index into the compacted scores / mask / kept-list arrays, or -1 for a dense image.  In the list of sparse images that the
// selection and scoring_kernel get with a QuadOrder: the image's place among the sparse ones in the attention's list.
// k_free[p]: free candidates kept per image row (select kernel).
struct ImgList {
    int n;
    int batch[RAPID3_MAX_IMG];
    int slot[RAPID3_MAX_IMG];
    int k_free[RAPID3_MAX_IMG];
};

// Device-resident plan of one gated step (filled by plan_kernel from device-resident actions):
// the two image lists the host path passes as kernel arguments.
struct DevPlan {
    ImgList sparse;   // images with keep ratio < 1, ascending batch order, slot = position
    ImgList all;      // every attending image, descending keep ratio (dense first)
    int n_dense;
};

// Keep counts per (sparse slot, head) for a policy that sets one ratio per head (Sec. 3.2: the
// sparsity head emits theta in R^{L x H}).  Travels as a kernel argument, so slots * H is bounded.
#define RAPID3_MAX_HEAD_ROWS 2048
struct HeadKeep {
    static constexpr int mode = 1;
    int k[RAPID3_MAX_HEAD_ROWS];
};
struct NoHeadKeep {
    static constexpr int mode = 0;
};
// Keep counts per row (image slot, head, query block) in device memory: the cumulative-mass rule
// arrives at a different count in every row.
struct RowKeep {
    static constexpr int mode = 2;
    const int32_t* k;
};
// Mass share tau per image of a launch (cumulative-mass selection).
struct MassShare {
    float tau[RAPID3_MAX_IMG];
};

struct TensorGeom {
    int H, D, N, nb, n_text_blocks;           // H: heads this launch covers
    int h0;                                   // first of them in the tensors (workspace arrays count heads from 0)
    int pair_stride;                          // 1, 2 or 3: which query blocks share an attention tile
    long long stride_b, stride_h, stride_n;   // elements
};

// Into how many parts the attention cuts the list of a quad of query blocks: of a dense image, of a sparse image's quads with
// text rows, of its other quads; and where the parts leave their results.
struct AttnParts {
    int dense = 1, text = 1, light = 1;
    bool keys = false;               // lists are whole; every tile has an SM to itself, whose two tiles take its key blocks by turns
    float4* partial = nullptr;       // attention_partial_bytes()
    int* given_up = nullptr;         // a wait of the launch has run out: its parts are not complete, and add_parts_kernel stores nothing
    __host__ __device__ bool any() const { return dense > 1 || text > 1 || light > 1; }
};
// Units of work of an attention launch over n_img images, n_dense of them dense.
__host__ __device__ inline int attention_units(const TensorGeom& g, const AttnParts& parts, int n_img, int n_dense) {
    const int nq = (g.nb + 3) / 4, t = (g.n_text_blocks + 3) / 4, ntq = t < nq ? t : nq;
    return g.H * (n_dense * nq * parts.dense + (n_img - n_dense) * (ntq * parts.text + (nq - ntq) * parts.light));
}

// Which two of the quad's four query blocks form a 128-row tile: neighbours, or, when a row of the image
// grid spans two blocks (pair_stride 2), vertical neighbours (i, i + 2), whose kept lists overlap far more
// (measured on the 128 x 128 grid at keep ratio 0.25: 90 % against 63 % of the tile's MMA work lands on
// kept 64 x 64 sub-tiles).  pair_stride 3 goes further on that grid: the whole quad is one column of it --
// members (i, i + 2, i + 4, i + 6), the left or the right halves of four consecutive grid rows -- so both
// tiles want nearly the same key blocks (union of the quad 98 instead of 134 blocks at keep ratio 0.25,
// both tiles busy on 68 % of them instead of 23 %).
__host__ __device__ inline int quad_block(const TensorGeom& g, int quad, int a) {
    int q = 4 * quad + (g.pair_stride == 2 ? ((a & 1) << 1) + (a >> 1) : a);
    if (g.pair_stride == 3 && q >= g.n_text_blocks) {
        const int r = q - g.n_text_blocks, w = r & 7;
        q = g.n_text_blocks + (r & ~7) + ((w & 3) << 1) + (w >> 2);
    }
    return q;
}

// The last ORDER_LAST quads of a launch (of sparse images, without text rows) by how long they take, longest first: the selection kernel, which
// knows a quad's lists, puts it into one of ORDER_CLASSES classes of equal width, and the attention kernel hands them out
// class by class.  In the order of images and heads the last quads of a launch may be long ones, for which the other SMs
// wait; the quads before them stay in that order, in which the thread blocks at work share the K and V of a few heads.  So do those that
// an SM begins with: all of them start at once, and without the order they start 1 us sooner (40 steps of 297 to 1000 quads 0.4 %).
// One quad for nearly every SM is enough, its last: of 448, 288, 192, 160, 144, 128, 112, 96 and 64 quads 128 were the best in launches above and
// below 1000 quads (36 and 40 steps drawn at random: -1.6 and -0.6 % against 448, which loses what the quads of a head share in the L2 and is
// longer to search).  For launches of more than ORDER_FROM quads, us, in order / so, by turns: two images of 288 quads at D = 64 39.7 / 38.5,
// 864 quads with a ratio for every head 193.9 / 180.6, by cumulative mass 354.5 / 335.0, one image of 432 at 0.5 from raw projections 195.3 / 189.5, 1584
// quads of one 16896-token image 1100 / 1104 (no difference shown); steps drawn at random, in the mean and the worst that differed by more than its own
// runs: 149 to 221 quads -0.8 % and +6.6 % (18; the worst 160 quads of rows of 5 blocks), 222 to 296 -3.7 % and +0.9 % (18), more -1.3 % (24).  With a
// quad an SM nothing is handed out.
constexpr int ORDER_CLASSES = 32, ORDER_LAST = 128, ORDER_FROM = SM_COUNT;
// Of `light` quads without text rows, behind `heavy` others, how many stay where they are.
__host__ __device__ inline int order_after(int light, int heavy) {
    const int begun = heavy < SM_COUNT ? SM_COUNT - heavy : 0, first = light - ORDER_LAST;
    return begun > light ? light : first > begun ? first : begun;
}
struct QuadOrder {
    int n_dense = 0;                 // dense images of the launch, where the host knows
    uint8_t* cls = nullptr;          // [ORDER_LAST] class of the quad at that place from the first of the last on; 4-byte aligned
};

// Programmatic dependent launch: every kernel of a step is launched so that it may start while the kernel before it in the stream
// is still running, and must call grid_dependency_wait() before it touches anything that kernel writes (and read it past
// the L1, whose lines the wait is not known to refresh); the kernel before it calls grid_dependency_launch() to let it
// start.  Every kernel here waits before it lets the next one start (the attention kernel, which signals nothing, before it
// ends; a thread block without work may leave at once where another waits): when a kernel runs, all kernels but the one
// right before it have ended -- so the attention kernel's thread blocks that need nothing
// of the selection may run beside it, and find Q, K and V of whatever kernel came before the call.
#ifdef __CUDACC__
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// `carveout`: percentage of the SM's first-level memory that the launch prefers as shared memory, -1 for the default.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel_carveout(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                          int carveout, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    cfg.numAttrs = carveout >= 0 ? 2 : 1;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[1].val.sharedMemCarveout = (unsigned)carveout;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
    if (e != cudaSuccess) cudaGetLastError();     // the caller has it: the next call must not find it again
    return e;
}
// The same for a kernel of clusters of that many thread blocks.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, int cluster,
                                         Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                 Args&&... args) {
    return launch_kernel_carveout(kernel, grid, block, smem, s, -1, static_cast<Args&&>(args)...);
}
#endif

// K1: block means of Q and K (fp64) for the listed images, then S = Qbar . Kbar^T -> fp32.
// With `plan` set the image list is read from device memory (plan->sparse) and the grid is sized
// for `n_cap` images; CTAs beyond the planned count return at once.  pooled is [2][n_cap][H][nb][D].
cudaError_t launch_block_pool(const void* q, const void* k, const TensorGeom& g, const ImgList& imgs,
                              double* pooled, cudaStream_t s, const DevPlan* plan = nullptr, int n_cap = 0);
cudaError_t launch_block_scores(const double* pooled, const TensorGeom& g, int n_img, float* scores,
                                cudaStream_t s, const DevPlan* plan = nullptr);
// K2: forced + top-k selection.
cudaError_t launch_select_mask(const float* scores, const TensorGeom& g, const ImgList& imgs,
                               uint64_t* bitmask, int32_t* kept_idx, int32_t* kept_cnt, cudaStream_t s,
                               const DevPlan* plan = nullptr, int n_cap = 0, const QuadOrder& order = QuadOrder());
cudaError_t launch_select_mask_heads(const float* scores, const TensorGeom& g, const ImgList& imgs,
                                     const HeadKeep& hk, uint64_t* bitmask, int32_t* kept_idx, int32_t* kept_cnt,
                                     cudaStream_t s, const QuadOrder& order = QuadOrder());
// K2, cumulative-mass variant: row_keep[row] = smallest count of best free candidates holding a share
// tau of the row's softmax mass (weights exp(scale * (S - row max)), fp64), then the top-k selection
// at that count.
cudaError_t launch_select_mask_mass(const float* scores, const TensorGeom& g, const ImgList& imgs,
                                    const MassShare& share, float scale, int32_t* row_keep, uint64_t* bitmask,
                                    int32_t* kept_idx, int32_t* kept_cnt, cudaStream_t s, const QuadOrder& order = QuadOrder());
// K6: means (pool = true; else they are there), scores and selection in one launch of clusters of `cluster` thread blocks.  heads: a count per (image, head); share: the cumulative-mass rule; neither: imgs.k_free.
cudaError_t launch_scoring(const void* q, const void* k, const TensorGeom& g, const ImgList& imgs, double* pooled, float* scores,
                           uint64_t* bitmask, int32_t* kept_idx, int32_t* kept_cnt, int cluster, bool pool, const HeadKeep* heads,
                           const MassShare* share, float mass_scale, cudaStream_t s, const QuadOrder& order = QuadOrder());
// The cluster size for that many (image, head) pairs of a step with `images` attending, beside heavy_us of SM time of attention
// that needs no mask; 0: not this way.
int scoring_cluster(const TensorGeom& g, int images, int pairs, bool pool, bool mass, double heavy_us);
// Scores and selection in one launch, from means that are there; whether it takes the place of the two kernels in a step with `images`
// attending.
cudaError_t launch_rows(const TensorGeom& g, const ImgList& imgs, double* pooled, float* scores, uint64_t* bitmask, int32_t* kept_idx,
                        int32_t* kept_cnt, const HeadKeep* heads, const MassShare* share, float mass_scale, cudaStream_t s,
                        const QuadOrder& order = QuadOrder(), const DevPlan* plan = nullptr, int n_cap = 0);
bool scoring_rows(const TensorGeom& g, int images);
// K5: Q/K producer (RMS norm + gain + rotary embedding -> bf16) that also writes the block means of
// the images with a workspace slot.  pooled is [2][n_sparse][H][nb][D].
struct PrepArgs {
    const void* q_raw;
    const void* k_raw;
    void* q_out;
    void* k_out;
    const float* q_gain;
    const float* k_gain;
    const float* rot;     // [N][D/2][2] (cos, sin) or nullptr
    float eps;
};
cudaError_t prepare_static_init();
cudaError_t launch_prepare(const PrepArgs& a, const TensorGeom& g, const ImgList& imgs, int n_sparse, double* pooled,
                           cudaStream_t s);
// Builds the plan from device-resident actions and keep ratios (one thread block; B <= RAPID3_MAX_IMG).
cudaError_t launch_plan(const int32_t* action_dev, const float* ratio_dev, int B, const TensorGeom& g,
                        DevPlan* plan, int* status, cudaStream_t s);
// K3: attention over kept tiles.  `bitmask` (optional) is the select kernel's bitmask of the same
// lists; when present the kernel reads it instead of walking the lists.  inject_stop_group >= 0
// launches the failure-injection build of the kernel (see rapid3_debug_inject_timeout).  wait_first = false: after the selection
// kernel, for whose masks the quads of sparse images wait themselves.  With `parts` lists may be worked on in parts, in one
// launch more (added to *launches).
cudaError_t launch_attention(const CUtensorMap& tmq, const CUtensorMap& tmk, const CUtensorMap& tmv,
                             void* out, const TensorGeom& g, const ImgList& imgs, const int32_t* kept_idx,
                             const int32_t* kept_cnt, const uint64_t* bitmask, float softmax_scale, int* status,
                             cudaStream_t s, const DevPlan* plan = nullptr, int n_cap = 0, int inject_stop_group = -1,
                             bool wait_first = true, const AttnParts* parts = nullptr, int64_t* launches = nullptr,
                             const QuadOrder& order = QuadOrder());
AttnParts attention_parts(const TensorGeom& g, int n_img);     // without its pointers
size_t attention_partial_bytes(const TensorGeom& g, int n_img, const AttnParts& parts);
// Kernel attributes on the current device; set when a context is created (scoring: also by the context-free entry).
cudaError_t attention_static_init();
cudaError_t scoring_static_init();
cudaError_t scoring_cluster_static_init();
