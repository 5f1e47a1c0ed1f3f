// K3: masked flash-style joint attention over the kept key tiles (sm_100a).
//
// The unit of work is a quad: one image, one head, four 64-token query blocks = two 128-row Q tiles (the native UMMA
// M).  The four query blocks' ascending kept lists are merged into one union list; the producer streams each key block
// of the union once through shared memory and both tiles use it, which nearly halves the L2 -> SM traffic per MMA and
// leaves room for deep K / V rings.  A tile issues no MMA for a key block that neither of its query blocks kept; inside
// a tile a 64x64 sub-tile whose key block is not in that query block's own list gets P = 0, so each query block attends
// exactly its own kept set.
//
// One thread block per SM works through quads until none is left: it starts with the quad of its own block index and
// then takes over those of blocks that have not started yet (clusterlaunchcontrol.try_cancel: the hardware's own
// scheduler hands them out, in index order, so nothing has to be kept or reset in memory).  The roles walk the quads
// each at its own pace -- while the softmax warps write the result of one quad, the next one's list is built, its Q, K
// and V are on their way and its first scores are computed.  With a thread block per quad, barrier set-up, TMEM
// allocation, mask read, first loads and first scores in front and the epilogue behind cost 6 us a quad, 12 % of a
// dense one at D = 128 and 4608 tokens (three such images, dense, against that kernel in the same run: 725 -> 663 us;
// at ratios 1, .5, .25: 530 -> 486 us; two images of 4429 tokens at D = 64 and ratio .25: 171 -> 160 us).
//
// Roles (640 threads):
//   warps 0-15  softmax, eight warps per tile and four per SM sub-partition: a warp owns 16 query rows, a
//               thread a quarter of two rows (16x256b fragments; 32 scores per key block); fp32 online
//               softmax with lazy rescale of O, P(n) written back over S(n) as bf16, final O / l store
//   warp 16     producer: TMA loads (cp.async.bulk.tensor, 128-byte swizzle) of Q, then the gathered K and V
//               blocks into two rings of shared-memory stages; K(g) and V(g - 1), which the MMA warps need
//               together, complete one barrier
//   warps 17,18 UMMA issue, one warp per tile (warp 17 also owns the TMEM allocation).  S of a
//               tile has NBUF buffers in TMEM (64 fp32 columns each): S(n + NBUF - 1) = Q K^T is
//               issued before O += P(n) V, so the tensor pipe works on the next scores while the
//               softmax warps are busy with the current ones.  Both warps walk the same union
//               list, K ahead of V; a stage is released when both have passed it
//   warp 19     the next quad: takes it over, reads its masks and builds its union list
// TMEM: tile t owns columns [256 t, 256 t + 256): S(n) at 64 (n mod NBUF), O behind the NBUF score buffers
// (two of them and O at 128 for D = 128; three and O at 192 for D = 64, where the columns allow it).
// Every mbarrier wait is bounded; a wait that runs out records RAPID3_ERR_TIMEOUT in the status
// word and the thread block drains its copies, releases its TMEM and exits normally.
#include <float.h>
#include <stddef.h>

#include <algorithm>

#include "common.cuh"
#include "ptx.cuh"

using namespace ptx;

// score buffers per tile: three where the TMEM columns allow it (D = 64: 3 x 64 + 64 of O), else two
#define RAPID3_NBUF(D) ((D) == 64 ? 3 : 2)
namespace {

constexpr int SOFTMAX_WARPS = 16;
constexpr int PRODUCER_WARP = 16, MMA_WARP0 = 17, LIST_WARP = 19;
constexpr int NTHREADS = 32 * (SOFTMAX_WARPS + 4);
constexpr int SOFTMAX_REGS = 104, LIGHT_REGS = 64;     // SPLIT build: registers a thread of the softmax warps, of the others
constexpr int TMEM_COLS = 512;
constexpr int TILE_COLS = 256;      // TMEM columns of one Q tile
constexpr int BLK_BYTES = 8192;     // 64 rows x 128 bytes: one 64-channel half of a 64-token block
constexpr int QHALF_BYTES = 16384;  // one 64-channel half of a 128-row Q tile
// A row's reference maximum moves when a P of it exceeds 2^8; the partial sum of eight that it is part of then does too.
// How far P may exceed 1 costs no precision (P, O and l are floating point throughout), but it costs range: O holds up to
// the row's sum of P times a value.  With sums of 2^16 and growth of 2^12 as the rule, values from 2^112 on overflowed,
// with this one from 2^118 on, and it takes as long (dense attention of three images of 4608 tokens at D = 128: 581.7 and
// 581.7 us; two of 4429 at D = 64: 310.6 and 310.1; bursts).
constexpr float GROWN_SUM = 256.0f, GROWN_LOG2 = 8.0f;
constexpr int MAX_STAGES = 8;
// The next quad is taken over when the producer has this many key blocks of the current one left to load (it runs up
// to a ring ahead of the MMAs): early enough to have its list built in time, late enough not to hold a quad that
// another SM could have started.
// (2, 4 and 10 measured the same.)
constexpr int TAKE_AHEAD = 4;
// Parts of a list; units of work whose results lie in memory between the attention kernel and add_parts_kernel (62 MB at
// D = 128); the shortest rows, in key blocks, and the most quads with which attention_parts() looks for a cut at all.
constexpr int MAX_PARTS = 8, MAX_LEFT = 444, MIN_CUT = 24, MAX_CUT = 600;
// The shortest rows whose blocks go to both tiles by turns (AttnParts::keys): what that saves has to pay for the exchange at the end.
// Attention of one image, every block kept, us, one tile an SM / by turns: D = 64 5 blocks 7.1 / 6.6 (but a step at ratio 0.5, lists of four,
// 11.9 / 12.3), 8 8.8 / 7.8, 12 12.1 / 10.0, 17 14.4 / 11.9, 36 25.4 / 19.9; D = 128 5 7.8 / 7.8, 8 9.9 / 9.5, 12 14.0 / 12.7, 17 16.9 / 15.0,
// 36 29.4 / 26.4 (steps of 6 blocks 15.3 / 15.7, of 8 to 10 1 to 5 % faster).  At D = 128 a block takes 0.58 us, not half of the 0.84 for two tiles: K and V come twice as
// fast, and more stages for them, or V in later groups, did not change that.  Forty steps of contexts of up to 74 quads drawn at random: 3.9 %
// faster in the mean, at worst 2.0 % slower (18 quads of 9 blocks at D = 128); ratios of 0.1 to 0.75 in 110 steps: at worst 1.7 % slower (rows of 6 blocks).
constexpr int KEYS_FROM_64 = 6, KEYS_FROM_128 = 8;
// After a wait has run out the softmax warps go on for up to this many key blocks, each a wait of 16 polls of about 8 us.
// (Over the whole of a quad, with 256 polls a block, that was 2.06 s at two heads of 1024 key blocks; now 4.7 ms.)
constexpr int ABORT_EVERY = 32;

struct AttnParams {
    TensorGeom g;
    ImgList imgs;
    const int32_t* kept_idx;
    const int32_t* kept_cnt;
    const uint32_t* bitmask32;     // optional: the same mask as 32-bit words, [slot][H][nb][words32]
    int words32;
    int n_dense;                   // leading images of the list that keep every block
    const DevPlan* plan;           // optional: image list and n_dense from device memory (grid sized for n_cap images)
    int* status;
    float scale_log2;
    QuadOrder order;               // optional: the order of the sparse images' quads without text rows
    AttnParts parts;               // SPLIT build: how many units of work the union list of a quad goes to
    uint32_t div_all, div_text, div_light, div_pure, div_mixed, div_heads;   // divider() of the quads of a head by kind, and of the heads
    bool wait_first;               // nothing is read before the kernel in front has ended
    int stop_group;                // failure-injection build of the kernel only: the producer stops before this group
};

// x / d as a product with divider(d): exact while x d < 2^32.  Quads number below 2^24 and those of a head 256 at most; pairs and
// heads below 2^16.  (A division takes some twenty instructions, which a thread block's first quad waits for: see the list warp.)
__host__ __device__ constexpr uint32_t divider(uint32_t d) { return d < 2 ? 0u : 0xffffffffu / d + 1u; }
__device__ __forceinline__ int divide(int x, uint32_t by) { return (int)__umulhi((uint32_t)x, by) + (by ? 0 : x); }

// Reference maximum, times -c2, of a row all of whose scores so far are -inf, where O and l may be added to others' (parts, blocks by turns).
constexpr float LOWEST = FLT_MAX;
// 1 / row sum: 0 for a row that keeps nothing, not a number for one that keeps blocks and has no score above -inf in any: softmax's 0 / 0.
__device__ __forceinline__ float one_over(float sum, float nm) {
    return sum > 0.f ? 1.f / sum : nm == LOWEST ? __int_as_float(0x7fffffff) : 0.f;
}

template <int D>
struct Cfg {
    static constexpr int DH = D / 64;                       // 64-channel halves per row
    static constexpr int QTILE_BYTES = 128 * D * 2;         // one 128-row Q tile
    static constexpr int KV_BYTES = 64 * D * 2;             // one key block of K or of V
    static constexpr int KS = (D == 128) ? 4 : 8;           // K ring stages
    static constexpr int VS = (D == 128) ? 4 : 8;           // V ring stages
    static constexpr int DATA_BYTES = 2 * QTILE_BYTES + (KS + VS) * KV_BYTES;
    static constexpr int NBUF = RAPID3_NBUF(D);             // score buffers (64 columns each) per tile
    static constexpr int O_COL = 64 * NBUF;                 // O accumulator behind them: 64 NBUF + D <= 256 columns per tile
};

// One quad as the roles see it, written by the list warp.
struct Quad {
    int n_u;                            // entries of the union list; -1: no more quads
    int b, h;                           // image, head (of the tensors)
    int tok[4];                         // first token of the quad's query blocks (>= N: there is no such block); tile t: 2 t, 2 t + 1
    int part, parts, store;             // SPLIT build: this unit's part of the quad's list, of how many; where part 0 leaves its results
    uint32_t ent[RAPID3_MAX_NB];        // ascending key blocks: ENT_BLK up; bit a: query block a keeps it; ENT_TAIL
};

struct __align__(16) Ctl {
    uint4 taken;                        // answer of the last try_cancel
    unsigned long long taken_full, near_end, first_known;
    unsigned long long quad_full[2], quad_empty[2];
    unsigned long long q_full, q_empty;
    unsigned long long k_full[MAX_STAGES], k_empty[MAX_STAGES];   // k_full[g % KS]: group g = K(g) and V(g - 1) have landed
    unsigned long long v_empty[MAX_STAGES];
    unsigned long long s_full[2][3], p_full[2][3];
    unsigned long long pv_done[2][2], o_done[2], drain[2], handed[SOFTMAX_WARPS];
    uint32_t tmem_base;
    int n_early;                        // groups of the first quad that the producer loads before its list is there
    volatile int abort_flag;
    uint32_t bm[4][32];                 // the list warp's scratch
    float nm[SOFTMAX_WARPS][16];        // SPLIT build: the reference maxima of a warp's rows, times -c2, as they last moved
    Quad quad[2];
};
constexpr uint32_t ENT_TAIL = 16u;      // the sequence ends inside this key block
template <int D>
constexpr int PARTIAL_F4 = D / 8 + 1;   // float4 that a lane leaves of a part: its share of O; reference maxima and sums of its two rows
constexpr int ENT_BLK = 8;              // the block's number from this bit on
constexpr int QUAD_USERS = SOFTMAX_WARPS + 3;   // warps that read a quad

template <int D>
constexpr size_t attn_smem_bytes() { return (size_t)Cfg<D>::DATA_BYTES + sizeof(Ctl) + 1024; }

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Lane c of a quad of lanes holds words 0..3 of column pairs (c, c + 4, c + 8, c + 12); afterwards it holds words
// 4 c .. 4 c + 3: a 4 x 4 transpose, two exchanges.
__device__ __forceinline__ uint4 quad_transpose(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, int c) {
    const bool b0 = c & 1, b1 = c & 2;
    const uint32_t x = __shfl_xor_sync(0xffffffffu, b0 ? w0 : w1, 1), y = __shfl_xor_sync(0xffffffffu, b0 ? w2 : w3, 1);
    const uint32_t p0 = b0 ? x : w0, p1 = b0 ? w1 : x, q0 = b0 ? y : w2, q1 = b0 ? w3 : y;
    const uint32_t r0 = __shfl_xor_sync(0xffffffffu, b1 ? p0 : q0, 2), r1 = __shfl_xor_sync(0xffffffffu, b1 ? p1 : q1, 2);
    return b1 ? make_uint4(r0, r1, q0, q1) : make_uint4(p0, p1, r0, r1);
}

// Place of the `rest`-th quad in the order of the classes; a lane holds those of quads 4 lane .. 4 lane + 3, 0xff: no quad.
__device__ __forceinline__ int order_find(uint32_t cls, int rest, int lane) {
    static_assert(ORDER_LAST == 4 * 32, "a lane holds four classes");
    auto below = [&](uint32_t c) { return __popc(__vcmpltu4(cls, c * 0x01010101u)) >> 3; };   // of the lane's quads, those of a class below c
    uint32_t c = 0u;                                     // the quad's class: the last with no more than `rest` quads below it
#pragma unroll
    for (uint32_t bit = ORDER_CLASSES / 2; bit > 0; bit >>= 1)
        if ((int)__reduce_add_sync(0xffffffffu, (uint32_t)below(c | bit)) <= rest) c |= bit;
    const int lower = below(c), own = below(c + 1u) - lower;
    int before = own;                                    // quads of the class in the lanes below this one
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, before, o);
        if (lane >= o) before += v;
    }
    int skip = rest - (int)__reduce_add_sync(0xffffffffu, (uint32_t)lower) - (before - own), at = -1;
#pragma unroll
    for (int x = 0; x < 4; ++x)
        if (((cls >> (8 * x)) & 0xffu) == c && skip-- == 0) at = 4 * lane + x;
    return (int)__reduce_max_sync(0xffffffffu, at);      // the other lanes have -1
}

// Maxima of a quad's two rows over one key block, from the four threads' 16x256b fragments.
__device__ __forceinline__ void row_maxima(const uint32_t (&r)[32], float& lo, float& hi) {
    lo = hi = -INFINITY;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        lo = max3(lo, __uint_as_float(r[4 * k]), __uint_as_float(r[4 * k + 1]));
        hi = max3(hi, __uint_as_float(r[4 * k + 2]), __uint_as_float(r[4 * k + 3]));
    }
    lo = fmaxf(lo, __shfl_xor_sync(0xffffffffu, lo, 1));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, 1));
    lo = fmaxf(lo, __shfl_xor_sync(0xffffffffu, lo, 2));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, 2));
}

// INJECT = true is the failure-injection build behind rapid3_debug_inject_timeout: the producer
// stops before group prm.stop_group and every wait gives up after 2^12 polls, so the waits of all
// roles run out and the abort path (status word, drain of the copies in flight, UMMA drain, TMEM
// release) is what runs.  The product launches only use INJECT = false.
//
// SPLIT = true is the build for contexts whose quads leave SMs without work: the union list of a quad is cut into
// parts of equal length, each a unit of work (attention_parts() says how many).  A softmax warp leaves its rows of a part -- O,
// not divided by the row sums, the sums and the reference maxima -- in global memory, and add_parts_kernel makes the result
// of them.  (Added up by the last part of a quad to arrive, in this kernel, they cost its main loop 12 to 14 %: registers.)
//
// ORDERED is the build for launches whose last quads are handed out by their length (QuadOrder).
//
// MASKS: the sparse images' blocks come as the selection kernel's bitmask, or there are none, and the code for the caller's lists is
// left out.  Both builds have 96 registers and spill the same five words; by turns, whole steps, us, with that code / without:
// 1296 quads at D = 128 530.7 / 524.7, 2592 1184.6 / 1170.0, 1584 of a 2048^2 image 1117.6 / 1110.4; all dense 1296 669.3 / 660.9,
// 1584 2848 / 2813.  Dense launches at D = 64 keep the build with it: 840 quads 304.5 / 306.3, 288 36.8 / 37.0.
//
// KEYS is the build for contexts in which every tile of the largest launch has an SM to itself (AttnParts::keys).  Both tiles of the
// thread block then hold the same query rows, and the blocks of the list go to them by turns; at the end each hands half of its
// channels to the other.
template <int D, bool INJECT = false, bool SPLIT = false, bool ORDERED = false, bool MASKS = ORDERED, bool KEYS = false>
__global__ void __launch_bounds__(NTHREADS, 1)
attn_kernel(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
            const __grid_constant__ CUtensorMap tmv, uint16_t* __restrict__ out, const __grid_constant__ AttnParams prm) {
    using C = Cfg<D>;
    constexpr int DH = C::DH, KS = C::KS, VS = C::VS, NBUF = C::NBUF, O_COL = C::O_COL;
    constexpr int AHEAD = (NBUF - 1) * (KEYS ? 2 : 1);   // how many blocks of the list the scores are ahead of the products P V
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t pad = ((raw + 1023u) & ~1023u) - raw;
    uint8_t* smem = smem_raw + pad;
    const uint32_t sQ = raw + pad, sK = sQ + 2 * C::QTILE_BYTES, sV = sK + KS * C::KV_BYTES;
    Ctl* ctl = reinterpret_cast<Ctl*>(smem + C::DATA_BYTES);

    const int tid = threadIdx.x, lane = tid % 32;
    // the shuffle makes the warp index provably warp-uniform, so role branches and the address
    // arithmetic inside them can live in uniform registers
    const int warp = __shfl_sync(0xffffffffu, tid / 32, 0);
    const TensorGeom& g = prm.g;
    const int nb = g.nb, N = g.N;
    const int n_images = prm.plan ? __ldcg(&prm.plan->all.n) : prm.imgs.n;
    int n_quads = ((nb + 3) >> 2) * g.H * n_images;      // units of work: quads, ...
    if constexpr (SPLIT) n_quads = attention_units(g, prm.parts, n_images, prm.plan ? __ldcg(&prm.plan->n_dense) : prm.n_dense);   // ... parts, ...
    // ... or halves of either: where the two tiles of every unit find an SM each, they go to two thread blocks.  A tile that
    // has the SM to itself goes through its key blocks in 0.66 and 0.56 us (D = 128, 64), where two that share it take 0.84 and
    // 0.72 (whole steps of one image: 6 heads x 11 blocks 16.4 -> 13.8 us, 2 heads x 22 blocks at D = 64 26.3 -> 23.8; with more
    // tiles than SMs the shared K and V stream wins).
    const int halves = 2 * n_quads <= SM_COUNT ? 1 : 0;
    n_quads <<= halves;
    if ((int)blockIdx.x >= n_quads) {                    // device-resident plan: fewer images than the grid covers
        // When none attends, no other thread block waits for the selection kernel: the grid must not end before that does
        // (it may still have the plan to read, which the next call rewrites).
        if (n_quads == 0) grid_dependency_wait();
        return;
    }

    const uint32_t bQ = smem_u32(&ctl->q_full), bQE = smem_u32(&ctl->q_empty);
    const uint32_t bKF = smem_u32(&ctl->k_full[0]), bKE = smem_u32(&ctl->k_empty[0]);
    const uint32_t bVE = smem_u32(&ctl->v_empty[0]);
    const uint32_t bSF = smem_u32(&ctl->s_full[0][0]), bPF = smem_u32(&ctl->p_full[0][0]);   // [tile][buf]: + 24 t + 8 buf
    const uint32_t bPV = smem_u32(&ctl->pv_done[0][0]);                                      // [tile][block parity]: + 16 t + 8 (n & 1)
    const uint32_t bOD = smem_u32(&ctl->o_done[0]);                                          // [tile]: + 8 t
    const uint32_t bUF = smem_u32(&ctl->quad_full[0]), bUE = smem_u32(&ctl->quad_empty[0]);  // quad i: + 8 (i & 1)
    const uint32_t bNE = smem_u32(&ctl->near_end), bT = smem_u32(&ctl->taken_full), bFK = smem_u32(&ctl->first_known);

    // ---------------------------------------------------------------- setup
    // The list warp needs nothing of it until it arrives on an mbarrier, so it only waits for warp 0 (named barrier 1), later on, and
    // meets the others on barrier 2 by arriving.  Barrier 2 is met nowhere else: nothing keeps the list warp back until the others are past it, and
    // on the teardown's barrier 0 a second arrival of its would stand in for a warp that is late (the one that allocates tensor memory, say).
    if (warp == 0) {
        constexpr uint32_t at = offsetof(Ctl, taken_full) / 8, bars = offsetof(Ctl, tmem_base) / 8 - at;
        auto has = [&](uint32_t x, size_t member, int n) { return x + at - (uint32_t)(member / 8) < (uint32_t)n; };
#pragma unroll
        for (uint32_t x = lane; x < bars; x += 32) {
            uint32_t count = 1;
            if (has(x, offsetof(Ctl, quad_empty), 2)) count = QUAD_USERS;
            if (has(x, offsetof(Ctl, q_empty), 1) || has(x, offsetof(Ctl, k_empty), 2 * MAX_STAGES)) count = 2;   // both tiles pass a stage before it is refilled
            if (has(x, offsetof(Ctl, p_full), 6)) count = 8;                   // one arrival per softmax warp of the tile
            if (has(x, offsetof(Ctl, handed), SOFTMAX_WARPS)) count = 32;
            mbar_init(smem_u32(ctl) + 8 * (at + x), count);
        }
        if (lane == 0) ctl->abort_flag = 0;
        fence_mbar_init();
        __syncwarp();
        bar_arrive(1, 64);
    }
    if (warp == PRODUCER_WARP && lane < 3) prefetch_tmap(lane == 0 ? &tmq : lane == 1 ? &tmk : &tmv);
    if (warp == LIST_WARP && !prm.plan) {
        // the kernel's arguments are not in the SM's cache yet: what the first quad's index arithmetic ends with is fetched beside it
        asm volatile("" ::"r"(prm.imgs.batch[0]), "r"(prm.imgs.slot[0]), "r"(g.pair_stride), "r"(g.h0));
    }
    if (warp == MMA_WARP0) {
        tmem_alloc(smem_u32(&ctl->tmem_base), TMEM_COLS);
        tmem_relinquish();
        tc_fence_before();
    }
    if (prm.wait_first) grid_dependency_wait();
    // The launch's own word (the status stays until the host has read it).  Thread blocks start in order, and a wait runs out only
    // after thousands of polls, so nothing sets it before this; what read it last has ended before the selection kernel began, if
    // that is in front.
    if (SPLIT && blockIdx.x == 0 && tid == 0) __stcg(prm.parts.given_up, 0);
    if (warp == LIST_WARP) bar_arrive(2, NTHREADS);
    else bar_sync(2, NTHREADS);
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;

    auto fail = [&]() {
        atomicExch(prm.status, RAPID3_ERR_TIMEOUT);
        if (SPLIT) atomicExch(prm.parts.given_up, 1);
        ctl->abort_flag = 1;
    };
    // bounded wait that also gives up quickly once another role has failed
    auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
        constexpr uint32_t limit = INJECT ? (1u << 12) : (1u << 22);
        for (uint32_t it = 0; it < limit; ++it) {
            if (mbar_try_wait(bar, parity)) return true;
            if ((it & 15u) == 15u && ctl->abort_flag) return false;
        }
        fail();
        return false;
    };
    // the same for a converged warp, with a warp-uniform result
    auto wait_warp = [&](uint32_t bar, uint32_t parity) -> bool {
        return __all_sync(0xffffffffu, wait(bar, parity));
    };
    // Q tiles of a quad, and groups of its K and V blocks: group gi = K block gi together with V block gi - 1, which the
    // MMA warps need as a pair before they issue S(gi) = Q K(gi)^T and O += P(gi - 1) V(gi - 1), so that the pair
    // completes ONE barrier and costs them one wait per key block instead of two.  Group 0 is K(0) alone, group n_u is
    // V(n_u - 1) alone.  Groups and V blocks are numbered through all quads of the thread block: group gi of a quad has
    // number G = G0 + gi (n_u + 1 of them, the last without a K block), V block j number W0 + j (n_u of them).
    auto load_q = [&](const Quad& u) {
        mbar_arrive_expect_tx(bQ, 2 * C::QTILE_BYTES);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int dh = 0; dh < DH; ++dh)
                tma_load_4d(sQ + (a >> 1) * C::QTILE_BYTES + dh * QHALF_BYTES + (a & 1) * BLK_BYTES, &tmq, bQ, dh * 64,
                            u.tok[a], u.h, u.b);
    };
    auto issue_group = [&](const Quad& u, uint32_t G, int kb, uint32_t W, int vb) {   // key blocks, -1: none
        const uint32_t bar = bKF + 8 * (G % KS);
        mbar_arrive_expect_tx(bar, (kb >= 0 ? C::KV_BYTES : 0) + (vb >= 0 ? C::KV_BYTES : 0));
        if (kb >= 0) {
#pragma unroll
            for (int dh = 0; dh < DH; ++dh)
                tma_load_4d(sK + (G % KS) * C::KV_BYTES + dh * BLK_BYTES, &tmk, bar, dh * 64, kb * 64, u.h, u.b);
        }
        if (vb >= 0) {
#pragma unroll
            for (int dh = 0; dh < DH; ++dh)
                tma_load_4d(sV + (W % VS) * C::KV_BYTES + dh * BLK_BYTES, &tmv, bar, dh * 64, vb * 64, u.h, u.b);
        }
    };

    // The pool is the launch's 640 x 96: 512 x 104 + 128 x 64.  Without it this build keeps ten words of the softmax warps in
    // local memory; in the other builds it gains nothing (ordered, D = 128: fused step of 432 quads 197.0 us without, 199.8 with).
    if ((SPLIT || KEYS) && warp >= SOFTMAX_WARPS) reg_dec<LIGHT_REGS>();
    if (warp == LIST_WARP) {
        // ------------------------------------------------------------ quads and their union lists
        // A thread block's first quad waits for this warp, whose code the SM has to fetch first: what lies in front of the first list is
        // short, and beside the set-up as far as it can be.  Divisions by the launch's constants as products, a member a lane
        // instead of four in a row, no masks where every block is kept, the arguments fetched early: the first list 2.1 -> 1.3 us
        // after the start of a thread block, the first Q's loads 1.6 -> 0.9 (steps of 288 quads at D = 64 41.7 -> 40.5 us, one dense
        // image of 12 quads 9.7 -> 9.1).
        // one lane polls: these waits are long, and the other lanes' polls would only take issue slots
        auto wait_lane0 = [&](uint32_t bar, uint32_t parity) -> bool {
            return __shfl_sync(0xffffffffu, (int)(lane != 0 || wait(bar, parity)), 0);
        };
        int L = blockIdx.x;
        bool waited = false;                             // for the selection kernel, see below
        uint32_t classes = 0;                            // of four quads in the order, once `have_classes`
        bool have_classes = false;
        for (uint32_t i = 0;; ++i) {
            Quad& u = ctl->quad[i & 1];
            if (i > 1 && !wait_lane0(bUE + 8 * (i & 1), ((i >> 1) & 1) ^ 1)) break;
            if (L < 0) {
                if (lane == 0) {
                    u.n_u = -1;
                    mbar_arrive(bUF + 8 * (i & 1));
                }
                break;
            }
            // Work order, longest first (quads are handed out in index order, so this is longest-processing-time-first
            // scheduling): every quad of the dense images and the quads of the sparse images that hold a text query
            // block walk all nb key blocks; the other quads of the sparse images follow, image by image in the list's
            // order (descending keep ratio).
            int quad, h, p;
            const int half = halves ? L & 1 : -1;    // the tile to work on, or both
            L >>= halves;
            int part = 0, parts = 1;
            {
                const int nq = (nb + 3) >> 2, ntq = min(nq, (g.n_text_blocks + 3) >> 2);
                const int n_all = prm.plan ? __ldcg(&prm.plan->all.n) : prm.imgs.n;
                const int nd = prm.plan ? __ldcg(&prm.plan->n_dense) : prm.n_dense, ns = n_all - nd;
                const int heavy_dense = nd * g.H * nq, heavy_sparse = ns * g.H * ntq;
                if constexpr (SPLIT) {                   // in units first: the parts of a quad follow one another
                    const AttnParts& ap = prm.parts;
                    const int ud = heavy_dense * ap.dense, ut = heavy_sparse * ap.text;
                    int store = 0, quads = 0;            // units before these that leave results; quads before these
                    if (L < ud) {
                        parts = ap.dense;
                    } else if (L < ud + ut) {
                        L -= ud;
                        parts = ap.text;
                        store = ap.dense > 1 ? ud : 0;
                        quads = heavy_dense;
                    } else {
                        L -= ud + ut;
                        parts = ap.light;
                        store = (ap.dense > 1 ? ud : 0) + (ap.text > 1 ? ut : 0);
                        quads = heavy_dense + heavy_sparse;
                    }
                    part = L % parts;
                    if (lane == 0) u.store = store + L - part;
                    L = quads + L / parts;
                    if (lane == 0) {
                        u.part = part;
                        u.parts = parts;
                    }
                }
                int first = 0, n = nq;                   // the quads of a head of this kind: so many from `first` on
                uint32_t by = prm.div_all;
                p = 0;
                if (L >= heavy_dense) {
                    L -= heavy_dense;
                    p = nd;
                    if (L < heavy_sparse) {
                        // those of text rows alone first: they need no mask, which may not be there yet
                        const int ntf = SPLIT ? ntq : g.n_text_blocks >> 2, n_full = ns * g.H * ntf;
                        const bool full = L < n_full;
                        first = full ? 0 : ntf;
                        n = full ? ntf : ntq - ntf;
                        by = SPLIT ? prm.div_text : full ? prm.div_pure : prm.div_mixed;
                        if (!full) L -= n_full;
                    } else {
                        L -= heavy_sparse;
                        first = ntq;
                        n = nq - ntq;
                        by = prm.div_light;
                        const int in_order = order_after(ns * g.H * n, heavy_dense + heavy_sparse), rest = L - in_order;
                        if (ORDERED && rest >= 0) {
                            // the quad at place `rest` of the order that the selection kernel has found: of four classes a lane
                            if (!have_classes) {
                                if (!waited) grid_dependency_wait();
                                waited = have_classes = true;
                                classes = __ldcg(reinterpret_cast<const uint32_t*>(prm.order.cls) + lane);
                                const int left = ns * g.H * n - in_order - 4 * lane;     // of the lane's, the bytes behind those count for nothing
                                if (left < 4) classes |= left > 0 ? 0xffffffffu << (8 * left) : 0xffffffffu;
                            }
                            L = in_order + order_find(classes, rest, lane);
                        }
                    }
                }
                const int pair = divide(L, by);          // (image, head) of this kind
                quad = first + L - pair * n;
                const int image = divide(pair, prm.div_heads);
                h = pair - image * g.H;
                p += image;
            }
            const int b = prm.plan ? __ldcg(&prm.plan->all.batch[p]) : prm.imgs.batch[p];
            const int slot = prm.plan ? __ldcg(&prm.plan->all.slot[p]) : prm.imgs.slot[p];
            // Lanes a, a + 4, ... hold member a's query block; which members there are, one of the other half counting like one past the end.
            // (KEYS: both tiles hold the unit's two.)
            const int own = quad_block(g, quad, KEYS ? 2 * half + (lane & 1) : lane & 3);
            const bool here_own = own < nb && (KEYS || half < 0 || ((lane & 3) >> 1) == half);
            const uint32_t here = __ballot_sync(0xffffffffu, here_own) & 15u;
            const bool masks = MASKS || prm.bitmask32 != nullptr;      // of the selection kernel (it finds the order), else lists of the caller's
            // a dense image's quad, or one of text rows in a mask of the selection kernel: every block is kept, no mask is read
            const bool all_kept = slot < 0 || (masks && 4 * quad + 3 < g.n_text_blocks);
            // the members whose kept blocks m[a] below holds: where a list is cut into parts depends on the whole quad
            const uint32_t listed = SPLIT && parts > 1 ? __ballot_sync(0xffffffffu, own < nb) & 15u : here;
            if (i == 0) bar_sync(1, 64);                 // the barriers are set up
            if (lane < 4) u.tok[lane] = (here_own ? own : nb) * 64;
            __syncwarp();
            if (lane == 0) {
                u.b = b;
                u.h = g.h0 + h;
                if (i == 0) {
                    // The first quad's Q tiles do not depend on the mask, nor do key blocks known before it is read: a
                    // dense image keeps every block, and a mask of the selection kernel keeps the text blocks in every
                    // row, so the union list starts 0, 1, ....  The producer loads them while the list is built (by this
                    // lane, ahead of the masks, they kept the first list back: steps of 288 quads at D = 64 41.6 -> 40.8 us,
                    // of 24 at D = 128 23.9 -> 23.0, lists of the caller's for 324 quads 80.2 -> 78.9).
                    // (no members: the second half of a ragged last quad)
                    int n_early = (!INJECT && here && (all_kept || masks)) ? min(min(all_kept ? nb : g.n_text_blocks, nb), KS) : 0;
                    if (SPLIT && parts > 1) n_early = part == 0 ? min(n_early, (all_kept ? nb : g.n_text_blocks) / parts) : 0;   // its part of the list is no shorter
                    ctl->n_early = n_early;
                    mbar_arrive(bFK);
                }
            }
            int n_u;
            auto entry = [&](uint32_t f, int j, int at) {
                return (KEYS ? f & (at & 1 ? 12u : 3u) : f) | ((j + 1) * 64 > N ? ENT_TAIL : 0u) | ((uint32_t)j << ENT_BLK);
            };
            if (all_kept) {
                const int first = SPLIT ? nb * part / parts : 0, last = !here ? first : SPLIT ? nb * (part + 1) / parts : nb;
                n_u = last - first;
                for (int j = first + lane; j < last; j += 32) u.ent[j - first] = entry(here, j, j - first);
            } else {
                // m[a] = 32 bits of the set of key blocks that member a keeps: from the bitmask when the caller has one,
                // else rebuilt from the kept list.
                const int nw = (nb + 31) >> 5;
                uint32_t m[4];
                // Launched as a dependent of the selection kernel, the masks have to be waited for once.  They are read
                // past the L1 (ld.global.cg): this thread block may have started before they were written, and an L1
                // line of an earlier step must not answer.
                if (!waited) grid_dependency_wait();
                waited = true;
                if (masks) {
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const long long row = ((long long)slot * g.H + h) * nb + __shfl_sync(0xffffffffu, own, a);
                        m[a] = ((listed >> a) & 1u) && lane < nw ? __ldcg(prm.bitmask32 + row * prm.words32 + lane) : 0u;
                    }
                } else {
#pragma unroll
                    for (int a = 0; a < 4; ++a) ctl->bm[a][lane] = 0u;
                    __syncwarp();
                    // the counts and the first 64 entries of all four rows on their way at once, the entries before their counts are
                    // known (324 quads of 10 to 33 blocks: whole staged calls 81.5 -> 80.3 us; 144 quads 40.9 -> 38.3)
                    const int32_t* lst[4];
                    int cnt[4], first[4], second[4];
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const bool in = (listed >> a) & 1u;
                        const int block = __shfl_sync(0xffffffffu, own, a);
                        const long long row = ((long long)slot * g.H + h) * nb + (in ? block : 0);
                        lst[a] = prm.kept_idx + row * nb;
                        cnt[a] = in ? __ldcg(prm.kept_cnt + row) : 0;
                        first[a] = in && lane < nb ? __ldcg(lst[a] + lane) : 0;
                        second[a] = in && 32 + lane < nb ? __ldcg(lst[a] + 32 + lane) : 0;
                    }
                    auto put = [&](int a, int e, int j) {
                        if (e >= min(cnt[a], nb)) return;
                        if ((unsigned)j < (unsigned)nb) atomicOr(&ctl->bm[a][j >> 5], 1u << (j & 31));
                        else atomicExch(prm.status, RAPID3_ERR_BAD_LIST);
                    };
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        put(a, lane, first[a]);
                        put(a, 32 + lane, second[a]);
                    }
                    const int most = min(max(max(cnt[0], cnt[1]), max(cnt[2], cnt[3])), nb);
                    for (int e = 64 + lane; e < most; e += 32) {
                        int j[4];
#pragma unroll
                        for (int a = 0; a < 4; ++a) j[a] = e < min(cnt[a], nb) ? __ldcg(lst[a] + e) : 0;
#pragma unroll
                        for (int a = 0; a < 4; ++a) put(a, e, j[a]);
                    }
                    __syncwarp();
#pragma unroll
                    for (int a = 0; a < 4; ++a) m[a] = ctl->bm[a][lane];
                }
                // the position of a key block in the ascending union list is the number of union bits below it
                auto union_bits_below = [&](uint32_t bits, int& all) -> int {
                    int x = __popc(bits);
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int v = __shfl_up_sync(0xffffffffu, x, o);
                        if (lane >= o) x += v;
                    }
                    all = __shfl_sync(0xffffffffu, x, 31);
                    return x - __popc(bits);
                };
                if (SPLIT && parts > 1) {                    // of the quad's union, the blocks from `first` up to `last` are this part's
                    uint32_t from = m[0] | m[1] | m[2] | m[3], to = from;
                    const int at = union_bits_below(from, n_u), first = n_u * part / parts, last = n_u * (part + 1) / parts;
                    for (int x = min(max(first - at, 0), 32); x > 0; --x) from &= from - 1u;
                    for (int x = min(max(last - at, 0), 32); x > 0; --x) to &= to - 1u;
#pragma unroll
                    for (int a = 0; a < 4; ++a) m[a] &= (here >> a) & 1u ? from & ~to : 0u;
                }
                const uint32_t un = m[0] | m[1] | m[2] | m[3];
                const int below = union_bits_below(un, n_u);
                for (int w = 0; w < nw; ++w) {
                    const uint32_t uw = __shfl_sync(0xffffffffu, un, w);
                    const int pos = __shfl_sync(0xffffffffu, below, w) + __popc(uw & ((1u << lane) - 1u));
                    uint32_t f = 0u;
#pragma unroll
                    for (int a = 0; a < 4; ++a) f |= ((__shfl_sync(0xffffffffu, m[a], w) >> lane) & 1u) << a;
                    if (f) {
                        const int j = 32 * w + lane;
                        u.ent[pos] = entry(f, j, pos);
                    }
                }
            }
            if (lane == 0) u.n_u = n_u;
            __syncwarp();
            if (lane == 0) mbar_arrive(bUF + 8 * (i & 1));
            if (KEYS) {                                  // the memory of K and V is used otherwise at the end
                L = -1;
                continue;
            }
            // the next quad, when this one is nearly through
            if (!wait_lane0(bNE, i & 1)) break;
            if (lane == 0) {
                mbar_arrive_expect_tx(bT, 16);
                clc_try_cancel(smem_u32(&ctl->taken), bT);
            }
            __syncwarp();
            // no way out before the answer is here: it is written into this thread block's shared memory
            if (!__all_sync(0xffffffffu, mbar_wait(bT, i & 1))) {
                if (lane == 0) fail();
                break;
            }
            L = clc_taken(smem_u32(&ctl->taken));
            if (L >= n_quads) L = -1;                    // none of the blocks behind it has work either
        }
        // A thread block that read no mask still ends after the selection kernel, so that the grid as a whole does.
        if (!waited) grid_dependency_wait();
    } else if (warp == PRODUCER_WARP) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            uint32_t G = 0, W0 = 0, n_q = 0;             // group to be issued next, the quad's first V block, Q loads so far
            bool ok = wait(bFK, 0);
            uint32_t i = 0;
            if (ok) {                                    // first use of all stages, nothing to wait for
                const int n_early = ctl->n_early;
                load_q(ctl->quad[0]);
                n_q = 1;
                for (; (int)G < n_early; ++G) issue_group(ctl->quad[0], G, G, G - 1, (int)G - 1);
            }
            for (; ok; ++i) {
                const Quad& u = ctl->quad[i & 1];
                if (!(ok = wait(bUF + 8 * (i & 1), (i >> 1) & 1))) break;
                const int n_u = u.n_u;
                if (n_u < 0) break;
                const int n_early = i == 0 ? ctl->n_early : 0;
                if (n_early > max(n_u - TAKE_AHEAD, 0)) mbar_arrive(bNE);
                for (int gi = n_early; gi <= n_u; ++gi) {
                    if (INJECT && gi == min(prm.stop_group, n_u)) { ok = false; break; }
                    if (gi == max(n_u - TAKE_AHEAD, 0)) mbar_arrive(bNE);
                    // A group is issued once both ring stages it fills have been released.  The K stage's release also
                    // tells that both MMA warps are past their wait on this barrier's previous phase (group G - KS),
                    // so it is awaited even when the group brings no K block.
                    if (!(ok = wait(bKE + 8 * (G % KS), ((G / KS) & 1) ^ 1))) break;
                    const uint32_t W = W0 + gi - 1;
                    if (gi > 0 && !(ok = wait(bVE + 8 * (W % VS), ((W / VS) & 1) ^ 1))) break;
                    issue_group(u, G, gi < n_u ? (int)(u.ent[gi] >> ENT_BLK) : -1, W, gi > 0 ? (int)(u.ent[gi - 1] >> ENT_BLK) : -1);
                    ++G;
                    if (gi == 0 && i > 0) {              // the quad before has computed its last scores: its Q can go
                        if (!(ok = wait(bQE, (i - 1) & 1))) break;
                        load_q(u);
                        ++n_q;
                    }
                }
                if (!ok) break;
                W0 += n_u;
                mbar_arrive(bUE + 8 * (i & 1));
            }
            if (INJECT || ctl->abort_flag) {
                // drain: do not leave the CTA while bulk copies may still land in its shared memory
                if (n_q > 0) mbar_wait(bQ, (n_q - 1) & 1, 1u << 20);
                for (uint32_t x = G > KS ? G - KS : 0; x < G; ++x)
                    mbar_wait(bKF + 8 * (x % KS), (x / KS) & 1, 1u << 20);
            }
        }
        __syncwarp();
    } else if (warp >= MMA_WARP0) {
        // ------------------------------------------------------------ UMMA issue, one warp per tile
        // At D = 64 the whole warp runs the loop converged and one elected lane issues the tcgen05 instructions; at
        // D = 128, with one block's scores fewer to bridge the time between a barrier's completion and the next issue,
        // the elected lane runs the loop alone, without the votes and warp barriers that convergence costs (attention
        // of three 1024^2 images at ratios 1, .5, .25: 497 against 505 us; a 2048^2 one: 1054 against 1081 us; at
        // D = 64 it is the other way round, 263 against 265 us).  Both warps pass over every block of
        // the union list, K one block ahead of V, also over blocks their tile does not use: the
        // stage barriers then see every phase in order and a stage is refilled only after both
        // tiles are past it.
        const int t = warp - MMA_WARP0;
        const uint32_t tile_bits = 3u << (2 * t);
        constexpr bool SOLO = (D == 128);
        const bool leader = elect_one();
        auto mma_wait = [&](uint32_t bar, uint32_t parity) -> bool {
            if constexpr (SOLO) return wait(bar, parity);
            else return wait_warp(bar, parity);
        };
        if (!SOLO || leader) {
            const uint32_t tbase = tmem_base + t * TILE_COLS;
            const uint32_t tO = tbase + O_COL;
            const uint32_t qb = sQ + t * C::QTILE_BYTES;
            const uint32_t bSFt = bSF + 24 * t, bPFt = bPF + 24 * t;
            constexpr uint32_t idesc_qk = idesc_bf16(128, 64, 0, 0);
            constexpr uint32_t idesc_pv = idesc_bf16(128, D, 0, 1);
            int n_qk = 0, n_pv = 0;                        // blocks of this tile issued so far, in all quads
            uint32_t G0 = 0, W0 = 0;
            bool ok = true;
            for (uint32_t i = 0; ok; ++i) {
                const Quad& u = ctl->quad[i & 1];
                if (!(ok = mma_wait(bUF + 8 * (i & 1), (i >> 1) & 1))) break;
                const int n_u = u.n_u;
                if (n_u < 0) break;
                const int n_pv0 = n_pv;
                // waits for group j (K(j) and V(j - 1), see the producer), then issues S = Q K(j)^T
                auto k_step = [&](int j) -> bool {
                    const uint32_t s = (G0 + j) % KS;
                    if (!(mma_wait(bKF + 8 * s, ((G0 + j) / KS) & 1))) return false;
                    if (j >= n_u) {                        // the last group holds V(n_u - 1) only
                        if (leader) {
                            mbar_arrive(bKE + 8 * s);
                            if (n_u == 0) tc_commit(bQE);
                        }
                        return true;
                    }
                    const bool use = u.ent[j] & tile_bits;
                    if (use) {
                        tc_fence_after();
                        const uint32_t tS = tbase + 64 * (n_qk % NBUF);
                        const uint32_t kb = sK + s * C::KV_BYTES;
                        if (leader) {
    #pragma unroll
                            for (int ks = 0; ks < D / 16; ++ks)
                                mma_ss(tS, smem_desc_sw128(qb + (ks / 4) * QHALF_BYTES + (ks % 4) * 32, 16, 1024),
                                       smem_desc_sw128(kb + (ks / 4) * BLK_BYTES + (ks % 4) * 32, 16, 1024), idesc_qk, ks > 0);
                            tc_commit(bKE + 8 * s);
                            tc_commit(bSFt + 8 * (n_qk % NBUF));
                        }
                        ++n_qk;
                    } else if (leader) {
                        mbar_arrive(bKE + 8 * s);
                    }
                    if (leader && j == n_u - 1) tc_commit(bQE);
                    if (!SOLO) __syncwarp();
                    return true;
                };
                if (!(ok = mma_wait(bQ, i & 1))) break;
                // the scores run NBUF - 1 of the tile's key blocks ahead of the P V products (KEYS: every other one of the list is)
                for (int j = 0; ok && j < AHEAD && j <= n_u; ++j) ok = k_step(j);
                for (int j = 0; ok && j < n_u; ++j) {
                    // S(n + NBUF - 1) reuses the buffer of P(n - 1); the MMAs of the issuing thread execute in issue
                    // order, so it is written only after P(n - 1) V has read it
                    if (j + AHEAD <= n_u && !(ok = k_step(j + AHEAD))) break;          // group j + 1 brings V(j)
                    const uint32_t s = (W0 + j) % VS;
                    const bool use = u.ent[j] & tile_bits;
                    if (use && !(ok = (mma_wait(bPFt + 8 * (n_pv % NBUF), (n_pv / NBUF) & 1)))) break;
                    if (use) {
                        tc_fence_after();
                        const uint32_t tP = tbase + 64 * (n_pv % NBUF);
                        const uint32_t vb = sV + s * C::KV_BYTES;
                        if (leader) {
                            // the first product of a quad overwrites O: that its P is there tells that every softmax
                            // warp of the tile has read the O of the quad before
    #pragma unroll
                            for (int ks = 0; ks < 4; ++ks)
                                mma_ts(tO, tP + ks * 8, smem_desc_sw128(vb + ks * 2048, BLK_BYTES, 1024), idesc_pv,
                                       (n_pv > n_pv0 || ks > 0) ? 1u : 0u);
                            tc_commit(bVE + 8 * s);
                            // pv_done: two barriers per tile, for the even and the odd blocks.  The softmax warps run up
                            // to NBUF - 1 <= 2 blocks ahead of these products, and the parity of one barrier taking every
                            // block could not tell "block n - 1 is done" from "block n - 3 is done"; with two, the one the
                            // rescale path waits on (block n - 1's) can only be one phase behind, because S(n) exists only
                            // once the product of block n - NBUF is over.  The epilogue may lag, so it has its own barrier.
                            tc_commit(bPV + 16 * t + 8 * (n_pv & 1));
                        }
                        ++n_pv;
                    } else if (leader) {
                        mbar_arrive(bVE + 8 * s);
                    }
                    if (!SOLO) __syncwarp();
                }
                if (!ok) break;
                if (leader) {
                    // only where the tile has blocks: the next phase then needs the softmax warps' P, and they have
                    // waited for this one by that time (a tile with nothing to do could complete two phases at once)
                    if (n_pv > n_pv0) tc_commit(bOD + 8 * t);
                    mbar_arrive(bUE + 8 * (i & 1));
                }
                if (!SOLO) __syncwarp();
                G0 += n_u + 1;
                W0 += n_u;
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ softmax / correction / epilogue
        // Sixteen warps, four per SM sub-partition, so that while one waits on a barrier or on tensor memory
        // the others keep the exponential unit busy.  Warp w works on tile (w >> 2) & 1, on the 16 rows
        // 32 (w & 3) + 16 (w >> 3) .. + 15 of it, with the 16x256b fragment layout: a thread owns two rows
        // (r_lo = lane / 4 and r_lo + 8 of the sixteen) and, of every group of eight score columns, the pair
        // 2 (lane % 4), + 1 -- 32 scores per key block.  The four threads of a quad share their rows' maximum
        // with two shuffles, and only when some row of the warp may have grown.
        if (SPLIT || KEYS) reg_inc<SOFTMAX_REGS>();
        const int t = (warp >> 2) & 1, wl = warp & 3, hf = warp >> 3;
        const int a = 2 * t + (wl >> 1);               // query block of the quad
        const uint32_t tile_bits = 3u << (2 * t), act_bit = 1u << a;
        const int cg = lane & 3;                        // column pair within a group of eight
        const int row_lo = wl * 32 + hf * 16 + (lane >> 2);
        const uint32_t lane_addr = tmem_base + ((uint32_t)(wl * 32 + hf * 16) << 16) + t * TILE_COLS;
        const uint32_t tO = lane_addr + O_COL;
        const uint32_t bSFt = bSF + 24 * t, bPFt = bPF + 24 * t, bPVt = bPV + 16 * t;
        const float c2 = prm.scale_log2;
        float* const ref = &ctl->nm[warp][lane >> 2];  // of the thread's rows: a thread of each quad writes it, all of them read it
        const int tail_valid = N - (nb - 1) * 64;      // valid tokens of the last block (1..64)
        int n = 0;                                     // blocks of this tile so far, in all quads
        uint32_t n_o = 0;                              // quads so far in which the tile had blocks
        bool ok = true;
        for (uint32_t i = 0;; ++i) {
        const Quad& u = ctl->quad[i & 1];
        if (!(ok = wait_warp(bUF + 8 * (i & 1), (i >> 1) & 1))) break;
        const int n_u = u.n_u;
        if (n_u < 0) break;
        float nm_lo = INFINITY, nm_hi = INFINITY;      // reference maxima of the two rows, times -c2
        float l0 = 0.f, l1 = 0.f, l2 = 0.f, l3 = 0.f;  // partial row sums: (l0, l1) first row, (l2, l3) second row
        uint32_t r[32];
        const int n0 = n;
        if (SPLIT && cg == 0) ref[0] = ref[8] = INFINITY;
        bool seeded = false;                           // the rows' reference maxima have been set (warp-uniform: a warp's rows share a query block)
        // A wait that runs out sets the abort flag; nothing up to the end of a quad depends on a wait's result, so no vote is
        // taken on the way, and the flag is looked at every ABORT_EVERY key blocks only.
        for (int j0 = 0; j0 < n_u; j0 += ABORT_EVERY) {
        if (__any_sync(0xffffffffu, ctl->abort_flag)) break;
        const int j1 = min(j0 + ABORT_EVERY, n_u);
        for (int j = j0; j < j1; ++j) {
            const uint32_t e = u.ent[j];
            if (!(e & tile_bits)) continue;            // neither query block of the tile kept it
            const bool act = e & act_bit;
            const int buf = n % NBUF;
            const uint32_t tS = lane_addr + 64 * buf;
            wait(bSFt + 8 * buf, (n / NBUF) & 1);
            __syncwarp();
            tc_fence_after();
            uint32_t pk[16];
            if (act) {
                tmem_ld16x256_x8(tS, r);
                tc_wait_ld();
                if (e & ENT_TAIL) {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
#pragma unroll
                        for (int x = 0; x < 2; ++x)
                            if (8 * k + 2 * cg + x >= tail_valid) {       // -inf: outside the sequence
                                r[4 * k + x] = 0xff800000u;
                                r[4 * k + 2 + x] = 0xff800000u;
                            }
                }
                // One pass over the 32 scores gives P = 2^(S c2 - m c2) (packed to bf16) and the block's partial row
                // sums.  The pass runs with the reference maxima as they stand, so the exponentials do not wait for
                // this block's maximum, and it takes no maximum at all: a P above 2^8 shows in the partial sum that it
                // is part of (eight terms, none negative).  Only when a partial sum exceeds 2^8 (rare after a query
                // block's first key block) the rows' maxima are taken, O and l are rescaled and the pass is repeated.
                // Bound by issue slots and the exponential unit: against maxima in the pass, packed products, votes on
                // the waits and P stored after the vote below, dense attention of two images of 4429 tokens at D = 64
                // went from 325 to 303 us, three of 4608 at D = 128 from 596 to 585 us (bursts at full clocks).
                float b0, b1, b2, b3;
                if (!seeded) {
                    // the first block this query block keeps: take the rows' maxima before the pass instead of running
                    // the pass twice (from -inf every row "grows")
                    row_maxima(r, nm_lo, nm_hi);
                    nm_lo *= -c2; nm_hi *= -c2;
                    // a part may begin with a block whose scores are all -inf: no NaN (-inf - -inf) from them, the next ones count
                    if (SPLIT || KEYS) { nm_lo = fminf(nm_lo, LOWEST); nm_hi = fminf(nm_hi, LOWEST); }
                    seeded = true;
                    if (SPLIT && cg == 0) { ref[0] = nm_lo; ref[8] = nm_hi; }
                }
                for (;;) {
                    b0 = b1 = b2 = b3 = 0.f;
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        float x0, x1, x2, x3;
                        x0 = fmaf(__uint_as_float(r[4 * k]), c2, nm_lo); x1 = fmaf(__uint_as_float(r[4 * k + 1]), c2, nm_lo);
                        x2 = fmaf(__uint_as_float(r[4 * k + 2]), c2, nm_hi); x3 = fmaf(__uint_as_float(r[4 * k + 3]), c2, nm_hi);
                        x0 = ex2(x0); x1 = ex2(x1); x2 = ex2(x2); x3 = ex2(x3);
                        add2(b0, b1, x0, x1);
                        add2(b2, b3, x2, x3);
                        pk[2 * k] = pack_bf16(x0, x1);
                        pk[2 * k + 1] = pack_bf16(x2, x3);
                    }
                    // P goes out before the vote on it is in, so that the two overlap; a repeated pass stores again before
                    // anything is told that P is there
                    tmem_st16x128_x8(tS, pk);
                    // if any thread of the warp sees growth, the quads combine their maxima and decide row by row
                    if (!__any_sync(0xffffffffu, max3(b0, b1, fmaxf(b2, b3)) > GROWN_SUM)) break;
                    {
                        float mx_lo, mx_hi;
                        row_maxima(r, mx_lo, mx_hi);
                        mx_lo *= -c2; mx_hi *= -c2;
                        const bool g_lo = nm_lo - mx_lo > GROWN_LOG2, g_hi = nm_hi - mx_hi > GROWN_LOG2;
                        // No row moves: done.  (Eight smaller P made the sum; or scores beyond 2^27 or so leave more than
                        // 2^8 of P to the rounding of their product with c2, which no maximum takes away.  A row moves at
                        // most once in a block.)
                        if (!__any_sync(0xffffffffu, g_lo || g_hi)) break;
                        tc_wait_st();                     // nothing else orders the repeated pass's store of P behind this one's
                        const bool f_lo = g_lo && nm_lo != INFINITY, f_hi = g_hi && nm_hi != INFINITY;   // not so where -inf was all it had
                        if (__any_sync(0xffffffffu, f_lo || f_hi)) {
                            // O must be at rest: wait for P(n-1) V, which by the issue order of the products also
                            // tells that every earlier one is done
                            wait(bPVt + 8 * ((n - 1) & 1), ((n - 1) >> 1) & 1);
                            __syncwarp();
                            tc_fence_after();
                            const float a_lo = f_lo ? ex2(mx_lo - nm_lo) : 1.f, a_hi = f_hi ? ex2(mx_hi - nm_hi) : 1.f;
                            l0 *= a_lo; l1 *= a_lo; l2 *= a_hi; l3 *= a_hi;
                            uint32_t o[16];
#pragma unroll
                            for (int ch = 0; ch < D / 32; ++ch) {
                                tmem_ld16x256_x4(tO + ch * 32, o);
                                tc_wait_ld();
#pragma unroll
                                for (int e = 0; e < 16; ++e)
                                    o[e] = __float_as_uint(__uint_as_float(o[e]) * ((e & 2) ? a_hi : a_lo));
                                tmem_st16x256_x4(tO + ch * 32, o);
                            }
                        }
                        if (g_lo) nm_lo = mx_lo;
                        if (g_hi) nm_hi = mx_hi;
                        if (SPLIT && cg == 0) { ref[0] = nm_lo; ref[8] = nm_hi; }
                    }
                }
                l0 += b0; l1 += b1; l2 += b2; l3 += b3;
            } else {
#pragma unroll
                for (int e = 0; e < 16; ++e) pk[e] = 0u;
                tmem_st16x128_x8(tS, pk);
            }
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bPFt + 8 * buf);
            ++n;
        }
        }
        if (n > n0) wait(bOD + 8 * t, n_o++ & 1);
        // where the other tile has blocks; else there is Q alone, which no product has waited for
        if (KEYS) wait(n_u > 1 - t ? bOD + 8 * (1 - t) : bQ, 0);
        if (!(ok = __all_sync(0xffffffffu, !ctl->abort_flag))) break;
        // epilogue: O / l -> bf16 -> 16 bytes a lane, four lanes a 64-byte piece of a row
        if (KEYS) {
            // No product and no copy is under way any more: what the other tile finishes -- O, not divided by the row sums, of half of
            // the channels, the sums and the reference maxima -- goes to it through the memory of Q, K and V.
            tc_fence_after();
            constexpr int HALF = D / 64, LEFT = (4 * HALF + 1) * 32;     // pieces of 32 channels; float4 that a warp hands on
            float4* const mine = reinterpret_cast<float4*>(smem) + warp * LEFT + lane;
            const float4* const other = reinterpret_cast<const float4*>(smem) + (warp ^ 4) * LEFT + lane;
            float s_lo = l0 + l1, s_hi = l2 + l3;
            s_lo += __shfl_xor_sync(0xffffffffu, s_lo, 1);
            s_hi += __shfl_xor_sync(0xffffffffu, s_hi, 1);
            s_lo += __shfl_xor_sync(0xffffffffu, s_lo, 2);
            s_hi += __shfl_xor_sync(0xffffffffu, s_hi, 2);
            uint32_t o[16];
            auto load_o = [&](int ch) {
                if (n > n0) {
                    tmem_ld16x256_x4(tO + ch * 32, o);
                    tc_wait_ld();
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e) o[e] = 0u;
                }
            };
#pragma unroll
            for (int x = 0; x < HALF; ++x) {
                load_o((1 - t) * HALF + x);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    mine[32 * (4 * x + k)] = make_float4(__uint_as_float(o[4 * k]), __uint_as_float(o[4 * k + 1]), __uint_as_float(o[4 * k + 2]),
                                                         __uint_as_float(o[4 * k + 3]));
            }
            mine[32 * 4 * HALF] = make_float4(nm_lo, nm_hi, s_lo, s_hi);
            mbar_arrive(smem_u32(&ctl->handed[warp]));
            if (!(ok = wait_warp(smem_u32(&ctl->handed[warp ^ 4]), 0))) break;
            const float4 v = other[32 * 4 * HALF];
            // a tile in which a row kept nothing (no maximum) counts for nothing
            const float m_lo = fminf(nm_lo, v.x), m_hi = fminf(nm_hi, v.y);
            float a_lo = nm_lo == INFINITY ? 0.f : ex2(m_lo - nm_lo), a_hi = nm_hi == INFINITY ? 0.f : ex2(m_hi - nm_hi);
            float b_lo = v.x == INFINITY ? 0.f : ex2(m_lo - v.x), b_hi = v.y == INFINITY ? 0.f : ex2(m_hi - v.y);
            s_lo = fmaf(a_lo, s_lo, b_lo * v.z);
            s_hi = fmaf(a_hi, s_hi, b_hi * v.w);
            const float inv_lo = one_over(s_lo, m_lo), inv_hi = one_over(s_hi, m_hi);
            a_lo *= inv_lo; b_lo *= inv_lo; a_hi *= inv_hi; b_hi *= inv_hi;
            const int tok_lo = u.tok[a] + (row_lo & 63), tok_hi = tok_lo + 8;
            uint16_t* o_lo = out + (long long)u.b * g.stride_b + (long long)u.h * g.stride_h + (long long)tok_lo * g.stride_n + 8 * cg;
            uint16_t* o_hi = o_lo + 8 * g.stride_n;
#pragma unroll
            for (int x = 0; x < HALF; ++x) {
                const int ch = t * HALF + x;
                load_o(ch);
                uint32_t w_lo[4], w_hi[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float4 p = other[32 * (4 * x + k)];
                    w_lo[k] = pack_bf16(fmaf(__uint_as_float(o[4 * k]), a_lo, p.x * b_lo), fmaf(__uint_as_float(o[4 * k + 1]), a_lo, p.y * b_lo));
                    w_hi[k] = pack_bf16(fmaf(__uint_as_float(o[4 * k + 2]), a_hi, p.z * b_hi), fmaf(__uint_as_float(o[4 * k + 3]), a_hi, p.w * b_hi));
                }
                const uint4 v_lo = quad_transpose(w_lo[0], w_lo[1], w_lo[2], w_lo[3], cg);
                const uint4 v_hi = quad_transpose(w_hi[0], w_hi[1], w_hi[2], w_hi[3], cg);
                if (tok_lo < N) *reinterpret_cast<uint4*>(o_lo + 32 * ch) = v_lo;
                if (tok_hi < N) *reinterpret_cast<uint4*>(o_hi + 32 * ch) = v_hi;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bUE + 8 * (i & 1));
        } else if (SPLIT && u.parts > 1) {
            // a part of the list: O as it is, the row sums and the reference maxima go to memory
            tc_fence_after();
            if (u.tok[a] < N) {                        // the same in every part of the quad
                uint32_t at = warp * (PARTIAL_F4<D> * 32) + lane;
                float4* mine = prm.parts.partial + (size_t)(u.store + u.part) * (SOFTMAX_WARPS * PARTIAL_F4<D> * 32) + at;
                uint32_t o[16];
#pragma unroll 1
                for (int ch = 0; ch < D / 32; ++ch) {
                    if (n > n0) {
                        tmem_ld16x256_x4(tO + ch * 32, o);
                        tc_wait_ld();
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; ++e) o[e] = 0u;
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        __stcg(mine + 32 * (4 * ch + k), make_float4(__uint_as_float(o[4 * k]), __uint_as_float(o[4 * k + 1]),
                                                                     __uint_as_float(o[4 * k + 2]), __uint_as_float(o[4 * k + 3])));
                }
                __syncwarp();                          // for `ref`
                float s_lo = l0 + l1, s_hi = l2 + l3;
                s_lo += __shfl_xor_sync(0xffffffffu, s_lo, 1);
                s_hi += __shfl_xor_sync(0xffffffffu, s_hi, 1);
                s_lo += __shfl_xor_sync(0xffffffffu, s_lo, 2);
                s_hi += __shfl_xor_sync(0xffffffffu, s_hi, 2);
                __stcg(mine + 32 * (PARTIAL_F4<D> - 1), make_float4(ref[0], ref[8], s_lo, s_hi));
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bUE + 8 * (i & 1));
        } else {
            tc_fence_after();
            float s_lo = l0 + l1, s_hi = l2 + l3;      // the quad's four partial sums make the row sum
            s_lo += __shfl_xor_sync(0xffffffffu, s_lo, 1);
            s_hi += __shfl_xor_sync(0xffffffffu, s_hi, 1);
            s_lo += __shfl_xor_sync(0xffffffffu, s_lo, 2);
            s_hi += __shfl_xor_sync(0xffffffffu, s_hi, 2);
            // (in builds without LOWEST the O of a row of scores of -inf is not a number as it is)
            const float inv_lo = one_over(s_lo, SPLIT ? nm_lo : 0.f), inv_hi = one_over(s_hi, SPLIT ? nm_hi : 0.f);
            const int tok_lo = u.tok[a] + (row_lo & 63), tok_hi = tok_lo + 8;
            uint16_t* o_lo = out + (long long)u.b * g.stride_b + (long long)u.h * g.stride_h + (long long)tok_lo * g.stride_n + 8 * cg;
            uint16_t* o_hi = o_lo + 8 * g.stride_n;
            uint32_t o[16];
#pragma unroll
            for (int ch = 0; ch < D / 32; ++ch) {
                if (n > n0) {
                    tmem_ld16x256_x4(tO + ch * 32, o);
                    tc_wait_ld();
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e) o[e] = 0u;
                }
                uint32_t w_lo[4], w_hi[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {          // channels 32 ch + 8 k + 2 cg, + 1
                    w_lo[k] = pack_bf16(__uint_as_float(o[4 * k]) * inv_lo, __uint_as_float(o[4 * k + 1]) * inv_lo);
                    w_hi[k] = pack_bf16(__uint_as_float(o[4 * k + 2]) * inv_hi, __uint_as_float(o[4 * k + 3]) * inv_hi);
                }
                const uint4 v_lo = quad_transpose(w_lo[0], w_lo[1], w_lo[2], w_lo[3], cg);
                const uint4 v_hi = quad_transpose(w_hi[0], w_hi[1], w_hi[2], w_hi[3], cg);
                if (tok_lo < N) *reinterpret_cast<uint4*>(o_lo + 32 * ch) = v_lo;
                if (tok_hi < N) *reinterpret_cast<uint4*>(o_hi + 32 * ch) = v_hi;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bUE + 8 * (i & 1));
        }
        }
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (warp >= MMA_WARP0 && warp < MMA_WARP0 + 2) {
        if (ctl->abort_flag) {
            // make sure no UMMA of this warp is still in flight before the TMEM columns are released
            const uint32_t bD = smem_u32(&ctl->drain[warp - MMA_WARP0]);
            if (elect_one()) {
                tc_commit(bD);
                mbar_wait(bD, 0, 1u << 20);
            }
            __syncwarp();
        }
    }
    __syncthreads();
    if (warp == MMA_WARP0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

// The results of the quads whose lists were worked on in parts: what the parts have left, added up in the order of the list.
// A warp does a softmax warp's sixteen rows, 32 channels of them, with every part's loads in flight at once: bound by two round
// trips to the L2.  The lanes hold what the attention kernel's lanes held.
template <int D>
__global__ void __launch_bounds__(128) add_parts_kernel(uint16_t* __restrict__ out, const TensorGeom g, const __grid_constant__ ImgList imgs,
                                                        int n_dense, const DevPlan* plan, const AttnParts ap) {
    constexpr int CH = D / 32;
    constexpr size_t part_f4 = (size_t)SOFTMAX_WARPS * PARTIAL_F4<D> * 32;
    const int lane = threadIdx.x % 32, cg = lane & 3;
    grid_dependency_wait();
    grid_dependency_launch();
    const int item = blockIdx.x * 4 + threadIdx.x / 32, warp = item / CH % SOFTMAX_WARPS, ch = item % CH;
    const int nq = (g.nb + 3) >> 2, ntq = min(nq, (g.n_text_blocks + 3) >> 2), nl = nq - ntq;
    const int nd = plan ? __ldcg(&plan->n_dense) : n_dense, ns = (plan ? __ldcg(&plan->all.n) : imgs.n) - nd;
    const int qd = ap.dense > 1 ? nd * g.H * nq : 0, qt = ap.text > 1 ? ns * g.H * ntq : 0, ql = ap.light > 1 ? ns * g.H * nl : 0;
    int x = item / CH / SOFTMAX_WARPS, p, h, quad, parts, store;
    if (x < qd) {
        parts = ap.dense; store = x * parts;
        p = x / (g.H * nq); x -= p * g.H * nq;
        h = x / nq; quad = x - h * nq;
    } else if (x < qd + qt) {
        x -= qd;
        parts = ap.text; store = qd * ap.dense + x * parts;
        p = x / (g.H * ntq); x -= p * g.H * ntq; p += nd;
        h = x / ntq; quad = x - h * ntq;
    } else {
        x -= qd + qt;
        if (x >= ql) return;
        parts = ap.light; store = qd * ap.dense + qt * ap.text + x * parts;
        p = x / (g.H * nl); x -= p * g.H * nl; p += nd;
        h = x / nl; quad = ntq + x - h * nl;
    }
    const int tok_lo = 64 * quad_block(g, quad, 2 * ((warp >> 2) & 1) + ((warp & 3) >> 1)) + (warp & 1) * 32 + (warp >> 3) * 16 + (lane >> 2);
    const int tok_hi = tok_lo + 8;
    if (tok_lo - (lane >> 2) >= g.N) return;             // nothing was left for rows past the end
    const int b = plan ? __ldcg(&plan->all.batch[p]) : imgs.batch[p];
    const int given_up = __ldcg(ap.given_up);
    const float4* base = ap.partial + (size_t)store * part_f4 + (size_t)warp * PARTIAL_F4<D> * 32 + lane;
    float4 v[MAX_PARTS], x4[MAX_PARTS][4];
#pragma unroll
    for (int i = 0; i < MAX_PARTS; ++i) {
        v[i] = make_float4(INFINITY, INFINITY, 0.f, 0.f);
        if (i < parts) {
            v[i] = __ldcg(base + i * part_f4 + 32 * (PARTIAL_F4<D> - 1));
#pragma unroll
            for (int k = 0; k < 4; ++k) x4[i][k] = __ldcg(base + i * part_f4 + 32 * (4 * ch + k));
        }
    }
    float m_lo = INFINITY, m_hi = INFINITY, s_lo = 0.f, s_hi = 0.f;      // maxima times -c2
#pragma unroll
    for (int i = 0; i < MAX_PARTS; ++i) {
        m_lo = fminf(m_lo, v[i].x);
        m_hi = fminf(m_hi, v[i].y);
    }
    float f[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) f[e] = 0.f;
#pragma unroll
    for (int i = 0; i < MAX_PARTS; ++i)
        if (i < parts) {
            // a part in which a row kept nothing (no maximum) counts for nothing
            const float w_lo = v[i].x == INFINITY ? 0.f : ex2(m_lo - v[i].x), w_hi = v[i].y == INFINITY ? 0.f : ex2(m_hi - v[i].y);
            s_lo = fmaf(w_lo, v[i].z, s_lo);
            s_hi = fmaf(w_hi, v[i].w, s_hi);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                f[4 * k] = fmaf(w_lo, x4[i][k].x, f[4 * k]); f[4 * k + 1] = fmaf(w_lo, x4[i][k].y, f[4 * k + 1]);
                f[4 * k + 2] = fmaf(w_hi, x4[i][k].z, f[4 * k + 2]); f[4 * k + 3] = fmaf(w_hi, x4[i][k].w, f[4 * k + 3]);
            }
        }
    const float inv_lo = one_over(s_lo, m_lo), inv_hi = one_over(s_hi, m_hi);
    uint32_t a_lo[4], a_hi[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        a_lo[k] = pack_bf16(f[4 * k] * inv_lo, f[4 * k + 1] * inv_lo);
        a_hi[k] = pack_bf16(f[4 * k + 2] * inv_hi, f[4 * k + 3] * inv_hi);
    }
    const uint4 o_lo = quad_transpose(a_lo[0], a_lo[1], a_lo[2], a_lo[3], cg);
    const uint4 o_hi = quad_transpose(a_hi[0], a_hi[1], a_hi[2], a_hi[3], cg);
    uint16_t* o = out + (long long)b * g.stride_b + (long long)(g.h0 + h) * g.stride_h + (long long)tok_lo * g.stride_n + 8 * cg + 32 * ch;
    if (given_up) return;                                // parts of an earlier launch, or of none, may be among these
    if (tok_lo < g.N) *reinterpret_cast<uint4*>(o) = o_lo;
    if (tok_hi < g.N) *reinterpret_cast<uint4*>(o + 8 * g.stride_n) = o_hi;
}

bool g_attr_set = false;

}  // namespace

cudaError_t attention_static_init() {
    const auto set = [](auto... kernels) {
        cudaError_t e = cudaSuccess;
        const int smem[] = {(int)attn_smem_bytes<128>(), (int)attn_smem_bytes<64>()};      // the builds come in pairs
        int i = 0;
        ((e = e != cudaSuccess ? e : cudaFuncSetAttribute(kernels, cudaFuncAttributeMaxDynamicSharedMemorySize, smem[i++ % 2])), ...);
        return e;
    };
    const cudaError_t e = set(attn_kernel<128>, attn_kernel<64>, attn_kernel<128, false, true>, attn_kernel<64, false, true>,
                              attn_kernel<128, false, false, true>, attn_kernel<64, false, false, true>,
                              attn_kernel<128, false, false, false, true>, attn_kernel<64, false, false, false, true>,
                              attn_kernel<128, true>, attn_kernel<64, true>, attn_kernel<128, true, true>, attn_kernel<64, true, true>,
                              attn_kernel<128, false, false, false, false, true>, attn_kernel<64, false, false, false, false, true>,
                              attn_kernel<128, true, false, false, false, true>, attn_kernel<64, true, false, false, false, true>);
    if (e != cudaSuccess) return e;
    // the warps that take registers wait for them: a build that is launched with fewer would wait for good
    for (const void* kernel : {(const void*)attn_kernel<128, false, true>, (const void*)attn_kernel<64, false, true>,
                               (const void*)attn_kernel<128, true, true>, (const void*)attn_kernel<64, true, true>,
                               (const void*)attn_kernel<128, false, false, false, false, true>,
                               (const void*)attn_kernel<64, false, false, false, false, true>,
                               (const void*)attn_kernel<128, true, false, false, false, true>,
                               (const void*)attn_kernel<64, true, false, false, false, true>}) {
        cudaFuncAttributes attr;
        const cudaError_t r = cudaFuncGetAttributes(&attr, kernel);
        if (r != cudaSuccess) return r;
        if (attr.numRegs * NTHREADS < 32 * (SOFTMAX_WARPS * SOFTMAX_REGS + 4 * LIGHT_REGS)) return cudaErrorInvalidKernelImage;
    }
    g_attr_set = true;
    return cudaSuccess;
}

// When the last SM is through with the units of work of three classes, n[i] of t[i] us, handed out in this order as SMs are free.
static double units_time(const int (&n)[3], const double (&t)[3]) {
    struct Group { double at; int sms; } group[5] = {{0.0, SM_COUNT}};   // SMs by when they are free
    int groups = 1;
    double end = 0.0;
    for (int i = 0; i < 3; ++i)
        for (int left = n[i]; left > 0;) {
            int g = 0;
            for (int j = 1; j < groups; ++j)
                if (group[j].at < group[g].at) g = j;
            if (left < group[g].sms) {                   // some of the group's SMs stay free
                group[groups++] = {group[g].at, group[g].sms - left};
                group[g].sms = left;
            }
            left -= group[g].sms;
            group[g].at += t[i];
            end = std::max(end, group[g].at);
        }
    return end;
}

// Units of work whose results are left in memory, at most, in a launch of such a context.
static size_t left_units(const TensorGeom& g, int n_img, const AttnParts& parts) {
    const int nq = (g.nb + 3) / 4, ntq = std::min(nq, (g.n_text_blocks + 3) / 4);
    const int d = parts.dense > 1 ? nq * parts.dense : 0;
    const int s = (parts.text > 1 ? ntq * parts.text : 0) + (parts.light > 1 ? (nq - ntq) * parts.light : 0);
    return (size_t)std::max(d, s) * g.H * n_img;
}

// Into how many parts the attention of a context of up to n_img images cuts the lists of its quads.  What an image gets must
// not depend on the launch it is in, so this is the context's and the image's own: quads of a dense image, of a sparse one's
// text rows (which keep every block), and the others.  Of all cuts, the one with the best times over these launches: every image
// dense; all sparse, the other quads' unions holding 0.3, 0.6 or 0.9 of the blocks; half of them dense; half of them
// attending at all.  It must be 10 % better than whole lists in the mean and in none of them worse by more than 2 %.  The
// times: 0.72 and 0.84 us a key block (D = 64, 128), 0.56 and 0.66 us where a tile has its SM to itself, 1 us a unit; a
// part's write 1 and 2 us, add_parts_kernel 3.5 us and what was left at 4.5 TB/s (1.5 us where it finds nothing).  Short rows
// (MIN_CUT) are left whole: their calls wait for the host, whom one more launch costs 2 us.
// Attention alone, us, whole lists / parts: 18 quads of 72 blocks 46.8 / 16.7 (D = 64, eight parts), 54.1 / 20.9 (D = 128);
// 36 quads of 72 47.3 / 23.2, 55.0 / 30.0 (four); 18 of 33 24.9 / 13.6 (eight), 28.6 / 16.2 (four); 72 of 72 48.6 / 36.7,
// 56.3 / 47.1 (two); 60 of 12 13.7 / 15.7, 15.5 / 21.0 (two).  Steps: 46 quads of 92 blocks at ratio 0.25, D = 64 61.6 / 31.8
// (text rows in five, the others in three); 132 of 264 at ratio 0.2, D = 128 231 / 135 (text rows in four); 198 of 262 at ratios
// 1, 0.5 and 0.2, D = 64 359, 289 and 196 / 289, 237 and 148 (in two, text rows in three).
// Where lists stay whole and every tile has an SM to itself in the largest launch, the two tiles of the SM take its blocks by turns.  The model has
// the times of a tile alone for such lists, not the 0.42 and 0.60 us a block that they take by turns: with these it would leave whole the lists of 0.7 % of
// the contexts drawn at random that it cuts now (54 quads of 36 blocks, D = 64).
AttnParts attention_parts(const TensorGeom& g, int n_img) {
    AttnParts best;
    const int nq = (g.nb + 3) / 4, ntq = std::min(nq, (g.n_text_blocks + 3) / 4);
    best.keys = 2ll * nq * g.H * n_img <= SM_COUNT && g.nb >= (g.D == 128 ? KEYS_FROM_128 : KEYS_FROM_64);
    if (g.nb < MIN_CUT || (long long)nq * g.H * n_img > MAX_CUT) return best;
    const bool wide = g.D == 128;
    auto time = [&](int dense, int sparse, double held, const AttnParts& p) {
        const int quads[3] = {nq * g.H * dense, ntq * g.H * sparse, (nq - ntq) * g.H * sparse}, parts[3] = {p.dense, p.text, p.light};
        const double blocks[3] = {(double)g.nb, (double)g.nb, held * g.nb};
        int n[3], units = 0, left = 0;
        for (int i = 0; i < 3; ++i) {
            units += n[i] = quads[i] * parts[i];
            if (parts[i] > 1) left += n[i];
        }
        const bool one = 2 * units <= SM_COUNT;
        double t[3];
        for (int i = 0; i < 3; ++i) {
            if (one) n[i] *= 2;
            t[i] = blocks[i] / parts[i] * (wide ? (one ? 0.66 : 0.84) : (one ? 0.56 : 0.72)) + 1.0 + (parts[i] > 1 ? g.D / 64 : 0);
        }
        return units_time(n, t) + 5.0 + (left > 0 ? 3.5 + left * (1.1e-3 * g.D / 4.5) : p.any() ? 1.5 : 0.0);
    };
    const int half = n_img / 2;
    const struct { int dense, sparse; double held; } launches[] = {
        {n_img, 0, 1.0}, {0, n_img, 0.3}, {0, n_img, 0.6}, {0, n_img, 0.9}, {half, n_img - half, 0.3}, {half, n_img - half, 0.6},
        {n_img - half, 0, 1.0}, {0, n_img - half, 0.6}};
    constexpr int N = sizeof launches / sizeof launches[0];
    double whole[N], least = 0.9 * N;
    for (int i = 0; i < N; ++i) whole[i] = time(launches[i].dense, launches[i].sparse, launches[i].held, AttnParts());
    for (int pd = 1; pd <= MAX_PARTS; ++pd)
        for (int pl = 1; pl <= MAX_PARTS; ++pl)
            for (int pt = ntq ? pl : 1; pt <= (ntq ? MAX_PARTS : 1); ++pt) {
                AttnParts p;
                p.dense = pd;
                p.text = pt;
                p.light = pl;
                if (!p.any() || left_units(g, n_img, p) > MAX_LEFT) continue;
                double sum = 0.0, most = 0.0;
                for (int i = 0; i < N && most <= 1.02 && sum < least; ++i) {
                    const double x = time(launches[i].dense, launches[i].sparse, launches[i].held, p) / whole[i];
                    sum += x;
                    most = std::max(most, x);
                }
                if (sum < least && most <= 1.02) {
                    least = sum;
                    best = p;
                }
            }
    return best;
}
size_t attention_partial_bytes(const TensorGeom& g, int n_img, const AttnParts& parts) {
    return left_units(g, n_img, parts) * SOFTMAX_WARPS * 32 * sizeof(float4) * (g.D == 128 ? PARTIAL_F4<128> : PARTIAL_F4<64>);
}
cudaError_t launch_attention(const CUtensorMap& tmq, const CUtensorMap& tmk, const CUtensorMap& tmv,
                             void* out,
                             const TensorGeom& g, const ImgList& imgs, const int32_t* kept_idx,
                             const int32_t* kept_cnt, const uint64_t* bitmask, float softmax_scale, int* status,
                             cudaStream_t s, const DevPlan* plan, int n_cap, int inject_stop_group, bool wait_first,
                             const AttnParts* parts, int64_t* launches, const QuadOrder& order) {
    if (!g_attr_set) {
        cudaError_t e = attention_static_init();
        if (e != cudaSuccess) return e;
    }
    AttnParams prm;
    prm.g = g;
    prm.imgs = imgs;
    prm.kept_idx = kept_idx;
    prm.kept_cnt = kept_cnt;
    prm.bitmask32 = reinterpret_cast<const uint32_t*>(bitmask);
    prm.words32 = 2 * ((g.nb + 63) / 64);
    prm.status = status;
    prm.scale_log2 = softmax_scale * 1.4426950408889634f;
    int n_dense = 0;
    while (n_dense < imgs.n && (imgs.slot[n_dense] < 0 || kept_idx == nullptr)) ++n_dense;
    prm.n_dense = n_dense;
    prm.plan = plan;
    prm.order = order;
    prm.wait_first = wait_first;
    {
        const int quads = (g.nb + 3) / 4, text = std::min(quads, (g.n_text_blocks + 3) / 4), pure = g.n_text_blocks / 4;
        prm.div_all = divider(quads);
        prm.div_text = divider(text);
        prm.div_pure = divider(pure);
        prm.div_mixed = divider(text - pure);
        prm.div_light = divider(quads - text);
        prm.div_heads = divider(g.H);
    }
    prm.stop_group = inject_stop_group;
    const int n_img = plan ? n_cap : imgs.n, pairs = g.H * n_img, nq = (g.nb + 3) / 4, ntq = std::min(nq, (g.n_text_blocks + 3) / 4);
    int left = 0;                              // quads whose lists are worked on in parts, at most
    if (parts) {
        const int d = parts->dense > 1 ? nq : 0, t = (parts->text > 1 ? ntq : 0) + (parts->light > 1 ? nq - ntq : 0);
        left = plan ? pairs * std::max(d, t) : g.H * (n_dense * d + (imgs.n - n_dense) * t);
        if (left > 0) prm.parts = *parts;
    }
    const int units = plan ? std::max(attention_units(g, prm.parts, n_img, n_img), attention_units(g, prm.parts, n_img, 0))
                           : attention_units(g, prm.parts, n_img, n_dense);
    // halves: up to as many thread blocks as SMs.  Where a plan may hold fewer units than the largest launch, it may halve them.
    dim3 grid(2 * units <= SM_COUNT ? 2 * units : plan ? std::max(units, SM_COUNT) : units, 1, 1);
    if (left > 0) {
        const auto kernel = inject_stop_group >= 0 ? (g.D == 128 ? attn_kernel<128, true, true> : attn_kernel<64, true, true>)
                                                   : (g.D == 128 ? attn_kernel<128, false, true> : attn_kernel<64, false, true>);
        cudaError_t e = launch_kernel(kernel, grid, dim3(NTHREADS), g.D == 128 ? attn_smem_bytes<128>() : attn_smem_bytes<64>(), s, tmq, tmk, tmv,
                                      static_cast<uint16_t*>(out), prm);
        if (e != cudaSuccess) return e;
        *launches += 1;
        return launch_kernel(g.D == 128 ? add_parts_kernel<128> : add_parts_kernel<64>, dim3(left * SOFTMAX_WARPS * (g.D / 32) / 4), dim3(128), 0, s,
                             static_cast<uint16_t*>(out), g, imgs, n_dense, plan, prm.parts);
    } else if (inject_stop_group >= 0) {
        const bool keys = parts && parts->keys;
        const auto kernel = g.D == 128 ? (keys ? attn_kernel<128, true, false, false, false, true> : attn_kernel<128, true>)
                                       : (keys ? attn_kernel<64, true, false, false, false, true> : attn_kernel<64, true>);
        kernel<<<grid, NTHREADS, g.D == 128 ? attn_smem_bytes<128>() : attn_smem_bytes<64>(), s>>>(tmq, tmk, tmv, static_cast<uint16_t*>(out), prm);
    } else {
        const bool masks = bitmask || (!kept_idx && g.D == 128);         // see MASKS
        if (parts && parts->keys)
            return launch_kernel(g.D == 128 ? attn_kernel<128, false, false, false, false, true> : attn_kernel<64, false, false, false, false, true>,
                                 grid, dim3(NTHREADS), g.D == 128 ? attn_smem_bytes<128>() : attn_smem_bytes<64>(), s, tmq, tmk, tmv,
                                 static_cast<uint16_t*>(out), prm);
        return launch_kernel(order.cls ? (g.D == 128 ? attn_kernel<128, false, false, true> : attn_kernel<64, false, false, true>)
                             : masks ? (g.D == 128 ? attn_kernel<128, false, false, false, true> : attn_kernel<64, false, false, false, true>)
                                       : (g.D == 128 ? attn_kernel<128> : attn_kernel<64>),
                             grid, dim3(NTHREADS), g.D == 128 ? attn_smem_bytes<128>() : attn_smem_bytes<64>(), s, tmq, tmk, tmv,
                             static_cast<uint16_t*>(out), prm);
    }
    return cudaGetLastError();
}
