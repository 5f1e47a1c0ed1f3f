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
#include <type_traits>

#include "common.cuh"

namespace {

constexpr int WARPS = 4;

// Order-preserving key of a score: unsigned integers with the same order as the floats (-0 and +0 made equal), at least
// 2^23 for any finite one.  Forced blocks and padding get key 0, below every trial prefix.
__device__ __forceinline__ uint32_t score_key(float x) {
    uint32_t u = __float_as_uint(x);
    if (u == 0x80000000u) u = 0u;
    return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}

// Bits of the candidates' keys (non-zero ones): the number of low bits in which two of them differ, and what the bits
// above are in all of them.
template <int IPL>
__device__ __forceinline__ int differing_bits(const uint32_t (&u)[IPL], uint32_t& common) {
    uint32_t k_and = 0xffffffffu, k_or = 0u;
#pragma unroll
    for (int x = 0; x < IPL; ++x)
        if (u[x]) { k_and &= u[x]; k_or |= u[x]; }
    k_and = __reduce_and_sync(0xffffffffu, k_and);
    k_or = __reduce_or_sync(0xffffffffu, k_or);
    const uint32_t diff = k_and ^ k_or;
    const int top = diff ? 32 - __clz(diff) : 0;
    common = top >= 32 ? 0u : (k_or & ~((1u << top) - 1u));
    return top;
}

// HK = NoHeadKeep: one keep count per image.  HK = HeadKeep: one per (image, head), passed by value.
// HK = RowKeep: one per row, read from device memory.
// ORDER: the quads' places in the attention's order come out too (see QuadOrder); imgs.slot then holds an image's place among the
// sparse ones in the attention's list.
template <typename HK, int IPL, bool ORDER>
__global__ void __launch_bounds__(WARPS * 32) select_kernel(const float* scores, TensorGeom g,
                                                            ImgList imgs, uint32_t* __restrict__ bitmask32,
                                                            int32_t* __restrict__ kept_idx,
                                                            int32_t* __restrict__ kept_cnt, int words32,
                                                            const DevPlan* plan, const QuadOrder order, const HK hk) {
    __shared__ uint32_t kept[ORDER ? WARPS : 1][ORDER ? IPL : 1];        // the thread block's rows: the four query blocks of a quad
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int nb = g.nb, ntb = g.n_text_blocks;
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
        const bool text_row = i < ntb;
        const int n_free = max(nb - ntb - ((i >= ntb) ? 1 : 0), 0);
        const bool select = !text_row && k > 0 && k < n_free;
        uint32_t u[IPL];
#pragma unroll
        for (int x = 0; x < IPL; ++x) {
            const int j = 32 * x + lane;
            u[x] = 0u;
            if (select && j < nb && j >= ntb && j != i) u[x] = score_key(__ldcg(src + j));   // past the L1: see the wait above
        }
        uint32_t prefix = 0u;
        int want = 0;                                       // of the keys that equal `prefix`, how many are kept
        if (select) {
            int hi = differing_bits(u, prefix);             // the candidates that decide equal `prefix` from bit `hi` up
            int at_least = n_free, above = 0;               // candidates at or above `prefix`, and above those that decide
            while (hi > 0 && at_least > k) {
                const int lo = max(hi - 2, 0);
                const uint32_t d = 1u << lo, t1 = prefix + d, t2 = t1 + d, t3 = t2 + d;
                uint32_t c = 0u;                            // candidates at or above the three trials
                if (hi - lo == 2) {
#pragma unroll
                    for (int x = 0; x < IPL; ++x) c += (u[x] >= t1 ? 1u : 0u) + (u[x] >= t2 ? 1u << 10 : 0u) + (u[x] >= t3 ? 1u << 20 : 0u);
                    c = __reduce_add_sync(0xffffffffu, c);
                } else {
#pragma unroll
                    for (int x = 0; x < IPL; ++x) c += u[x] >= t1 ? 1u : 0u;
                    c = __reduce_add_sync(0xffffffffu, c) | ((uint32_t)above << 10) | ((uint32_t)above << 20);   // no digit 2 or 3
                }
                const int c1 = c & 1023u, c2 = (c >> 10) & 1023u, c3 = c >> 20;
                // the digit is the largest with k candidates or more at or above it
                if (c3 >= k) { prefix = t3; at_least = c3; }
                else if (c2 >= k) { prefix = t2; at_least = c2; above = c3; }
                else if (c1 >= k) { prefix = t1; at_least = c1; above = c2; }
                else above = c1;
                hi = lo;
            }
            want = at_least > k ? k - above : nb;           // exactly k at or above `prefix`: all of them
        }
        int32_t* out_idx = kept_idx + (long long)row * nb;
        uint32_t* out_bits = bitmask32 + (long long)row * words32;
        int total = 0, eq_seen = 0;
#pragma unroll
        for (int x = 0; x < IPL; ++x) {
            const int j = 32 * x + lane;
            if (32 * x >= nb) break;
            bool keep = false, eq = false;
            if (j < nb) {
                if (text_row || j < ntb || j == i) keep = true;
                else if (select) {
                    keep = u[x] > prefix;
                    eq = u[x] == prefix;
                } else keep = k >= n_free && k > 0;         // every free candidate, or none
            }
            // equal keys: the lowest block indices first, `want` of them in all
            const uint32_t beq = __ballot_sync(0xffffffffu, eq);
            if (eq && eq_seen + __popc(beq & ((1u << lane) - 1u)) < want) keep = true;
            eq_seen += __popc(beq);
            const uint32_t bal = __ballot_sync(0xffffffffu, keep);
            if (lane == 0) {
                out_bits[x] = bal;
                if constexpr (ORDER) kept[warp][x] = bal;
            }
            if (keep) out_idx[total + __popc(bal & ((1u << lane) - 1u))] = j;
            total += __popc(bal);
        }
        for (int c = (nb + 31) / 32 + lane; c < words32; c += 32) out_bits[c] = 0;   // odd 32-bit half of the last word
        for (int e = total + lane; e < nb; e += 32) out_idx[e] = -1;
        if (lane == 0) kept_cnt[row] = total;
    } else if (ORDER && lane < IPL) {
        kept[ORDER ? warp : 0][ORDER ? lane : 0] = 0u;
    }
    if constexpr (ORDER) {
        __syncthreads();
        const int nq = (nb + 3) >> 2, ntq = (ntb + 3) >> 2, quad = blockIdx.x;
        if (warp > 0 || quad < ntq) return;             // quads with text rows come earlier
        int rank = imgs.slot[p], n_sparse = imgs.n;
        if (plan) {
            n_sparse = __ldcg(&plan->sparse.n);
            const int n_all = __ldcg(&plan->all.n);
            auto here = [&](int at) { return at < n_all && __ldcg(&plan->all.slot[at]) == p; };
            const uint32_t lo = __ballot_sync(0xffffffffu, here(lane)), hi = __ballot_sync(0xffffffffu, here(32 + lane));
            rank = (lo ? __ffs(lo) - 1 : 31 + __ffs(hi)) - __ldcg(&plan->n_dense);
        }
        const int nl = nq - ntq;
        if ((rank * g.H + ph % g.H) * nl + quad - ntq < n_sparse * g.H * nl - ORDER_LAST) return;
        // the quad's time, in quarters of a key block of two tiles: one that only one tile uses takes three quarters
        int time = 0;
        if (32 * lane < nb) {
            const uint32_t t0 = kept[0][lane] | kept[1][lane], t1 = kept[2][lane] | kept[3][lane];
            time = 2 * __popc(t0 | t1) + __popc(t0) + __popc(t1);
        }
        time = __reduce_add_sync(0xffffffffu, time);
        if (lane == 0) {
            const int c = ORDER_CLASSES - 1 - time * (ORDER_CLASSES - 1) / (4 * nb);
            order.list[c * ORDER_LAST + atomicAdd(order.count + c, 1u)] = (rank * g.H + ph % g.H) * nq + quad;
        }
    }
}

// Cumulative-mass rule: one warp per row finds the smallest count k of best free candidates (score
// descending, index ascending) whose weights w = exp(scale * (S - row max)) sum to at least
// tau * (sum of all free weights).  No sort: the boundary candidate is found by descending the
// bits of the order-preserving keys, each round summing the weights of the candidates that match
// the trial prefix (a weighted radix select); candidates equal to the boundary key are then added
// one by one.  fp64 throughout, the precision in which the decision is defined.  Keys and weights are in registers, IPL
// of each a lane as above.  Bits that all candidates share decide nothing (a trial holds all of the mass or none of it),
// and a group of one candidate is the boundary whatever its lower bits are, so both are left out (with the selection
// after it: 25.6 -> 12.0 us for two images of 24 heads x 70 rows, 61 -> 36 us for one of 264).
constexpr int MASS_WARPS = 2;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int IPL>
__global__ void __launch_bounds__(MASS_WARPS * 32) mass_count_kernel(const float* scores, TensorGeom g, MassShare share,
                                                                     float scale, int32_t* __restrict__ row_keep) {
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int nb = g.nb, ntb = g.n_text_blocks;
    const int ph = blockIdx.y, p = ph / g.H, i = blockIdx.x * MASS_WARPS + warp;
    const int row = ph * nb + i;
    grid_dependency_wait();                                // for the scores
    grid_dependency_launch();
    if (i >= nb) return;
    const int n_free = (i < ntb) ? 0 : max(nb - ntb - 1, 0);
    const float tau = share.tau[p];
    if (n_free == 0 || tau >= 1.f) {                       // warp-uniform
        if (lane == 0) row_keep[row] = n_free;
        return;
    }
    const float* src = scores + (long long)row * nb;
    float sj[IPL];
    float mx = -INFINITY;
#pragma unroll
    for (int x = 0; x < IPL; ++x) {
        const int j = 32 * x + lane;
        sj[x] = -INFINITY;
        if (j < nb && j >= ntb && j != i) sj[x] = __ldcg(src + j);
        mx = fmaxf(mx, sj[x]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    uint32_t u[IPL];
    double w[IPL];                                         // forced and padding entries weigh nothing
    double part = 0.0;
#pragma unroll
    for (int x = 0; x < IPL; ++x) {
        const int j = 32 * x + lane;
        u[x] = 0u;
        w[x] = 0.0;
        if (j < nb && j >= ntb && j != i) {
            u[x] = score_key(sj[x]);
            w[x] = exp((double)scale * ((double)sj[x] - (double)mx));
        }
        part += w[x];
    }
    const double total = warp_sum(part);
    if (total != total) {
        // A weight is not a number (a NaN among the scores, an infinite maximum): no share compares with it, and every
        // candidate is kept -- those of key 0, which only a NaN with all bits set has, as one.
        int c = 0;
#pragma unroll
        for (int x = 0; x < IPL; ++x) c += u[x] != 0u;
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) row_keep[row] = min(c + 1, n_free);
        return;
    }
    double want = (double)tau * total;                     // mass still to be covered inside the prefix group
    uint32_t prefix;
    int hi = differing_bits(u, prefix);                    // the group: candidates that equal `prefix` from bit `hi` up
    int above = 0, group = n_free;                         // candidates above the group, and in it
    while (hi > 0 && group > 1) {
        const uint32_t bit = 1u << (hi - 1), trial = prefix | bit, rest = bit - 1u;
        double m1 = 0.0;
        int c1 = 0;
#pragma unroll
        for (int x = 0; x < IPL; ++x) {
            const bool in = (u[x] & ~rest) == trial;
            m1 += in ? w[x] : 0.0;
            c1 += in;
        }
        m1 = warp_sum(m1);
        c1 = __reduce_add_sync(0xffffffffu, c1);
        if (m1 >= want) {
            prefix = trial;
            group = c1;
        } else {
            want -= m1;
            above += c1;
            group -= c1;
        }
        --hi;
    }
    // The group's candidates have equal keys now (or there is one; or none, when the mass above them fell short of the
    // share by rounding alone): added one by one until the mass is reached.
    double w_eq = 0.0;
#pragma unroll
    for (int x = 0; x < IPL; ++x)
        if (u[x] && (hi >= 32 || (u[x] >> hi) == (prefix >> hi))) w_eq = w[x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w_eq = fmax(w_eq, __shfl_xor_sync(0xffffffffu, w_eq, o));
    int r = 0;
    double acc = 0.0;
    while (r < group && (r == 0 || acc < want)) {
        acc += w_eq;
        ++r;
    }
    if (lane == 0) row_keep[row] = min(max(above + r, 1), n_free);
}

// Calls f with a register count per lane that holds a row of nb scores.  A kernel takes the time that its count takes, not
// the row, so the counts lie no further apart than by a half.  One image of 24 heads, us, with the counts 3, 9 and 32 alone /
// as it is / the histograms in shared memory that this replaces.  Top-k: 150 blocks 11.9 / 7.8 / 11.5, 200 13.2 / 13.1 / 14.7,
// 289 30.8 / 19.6 / 22.2, 400 42.7 / 27.6 / 32.9, 512 55.2 / 35.7 / 47.8, 600 67.0 / 55.3 / 64.4, 1024 145 / 144 / 262.
// Cumulative mass with its selection: 150 28.2 / 19.1 / 36.1, 289 86.5 / 52.9 / 72.5, 512 157 / 95.9 / 158, 1024 385 / 384 / 748.
template <typename F>
cudaError_t with_ipl(int nb, F&& f) {
    if (nb <= 96) return f(std::integral_constant<int, 3>());
    if (nb <= 192) return f(std::integral_constant<int, 6>());
    if (nb <= 288) return f(std::integral_constant<int, 9>());
    if (nb <= 512) return f(std::integral_constant<int, 16>());
    if (nb <= 768) return f(std::integral_constant<int, 24>());
    return f(std::integral_constant<int, RAPID3_MAX_NB / 32>());
}

template <typename HK>
cudaError_t launch_select(const float* scores, const TensorGeom& g, const ImgList& imgs, uint64_t* bitmask, int32_t* kept_idx,
                          int32_t* kept_cnt, cudaStream_t s, const DevPlan* plan, int n_img, const QuadOrder& order, const HK& hk) {
    const dim3 grid((g.nb + WARPS - 1) / WARPS, n_img * g.H);
    return with_ipl(g.nb, [&](auto ipl) {
        return launch_kernel(order.count ? select_kernel<HK, decltype(ipl)::value, true> : select_kernel<HK, decltype(ipl)::value, false>, grid, dim3(WARPS * 32), 0, s, scores, g, imgs,
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

// One thread decides; the loads, which would cost it a round trip each, and the stores are the whole block's.
__global__ void __launch_bounds__(RAPID3_MAX_IMG) plan_kernel(const int32_t* action, const float* ratio, int B, int n_free_img,
                                                              DevPlan* __restrict__ plan, int* __restrict__ status) {
    __shared__ DevPlan out;
    __shared__ int act[RAPID3_MAX_IMG];
    __shared__ float rat[RAPID3_MAX_IMG], ratio_of[RAPID3_MAX_IMG];
    constexpr int WORDS = sizeof(DevPlan) / sizeof(int);
    static_assert(sizeof(DevPlan) % sizeof(int) == 0, "copied word by word");
    grid_dependency_wait();                           // first kernel of a call
    grid_dependency_launch();
    for (int x = threadIdx.x; x < WORDS; x += RAPID3_MAX_IMG) reinterpret_cast<int*>(&out)[x] = 0;
    if (threadIdx.x < B) {
        act[threadIdx.x] = __ldcg(action + threadIdx.x);
        rat[threadIdx.x] = __ldcg(ratio + threadIdx.x);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        ImgList& sp = out.sparse;
        ImgList& al = out.all;
        int n_dense = 0;
        for (int b = 0; b < B; ++b) {
            const int a = act[b];
            if (a != RAPID3_ACT_SKIP && a != RAPID3_ACT_REUSE && a != RAPID3_ACT_ATTEND) {
                atomicExch(status, RAPID3_ERR_INVALID_ARG);   // unknown action: treated as a skip
                continue;
            }
            if (a != RAPID3_ACT_ATTEND) continue;
            const float r = rat[b];
            if (!(r > 0.f) || !(r <= 1.f)) {
                atomicExch(status, RAPID3_ERR_INVALID_ARG);   // ratio outside (0, 1]: image not processed
                continue;
            }
            int slot = -1;
            if (r < 1.f) {
                slot = sp.n++;
                sp.batch[slot] = b;
                sp.slot[slot] = slot;
                double x = ceil((double)r * (double)n_free_img - 1e-6);
                x = x < 0.0 ? 0.0 : (x > (double)n_free_img ? (double)n_free_img : x);
                sp.k_free[slot] = (int)x;
            } else {
                ++n_dense;
            }
            int pos = al.n++;
            while (pos > 0 && ratio_of[pos - 1] < r) {        // insertion sort, descending ratio, stable
                al.batch[pos] = al.batch[pos - 1];
                al.slot[pos] = al.slot[pos - 1];
                ratio_of[pos] = ratio_of[pos - 1];
                --pos;
            }
            al.batch[pos] = b;
            al.slot[pos] = slot;
            ratio_of[pos] = r;
        }
        out.n_dense = n_dense;
    }
    __syncthreads();
    for (int x = threadIdx.x; x < WORDS; x += RAPID3_MAX_IMG) reinterpret_cast<int*>(plan)[x] = reinterpret_cast<const int*>(&out)[x];
}

}  // namespace

cudaError_t launch_plan(const int32_t* action_dev, const float* ratio_dev, int B, const TensorGeom& g, DevPlan* plan,
                        int* status, cudaStream_t s) {
    const int n_free_img = g.nb - g.n_text_blocks - 1;
    return launch_kernel(plan_kernel, dim3(1), dim3(RAPID3_MAX_IMG), 0, s, action_dev, ratio_dev, B, n_free_img > 0 ? n_free_img : 0,
                         plan, status);
}
