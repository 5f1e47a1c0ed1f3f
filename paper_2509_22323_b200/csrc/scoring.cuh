// Device code that the kernels of the scoring pass share: the mean of a block, the fp64 tensor-core step of the scores, and
// the selection of one row by one warp.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace scoring {

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// Adds a lane's eight bf16 channels to its fp64 accumulators.  The conversion unit takes 16 numbers a clock and SM, so only the low
// halves go through it (WIDE: all of them).  A high half becomes a double by its bits alone: sign, exponent and significand
// moved to their places, with the exponent's bias left as it is, which is the number times 2^-896 -- exactly, zeros and
// subnormal numbers included, and the sums of such numbers round as the sums of the numbers themselves do.  Infinities and NaN would
// come out as numbers: times zero they leave a NaN in `finite`, and the block is summed again the wide way.
// (48 thread blocks of 24 warps on 2.36 MB each 54.5 -> 52.4 us, 24 on 1.15 MB 27.3 -> 24.8.)
template <bool WIDE>
__device__ __forceinline__ void add_row(double (&acc)[8], float& finite, const uint4& v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        acc[2 * e] += (double)bf16_lo(w[e]);
        if constexpr (WIDE) {
            acc[2 * e + 1] += (double)bf16_hi(w[e]);
        } else {
            acc[2 * e + 1] += __hiloint2double(((int)w[e] >> 3) & 0x8fffe000, 0);
            finite = fmaf(__uint_as_float(w[e]), 0.f, finite);
        }
    }
}

// The mean of `valid` rows from the lanes' sums (add_row's), to `out`.
template <int D, bool WIDE>
__device__ __forceinline__ void write_mean(double (&acc)[8], int valid, double* out, int lane) {
    constexpr int TPR = D / 8;          // lanes that hold different channels
    if constexpr (!WIDE) {
#pragma unroll
        for (int e = 1; e < 8; e += 2) acc[e] *= 0x1p896;
    }
#pragma unroll
    for (int off = TPR; off < 32; off <<= 1)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], off);
    if (lane < TPR) {
        const double inv = 1.0 / (double)valid;
#pragma unroll
        for (int e = 0; e < 8; e += 2) *reinterpret_cast<double2*>(out + lane * 8 + e) = make_double2(acc[e] * inv, acc[e + 1] * inv);
    }
}

// Mean of `valid` token rows (stride elements apart) by one warp, in fp64, to `out`.  A row of D channels is D / 8 lanes of 16 bytes,
// so a warp-wide load covers 32 / (D / 8) rows; a lane keeps fp64 sums of its 8 channels over the rows that it sees, eight
// loads in flight, and the lanes that hold the same channels are then added with shuffles.
// `loaded` is called when the last load is through.  False: nothing is written, a number is not finite.
template <int D, bool WIDE, typename Loaded>
__device__ __forceinline__ bool pool_block_as(const uint16_t* base, long long stride, int valid, double* out, int lane, Loaded&& loaded) {
    constexpr int TPR = D / 8;          // lanes per token row (8 channels = 16 bytes each)
    constexpr int RPL = 32 / TPR;       // rows per warp-wide load
    constexpr int ITERS = 64 / RPL;     // loads per lane
    const int c = lane % TPR, r0 = lane / TPR;
    double acc[8];
    float finite = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.0;
#pragma unroll 1
    for (int it0 = 0; it0 < ITERS; it0 += 8) {
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int row = (it0 + u) * RPL + r0;
            v[u] = make_uint4(0, 0, 0, 0);
            if (row < valid) v[u] = __ldcg(reinterpret_cast<const uint4*>(base + (long long)row * stride + c * 8));
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) add_row<WIDE>(acc, finite, v[u]);
    }
    if (!WIDE && __any_sync(0xffffffffu, finite != 0.f)) return false;
    loaded();
    write_mean<D, WIDE>(acc, valid, out, lane);
    return true;
}
template <int D, typename Loaded>
__device__ __forceinline__ void pool_block(const uint16_t* base, long long stride, int valid, double* out, int lane, Loaded&& loaded) {
    if (!pool_block_as<D, false>(base, stride, valid, out, lane, loaded)) pool_block_as<D, true>(base, stride, valid, out, lane, loaded);
}

// D(8 x 8, fp64) += A(8 x 4, row) * B(4 x 8, col) on the fp64 tensor path (four times the rate of the fp64 FMA pipe
// on this part).  Lane l holds a = A[l / 4][l % 4], b = B[l % 4][l / 4] and c0, c1 = D[l / 4][2 (l % 4) + {0, 1}].
__device__ __forceinline__ void dmma_8x8x4(double& c0, double& c1, double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                 : "+d"(c0), "+d"(c1)
                 : "d"(a), "d"(b));
}

__device__ __forceinline__ void copy16_async(double* dst, const double* src, bool valid) {   // past the L1; zeros if not valid
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                 ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

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

// One row by one warp: of its free candidates the k with the best scores, IPL = ceil(nb / 32) or more of them a lane; `score(j)` reads
// one.  Writes the row's bit mask, kept list and count; `word(x, bits)` gets the mask's 32-bit words on lane 0.
template <int IPL, typename Score, typename Word>
__device__ __forceinline__ void select_row(Score&& score, int i, int nb, int ntb, int k, int lane, uint32_t* out_bits, int words32,
                                           int32_t* out_idx, int32_t* out_cnt, Word&& word) {
    const bool text_row = i < ntb;
    const int n_free = max(nb - ntb - ((i >= ntb) ? 1 : 0), 0);
    const bool select = !text_row && k > 0 && k < n_free;
    uint32_t u[IPL];
#pragma unroll
    for (int x = 0; x < IPL; ++x) {
        const int j = 32 * x + lane;
        u[x] = 0u;
        if (select && j < nb && j >= ntb && j != i) u[x] = score_key(score(j));
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
            word(x, bal);
        }
        if (keep) out_idx[total + __popc(bal & ((1u << lane) - 1u))] = j;
        total += __popc(bal);
    }
    for (int c = (nb + 31) / 32 + lane; c < words32; c += 32) out_bits[c] = 0;   // odd 32-bit half of the last word
    for (int e = total + lane; e < nb; e += 32) out_idx[e] = -1;
    if (lane == 0) *out_cnt = total;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
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
template <int IPL, typename Score>
__device__ __forceinline__ int mass_row(Score&& score, int i, int nb, int ntb, float tau, float scale, int lane) {
    const int n_free = (i < ntb) ? 0 : max(nb - ntb - 1, 0);
    if (n_free == 0 || tau >= 1.f) return n_free;          // warp-uniform
    float sj[IPL];
    float mx = -INFINITY;
#pragma unroll
    for (int x = 0; x < IPL; ++x) {
        const int j = 32 * x + lane;
        sj[x] = -INFINITY;
        if (j < nb && j >= ntb && j != i) sj[x] = score(j);
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
        return min(c + 1, n_free);
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
    return min(max(above + r, 1), n_free);
}

// An image's place among the sparse ones in the attention's list, from a plan on the device.
__device__ __forceinline__ int plan_place(const DevPlan* plan, int p, int lane) {
    const int n_all = __ldcg(&plan->all.n);
    auto here = [&](int at) { return at < n_all && __ldcg(&plan->all.slot[at]) == p; };
    const uint32_t lo = __ballot_sync(0xffffffffu, here(lane)), hi = __ballot_sync(0xffffffffu, here(32 + lane));
    return (lo ? __ffs(lo) - 1 : 31 + __ffs(hi)) - __ldcg(&plan->n_dense);
}

// A quad's class in the attention's order (QuadOrder), by one warp: m[a] are the 32 bits of member a's mask from block 32 * lane
// on.  `place`: the image's place among the sparse ones in the attention's list.
__device__ __forceinline__ void order_quad(const QuadOrder& order, const TensorGeom& g, int n_dense, int n_sparse, int place, int h, int quad,
                                           const uint32_t (&m)[4], int lane) {
    const int nq = (g.nb + 3) >> 2, ntq = (g.n_text_blocks + 3) >> 2, nl = nq - ntq;
    const int at = (place * g.H + h) * nl + quad - ntq - order_after(n_sparse * g.H * nl, g.H * (n_dense * nq + n_sparse * ntq));
    if (quad < ntq || at < 0) return;                      // quads with text rows, and all but the last of the others, come as they are
    // the quad's time, in quarters of a key block of two tiles: one that only one tile uses takes three quarters
    const uint32_t t0 = m[0] | m[1], t1 = m[2] | m[3];
    const int time = __reduce_add_sync(0xffffffffu, 2 * __popc(t0 | t1) + __popc(t0) + __popc(t1));
    if (lane == 0) order.cls[at] = (uint8_t)(ORDER_CLASSES - 1 - time * (ORDER_CLASSES - 1) / (4 * g.nb));
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

}  // namespace scoring
