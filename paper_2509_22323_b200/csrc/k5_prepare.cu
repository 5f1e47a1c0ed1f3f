// K5: Q/K producer with the block pooling folded in.  Per-head RMS normalisation with a learned
// gain, rotary embedding (adjacent channel pairs, cos / sin per token from a caller-given table),
// one rounding to bf16 -- and, in the same pass, the fp64 block means of the ROUNDED values for the
// images that will be scored, so that the scoring pass does not have to read Q and K again.
// Layout of the work as in the pooling kernel: one warp per (Q|K, image, head, 64-token block), a
// token row of D channels is D / 8 lanes of 16 bytes; the row's sum of squares is reduced over
// those lanes with shuffles, the rotation is lane-local (a lane holds four whole pairs).
// Reads the raw Q and K once, writes Q and K once: 4.4 to 4.7 TB/s of that in launches of 24 heads, bound by issue slots (118 instructions for 256
// numbers, 56 % of the slots) and the chain of a warp's rows.  The kernel alone, us, before its warps shared a table / since (one run of ncu, caches
// as they are): D = 128 one image of 4608 tokens 28.6 / 26.1, three 79.9 / 71.8, one of 16896 100.8 / 90.7; D = 64 two of 4480 29.4 / 23.8.
#include <algorithm>

#include "ptx.cuh"
#include "scoring.cuh"

using namespace ptx;
using scoring::bf16_hi;
using scoring::bf16_lo;

namespace {

// A thread block does WARPS of the 2 H (Q|K, head) pairs of a 64-token block, which share the block's part of the rotary table: it comes
// to shared memory once (32 KB at D = 128, twice the bytes of one head's rows), while the first rows are on their way; fetched for every
// row by every warp it was two thirds of the traffic from the L2.  The numbers go in packed pairs, so arranged that products and
// rotations are two to an instruction (157 instructions for 256 numbers without); both conversions of a mean's summands go through the
// conversion unit, which has room (a third of its rate), where bits would cost issue slots.
// INFL rows are in flight a lane, each replaced by the one INFL further on as soon as it is taken.  Four of them and 24 warps an SM
// were the best for large launches (two 27.3, 16 warps 38.5, 32 warps with fewer registers 29 us for one image of 4608 tokens; thread blocks of 8 warps
// 26.0, of 4 23.3, by events in one run); eight where the thread blocks have an SM to themselves or nearly so and the time is the chain of their loads
// (steps of one image from raw projections: 2 heads x 36 blocks at D = 64 26.6 -> 25.5 us, 12 heads x 10 blocks at D = 128 29.0 -> 27.4).
template <int D, int INFL, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, INFL > 4 ? 8 / WARPS : 24 / WARPS) prepare_kernel(const uint16_t* q_raw,
                                                      const uint16_t* k_raw, uint16_t* q_out,
                                                      uint16_t* k_out, const float* q_gain,
                                                      const float* k_gain, const float* rot, float eps, TensorGeom g,
                                                      ImgList imgs, int n_sparse, double* __restrict__ pooled) {
    constexpr int TPR = D / 8;          // lanes per token row (8 channels = 16 bytes each)
    constexpr int RPL = 32 / TPR;       // rows per warp-wide load
    constexpr int ITERS = 64 / RPL;     // loads per lane
    // [row][half][lane]: of two channel pairs cos, cos, sin, sin; a lane's next to those of the lanes beside it
    __shared__ float4 table[64 * 2 * TPR];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int blk = blockIdx.x, p = blockIdx.z, pair = blockIdx.y * WARPS + warp;
    const int n0 = blk * 64;
    const int valid = min(64, g.N - n0);
    grid_dependency_wait();                           // first kernel of a call: what comes before it may still be running
    const int which = pair >= g.H, h = pair - which * g.H;               // 0 = Q, 1 = K
    const int batch = imgs.batch[p], slot = imgs.slot[p];
    const long long off = (long long)batch * g.stride_b + (long long)(g.h0 + h) * g.stride_h + (long long)n0 * g.stride_n;
    const uint16_t* src = (which ? k_raw : q_raw) + off;
    uint16_t* dst = (which ? k_out : q_out) + off;
    const int c = lane % TPR, r0 = lane / TPR;
    const bool work = pair < 2 * g.H;
    auto load_raw = [&](int it) {
        const int row = it * RPL + r0;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (work && row < valid) v = __ldcg(reinterpret_cast<const uint4*>(src + (long long)row * g.stride_n + c * 8));
        return v;
    };
    uint4 next[INFL];
#pragma unroll
    for (int u = 0; u < INFL; ++u) next[u] = load_raw(u);
    {
        const float4* from = reinterpret_cast<const float4*>(rot + (long long)n0 * D);
        // many loads at once: a thread block waits for them (4 at a time 0.4 to 1.1 us a launch)
#pragma unroll(INFL > 4 ? 16 : 8)
        for (int x = threadIdx.x; x < 64 * 2 * TPR; x += 32 * WARPS) {
            float4 t = make_float4(1.f, 0.f, 1.f, 0.f);
            if (rot && x < valid * 2 * TPR) t = __ldcg(from + x);
            const int row = x / (2 * TPR), piece = x % (2 * TPR);
            table[(row * 2 + (piece & 1)) * TPR + (piece >> 1)] = make_float4(t.x, t.z, t.y, t.w);
        }
    }
    // Channels 0 and 2, 4 and 6 of the lane's eight (first of their pairs) go together as packed numbers, and 1 and 3, 5 and 7.
    uint64_t gain_a[2], gain_b[2], minus_b[2];
    {
        const float* gain = (which ? k_gain : q_gain) + c * 8;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float4 v = __ldcg(reinterpret_cast<const float4*>(gain) + i);
            gain_a[i] = pair_of(v.x, v.z);
            gain_b[i] = pair_of(v.y, v.w);
            minus_b[i] = pair_of(-v.y, -v.w);
        }
    }
    __syncthreads();
    if (!work) {
        grid_dependency_launch();
        return;
    }
    double acc[8];
    float finite = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.0;
#pragma unroll 1
    for (int it0 = 0; it0 < ITERS; it0 += INFL) {
#pragma unroll
        for (int u = 0; u < INFL; ++u) {
            const int row = (it0 + u) * RPL + r0;
            const uint4 v = next[u];                  // (a lane reads its rows before it writes them, should the output lie over the input)
            if (it0 + INFL < ITERS) next[u] = load_raw(it0 + INFL + u);
            const uint32_t in[4] = {v.x, v.y, v.z, v.w};
            float ss = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) ss = fmaf(bf16_hi(in[e]), bf16_hi(in[e]), fmaf(bf16_lo(in[e]), bf16_lo(in[e]), ss));
#pragma unroll
            for (int o = 1; o < TPR; o <<= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            const float r = rsqrtf(ss * (1.0f / (float)D) + eps);       // 2 ulp: far inside the bf16 rounding of the result
            const uint64_t rr = pair_of(r, r);
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const uint64_t xa = mul2(pair_of(bf16_lo(in[2 * i]), bf16_lo(in[2 * i + 1])), rr);
                const uint64_t xb = mul2(pair_of(bf16_hi(in[2 * i]), bf16_hi(in[2 * i + 1])), rr);
                const float4 t = table[(row * 2 + i) * TPR + c];
                const uint64_t cosine = pair_of(t.x, t.y), sine = pair_of(t.z, t.w), ya = mul2(xa, gain_a[i]);
                const float2 za = of_pair(fma2(ya, cosine, mul2(mul2(xb, minus_b[i]), sine)));
                const float2 zb = of_pair(fma2(ya, sine, mul2(mul2(xb, gain_b[i]), cosine)));
                w[2 * i] = pack_bf16(za.x, zb.x);
                w[2 * i + 1] = pack_bf16(za.y, zb.y);
            }
            if (row < valid) {
                const uint4 z = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4*>(dst + (long long)row * g.stride_n + c * 8) = z;
                if (slot >= 0) scoring::add_row<true>(acc, finite, z);  // only scored images need their block means
            }
        }
    }
    // Only now may the scores kernel's thread blocks come in: let in at the top, they cost a small launch more than their
    // early start saves (steps of 144 and 28 quads from raw projections 25.5 -> 22.3 and 30.5 -> 27.4 us).
    grid_dependency_launch();
    if (slot < 0) return;                             // a dense image is not scored (warp-uniform)
    double* mean = pooled + ((((long long)which * n_sparse + slot) * g.H + h) * g.nb + blk) * D;
    scoring::write_mean<D, true>(acc, valid, mean, lane);
}

// Shared memory, beside the table, that a thread block of a launch of few asks for: so much that no more of them fit an SM than the launch needs.
// They may be let in while add_parts_kernel of the call before still holds most SMs (two of its thread blocks fit one), and would pile up on those with
// room: 2 heads of 24 to 32 blocks at D = 128, whole steps from raw projections, us, without / with 31.0 to 33.2 / 26.8 to 29.3; one head of 36 32.4 / 27.9;
// 96 steps of 1 to 6 heads of 20 to 58 blocks 3 % faster in the mean.
int spread_smem_bytes(int D, int blocks) {
    const int sm_bytes = 228 << 10, per_sm = (blocks + SM_COUNT - 1) / SM_COUNT;
    return std::max(0, sm_bytes / (per_sm + 1) - 256 * D);              // 256 D: the table; each thread block takes 1 KB more
}

}  // namespace

cudaError_t prepare_static_init() {
    const cudaError_t e = cudaFuncSetAttribute(prepare_kernel<128, 8, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, spread_smem_bytes(128, 1));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(prepare_kernel<64, 8, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, spread_smem_bytes(64, 1));
}

cudaError_t launch_prepare(const PrepArgs& a, const TensorGeom& g, const ImgList& imgs, int n_sparse, double* pooled,
                           cudaStream_t s) {
    const uint16_t* qr = static_cast<const uint16_t*>(a.q_raw);
    const uint16_t* kr = static_cast<const uint16_t*>(a.k_raw);
    uint16_t* qo = static_cast<uint16_t*>(a.q_out);
    uint16_t* ko = static_cast<uint16_t*>(a.k_out);
    const bool few = (g.nb + 3) / 4 * 2ll * g.H * imgs.n <= 2 * SM_COUNT;
    const int warps = few ? 2 : 4;
    const dim3 grid(g.nb, (2 * g.H + warps - 1) / warps, imgs.n);
    const auto kernel = few ? (g.D == 128 ? prepare_kernel<128, 8, 2> : prepare_kernel<64, 8, 2>)
                            : (g.D == 128 ? prepare_kernel<128, 4, 4> : prepare_kernel<64, 4, 4>);
    return launch_kernel(kernel, grid, dim3(32 * warps), few ? spread_smem_bytes(g.D, (int)(grid.x * grid.y * grid.z)) : 0, s, qr, kr, qo, ko,
                         a.q_gain, a.k_gain, a.rot, a.eps, g, imgs, n_sparse, pooled);
}
