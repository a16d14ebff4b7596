// k_field_tc.cu - the field on the 5th-generation tensor cores (FP16 or BF16
// operands, FP32 accumulation in tensor memory): hash encoding, density MLP
// (sigma = exp(h_0)), SH view encoding and colour MLP forward (steps a3-a6), and the
// recomputing backward pass with the weight gradients accumulated in tensor memory
// across a persistent block's tiles (steps a10-a11).
//
// A group of 128 threads takes a tile of 128 samples through the layers: thread r of
// the group owns operand row r, which is TMEM lane r of every 128-row accumulator.  Each
// layer is one chain of tcgen05.mma instructions issued by an elected lane of the group's
// first warp on shared-memory operands (layout in tc_ptx.cuh), committed to an mbarrier;
// the group then reads the accumulator rows back with tcgen05.ld, applies the activation
// in FP32, rounds to the MLP type and writes the next operand tile.
// Forward: the groups of a block (six; one in a grouped render of several maps) share one
// copy of the weights and take tiles on their own; the rows of a warp hold its samples in
// the encoding's pair order.  Backward: a block has one such group, and two more that load
// the tiles' inputs and scatter the table gradients; rows are in sample order.  Weight
// gradients are M=64 products over the tile's samples (MN-major operands of the same
// tiles) that keep accumulating in TMEM until the block has no tiles left.
//
// Gradient tiles are scaled by powers of two before rounding to the MLP type: the
// colour branch (dL/dz through the colour MLP down to its input, weights W3-W5) by
// S_c, which brings the step's largest colour seed |dL/dc| to about 2^8, and the
// density branch (from dL/dh on, weights W1-W2 and the tables) by S_d, which does the
// same for the larger of the density seeds |dL/dsigma * sigma| and the colour seeds.
// The depth term's seeds are usually far larger than the colour ones, so one shared
// scale would push the colour gradients into FP16's subnormal range.  2^8 leaves a
// factor 2^8 of headroom below FP16's largest value for the growth of the gradient
// through the layers (fan-in 64) and keeps seeds down to 2^-22 of the largest one
// normal; with 2^13 the deepest colour-branch tiles saturated in trained fields.
// FP16 encodings enter the MLP scaled by 2^8 (table values start near 1e-4, below
// FP16's normal range).  Both scales are exact and are removed in FP32.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "encoding.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace nm {

using namespace tc;

namespace {

constexpr float kGradTarget = 256.f;  // largest scaled gradient seed (see above)

// Two values rounded to the MLP type, a in the low half: one cvt to a packed pair
// (the pair's first source operand fills the upper half).  FP16 saturates at the
// largest finite value (+-65504) instead of overflowing; RELU also maps negative
// values to zero.
template <bool BF16, bool RELU = false>
__device__ __forceinline__ uint32_t pack2(float a, float b) {
    uint32_t d;
    if constexpr (BF16) {
        if constexpr (RELU) asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
        else asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    } else {
        if constexpr (RELU) asm("cvt.rn.relu.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
        else asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    }
    return d;
}

template <bool BF16>
__device__ __forceinline__ uint16_t pack1(float a) {
    if constexpr (BF16) {
        return __bfloat16_as_ushort(__float2bfloat16_rn(a));
    } else {
        return __half_as_ushort(__float2half_rn(fminf(fmaxf(a, -65504.f), 65504.f)));
    }
}

// Row r (of 128) of a tile with C columns, from C floats.
template <bool BF16, int C>
__device__ __forceinline__ void store_row(uint8_t* tile, int r, const float* v) {
#pragma unroll
    for (int g = 0; g < C / 8; ++g) {
        uint4 q;
        q.x = pack2<BF16>(v[8 * g + 0], v[8 * g + 1]);
        q.y = pack2<BF16>(v[8 * g + 2], v[8 * g + 3]);
        q.z = pack2<BF16>(v[8 * g + 4], v[8 * g + 5]);
        q.w = pack2<BF16>(v[8 * g + 6], v[8 * g + 7]);
        *reinterpret_cast<uint4*>(tile + tile_offset(r, 8 * g, 128)) = q;
    }
}

// C columns of row r of a 128-row tile from C floats, starting at column c0
// (RELU: max(v, 0) is stored).
template <bool BF16, int C, bool RELU = false>
__device__ __forceinline__ void store_row_at(uint8_t* tile, int r, int c0, const float* v) {
#pragma unroll
    for (int g = 0; g < C / 8; ++g) {
        uint4 q;
        q.x = pack2<BF16, RELU>(v[8 * g + 0], v[8 * g + 1]);
        q.y = pack2<BF16, RELU>(v[8 * g + 2], v[8 * g + 3]);
        q.z = pack2<BF16, RELU>(v[8 * g + 4], v[8 * g + 5]);
        q.w = pack2<BF16, RELU>(v[8 * g + 6], v[8 * g + 7]);
        *reinterpret_cast<uint4*>(tile + tile_offset(r, c0 + 8 * g, 128)) = q;
    }
}

// N consecutive accumulator columns of this thread's lane.
template <int N>
__device__ __forceinline__ void ld_cols(uint32_t trow, uint32_t col, float* v) {
#pragma unroll
    for (int c = 0; c < N; c += 16) tmem_ld16(trow + col + c, v + c);
    tmem_wait_ld();
}

// An operand tile at byte offset OFF of the block's shared memory, R rows.  K-major: rows
// index M (or N), columns K.  MN-major: rows index K, columns M (or N).
template <uint32_t OFF, int R>
struct KMaj {
    static constexpr uint32_t lo = desc_lo(OFF, (uint32_t)(R / 8) * 128u), hi = desc_hi(128u);
    static constexpr uint32_t kstep = (uint32_t)(R / 8) * 256u;
    static constexpr bool mn = false;
};
template <uint32_t OFF, int R>
struct MnMaj {
    static constexpr uint32_t lo = desc_lo(OFF, 128u), hi = desc_hi((uint32_t)(R / 8) * 128u);
    static constexpr uint32_t kstep = 256u;
    static constexpr bool mn = true;
};

// D (M x N, at TMEM address d) (+)= A B over KS steps of K = 16; a4, b4: the shared-memory
// bases of the operands' tiles / 16.
template <bool BF16, int M, int N, class A, class B, int KS>
__device__ __forceinline__ void gemm(uint32_t d, uint32_t a4, uint32_t b4, bool acc) {
    asm volatile("" : "+r"(a4), "+r"(b4), "+r"(d));  // the adds stay here: hoisted out of the tile loop they spill
#pragma unroll
    for (int k = 0; k < KS; ++k)
        mma_f16<A::hi, B::hi, idesc_f16(M, N, BF16, A::mn, B::mn)>(
            d, a4 + A::lo + k * (A::kstep >> 4), b4 + B::lo + k * (B::kstep >> 4), (acc || k > 0) ? 1u : 0u);
}

__device__ __forceinline__ void nb_sync(int id, int n) {
    asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void nb_arrive(int id, int n) {
    asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(n) : "memory");
}

// Whether any of the barrier's n threads passes true.
__device__ __forceinline__ bool nb_or(int id, int n, bool v) {
    uint32_t r;
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %3, 0;\n"
        "bar.red.or.pred q, %1, %2, p;\n"
        "selp.u32 %0, 1, 0, q;\n"
        "}\n" : "=r"(r) : "r"(id), "r"(n), "r"((uint32_t)v) : "memory");
    return r != 0u;
}

// Makes this thread's operand writes visible to the tensor core and orders its
// earlier TMEM reads before the next MMA; block-wide.
__device__ __forceinline__ void to_tensor() {
    fence_proxy_async();
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
}

// The same for the 128 threads of one group of the block (barrier `id`).
__device__ __forceinline__ void to_tensor_group(int id) {
    fence_proxy_async();
    fence_before_sync();
    nb_sync(id, 128);
    fence_after_sync();
}

// Waits for the MMAs committed to `bar` (at most `polls` polls; 0 makes the wait
// expire at once).  After a timeout the thread stops waiting, the rest of its work is
// garbage, and the block drains its MMAs before it frees tensor memory (drain_mma).
__device__ __forceinline__ void wait_mma(uint64_t* bar, uint32_t& phase, bool& timed_out, uint32_t polls) {
    if (!timed_out) timed_out = !mbar_wait(bar, phase, polls);
    phase ^= 1u;
    fence_after_sync();
}

// After a timeout: the MMA-issuing thread commits once more, to a barrier that has
// seen no other commit, and waits for it (bounded by the default limit).  The commit
// arrives when every MMA that thread has issued has completed, so the tensor memory
// can be freed afterwards; the phases of the main barrier are not trusted (several
// of its phases may have completed while nobody waited).
__device__ __forceinline__ void drain_mma(uint64_t* drain_bar) {
    mma_commit(drain_bar);
    mbar_wait(drain_bar, 0u, kWaitPollsDefault);
    fence_after_sync();
}

constexpr int kW1B = 64 * 32 * 2, kW2B = 16 * 64 * 2, kW3B = 64 * 32 * 2, kW4B = 64 * 64 * 2, kW5B = 16 * 64 * 2;
constexpr int kWB = kW1B + kW2B + kW3B + kW4B + kW5B;  // 20480
constexpr int kT32 = 128 * 32 * 2, kT64 = 128 * 64 * 2, kT16 = 128 * 16 * 2;
// byte offsets of the weight tiles in the block's shared memory
constexpr uint32_t kOW1 = 0, kOW2 = kOW1 + kW1B, kOW3 = kOW2 + kW2B, kOW4 = kOW3 + kW3B, kOW5 = kOW4 + kW4B;

// Weight tiles (MLP type) from the FP32 master weights: W1 64x32, W2 16x64,
// W3 64x32, W4 64x64, W5 padded to 16x64 (rows 3..15 zero).  smem: the block's shared
// memory, whose start holds the tiles; NT threads (tid 0 .. NT - 1).  Every launch pays
// this once per block before its first tile, so the loads are 16 bytes and up to 7 in
// flight per thread (one 4-byte load at a time: 30 us of a small render's or step's
// forward launch).
template <bool BF16, int NT>
__device__ void load_weight_tiles(const float* __restrict__ mlp, uint8_t* smem, int tid) {
    constexpr int kQuads = kMlpParams / 4, kIters = (kQuads + NT - 1) / NT, kBatch = kIters < 7 ? kIters : 7;
    static_assert(kMlpParams % 4 == 0 && kOffW2 % 4 == 0 && kOffW3 % 4 == 0 && kOffW4 % 4 == 0 && kOffW5 % 4 == 0,
                  "four weights of one row at a time");
#pragma unroll 1
    for (int b = 0; b < kIters; b += kBatch) {
        float4 w[kBatch];
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int q = (b + k) * NT + tid;
            w[k] = q < kQuads ? __ldg(reinterpret_cast<const float4*>(mlp) + q) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int i = 4 * ((b + k) * NT + tid);
            if (i >= kMlpParams) continue;
            uint32_t o;
            if (i < kOffW2) o = kOW1 + tile_offset(i / 32, i % 32, 64);
            else if (i < kOffW3) o = kOW2 + tile_offset((i - kOffW2) / 64, (i - kOffW2) % 64, 16);
            else if (i < kOffW4) o = kOW3 + tile_offset((i - kOffW3) / 32, (i - kOffW3) % 32, 64);
            else if (i < kOffW5) o = kOW4 + tile_offset((i - kOffW4) / 64, (i - kOffW4) % 64, 64);
            else o = kOW5 + tile_offset((i - kOffW5) / 64, (i - kOffW5) % 64, 16);
            *reinterpret_cast<uint2*>(smem + o) =
                make_uint2(pack1<BF16>(w[k].x) | ((uint32_t)pack1<BF16>(w[k].y) << 16),
                           pack1<BF16>(w[k].z) | ((uint32_t)pack1<BF16>(w[k].w) << 16));
        }
    }
    for (int j = 192 + 4 * tid; j < 16 * 64; j += 4 * NT)
        *reinterpret_cast<uint2*>(smem + kOW5 + tile_offset(j / 64, j % 64, 16)) = make_uint2(0u, 0u);
}

__device__ __forceinline__ float3 sample_pos_tc(const DevCfg& c, const float* __restrict__ rays, uint32_t cap,
                                                uint32_t r, float t, float3& d) {
    const float3 o = make_float3(rays[kOx * cap + r], rays[kOy * cap + r], rays[kOz * cap + r]);
    d = make_float3(rays[kDx * cap + r], rays[kDy * cap + r], rays[kDz * cap + r]);
    return grid_pos(c, o, d, t);
}

using W1K = KMaj<kOW1, 64>;
using W2K = KMaj<kOW2, 16>;
using W3K = KMaj<kOW3, 64>;
using W4K = KMaj<kOW4, 64>;
using W5K = KMaj<kOW5, 16>;
using W1M = MnMaj<kOW1, 64>;
using W2M = MnMaj<kOW2, 16>;
using W3M = MnMaj<kOW3, 64>;
using W4M = MnMaj<kOW4, 64>;
using W5M = MnMaj<kOW5, 16>;

}  // namespace

// A forward block has NG groups of 128 threads, each with its own tile buffers, TMEM columns,
// MMA barriers and hardware barrier (1 + group), and one copy of the weight tiles.  Step and
// render launch one block of six groups per SM, which leaves the L1 about 90 KB for the
// gathers: field_fwd of 19.5 M samples 2.82 ms (five groups 2.87, four 3.09, three 3.63).  Four blocks
// with a copy of the weights each left 60 KB and took 3.33, five 3.84.  The grouped render
// switches weights between tiles and has one group per block.
constexpr int kFwdGroups = 6;
constexpr int kFwdTile = kT32 + kT64;
constexpr int kFwdSmem = kWB + kFwdTile;                // one group
constexpr int kFwdSmemN = kWB + kFwdGroups * kFwdTile;  // 167936
// TMEM columns of NG groups: an allocation is a power of two
constexpr uint32_t fwd_cols(int NG) { return NG == 1 ? 64u : NG == 2 ? 128u : NG <= 4 ? 256u : 512u; }

// ------------------------------------------------------------------ forward
// One tile of the forward: samples i0 .. min(i0 + 128, i_end) - 1; thread r of the
// group owns sample row r, the samples of a warp in pair_sample order.  smem: the weight
// tiles, then per group tA (128 x 32: X0, X3) and tB (128 x 64: H1, H3, H4; a layer's MMAs
// have completed before its output overwrites its input).  Returns after the tile's last
// MMA wait.
// kSel: row r evaluates sample sel[i0 + r] of the batch instead of i0 + r (a render's
// passes over a subset of the samples).
// kSplit: the levels from split_level(c) on have been gathered level by level
// (k_gather_levels); their packed features are read from `fine`.
template <bool BF16, bool kSel = false, bool kSplit = false>
__device__ __forceinline__ void fwd_tile(const DevCfg& c, const float2* __restrict__ tables,
                                         const float* __restrict__ rays, uint32_t cap,
                                         const uint32_t* __restrict__ ray_id, const float* __restrict__ ts,
                                         float4* __restrict__ sig_rgb, uint4* __restrict__ feat_out,
                                         float feat_scale, uint32_t i0, uint32_t i_end, uint8_t* smem,
                                         uint32_t tmem, uint64_t* bar, uint32_t& phase, bool& timed_out,
                                         const uint32_t* __restrict__ sel = nullptr,
                                         const uint32_t* __restrict__ fine = nullptr, size_t fine_stride = 0) {
    const int tid = threadIdx.x & 127, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int group = __shfl_sync(0xffffffffu, threadIdx.x >> 7, 0), bid = 1 + group;
    uint8_t* tA = smem + kWB + group * kFwdTile;
    uint8_t* tB = tA + kT32;
    using TA = KMaj<kWB, 128>;
    using TB = KMaj<kWB + kT32, 128>;
    const uint32_t b4 = smem_u32(smem) >> 4, a4 = b4 + group * (kFwdTile >> 4);
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
    const float inv_fs = 1.f / feat_scale;
    // which sample a row holds is free: the rows of a warp follow the encoding's pairs
    const uint32_t ti = i0 + (tid & ~31) + pair_sample(tid & 31);
    const bool valid = ti < i_end;
    const uint32_t i = kSel ? (valid ? sel[ti] : 0u) : ti;
    float v[32];
    float3 d = make_float3(0.f, 0.f, 0.f);
    float3 x = make_float3(0.f, 0.f, 0.f);
    if (valid) x = sample_pos_tc(c, rays, cap, ray_id[i], ts[i], d);
    // one group of kGatherGroup = 4 levels = 8 features = one 16-byte chunk of the row
#pragma unroll 1
    for (int g = 0; g < kEnc / 8; ++g) {
        uint4 q;
        if constexpr (kSplit) {
            uint32_t w[4];
            const int l0 = (int)split_level(c.L);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int l = kGatherGroup * g + k;
                w[k] = 0u;
                if (l < l0) {
                    encode_level(c, tables, x, l, v);
                    w[k] = valid ? pack2<BF16>(v[0] * feat_scale, v[1] * feat_scale) : 0u;
                } else if (l < (int)c.L && valid) {
                    w[k] = __ldcs(fine + (size_t)(l - l0) * fine_stride + i);
                }
            }
            q = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
            encode_group(c, tables, x, kGatherGroup * g, v);  // whole warps (an invalid row: position 0)
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = valid ? v[k] * feat_scale : 0.f;
            q.x = pack2<BF16>(v[0], v[1]);
            q.y = pack2<BF16>(v[2], v[3]);
            q.z = pack2<BF16>(v[4], v[5]);
            q.w = pack2<BF16>(v[6], v[7]);
        }
        *reinterpret_cast<uint4*>(tA + tile_offset(tid, 8 * g, 128)) = q;
        if (!kSel && feat_out && valid) feat_out[(size_t)i * 4 + g] = q;
    }
    // layer 1: D = X0 W1^T (128 x 64)
    to_tensor_group(bid);
    if (warp == 0 && elect_one()) {
        gemm<BF16, 128, 64, TA, W1K, 2>(tmem, a4, b4, false);
        mma_commit(bar);
    }
    wait_mma(bar, phase, timed_out, c.wait_polls);
#pragma unroll
    for (int h = 0; h < 64; h += 32) {  // 32-column halves keep fewer values live
        ld_cols<32>(trow, h, v);
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] *= inv_fs;
        store_row_at<BF16, 32, true>(tB, tid, h, v);
    }
    // layer 2: y = H1 W2^T (128 x 16)
    to_tensor_group(bid);
    if (warp == 0 && elect_one()) {
        gemm<BF16, 128, 16, TB, W2K, 4>(tmem, a4, b4, false);
        mma_commit(bar);
    }
    wait_mma(bar, phase, timed_out, c.wait_polls);
    ld_cols<16>(trow, 0, v);
    const float sigma = expf(fminf(v[0], kSigmaHMax));
    if (valid) sh16(d.x, d.y, d.z, v + kGeo);
    else {
#pragma unroll
        for (int k = kGeo; k < 32; ++k) v[k] = 0.f;
    }
    store_row<BF16, 32>(tA, tid, v);
    // layer 3: H3 = relu(X3 W3^T)
    to_tensor_group(bid);
    if (warp == 0 && elect_one()) {
        gemm<BF16, 128, 64, TA, W3K, 2>(tmem, a4, b4, false);
        mma_commit(bar);
    }
    wait_mma(bar, phase, timed_out, c.wait_polls);
#pragma unroll
    for (int h = 0; h < 64; h += 32) {
        ld_cols<32>(trow, h, v);
        store_row_at<BF16, 32, true>(tB, tid, h, v);
    }
    // layer 4: H4 = relu(H3 W4^T)
    to_tensor_group(bid);
    if (warp == 0 && elect_one()) {
        gemm<BF16, 128, 64, TB, W4K, 4>(tmem, a4, b4, false);
        mma_commit(bar);
    }
    wait_mma(bar, phase, timed_out, c.wait_polls);
#pragma unroll
    for (int h = 0; h < 64; h += 32) {
        ld_cols<32>(trow, h, v);
        store_row_at<BF16, 32, true>(tB, tid, h, v);
    }
    // layer 5: z = H4 W5^T (3 of 16 columns used)
    to_tensor_group(bid);
    if (warp == 0 && elect_one()) {
        gemm<BF16, 128, 16, TB, W5K, 4>(tmem, a4, b4, false);
        mma_commit(bar);
    }
    wait_mma(bar, phase, timed_out, c.wait_polls);
    ld_cols<16>(trow, 0, v);
    if (valid) sig_rgb[i] = make_float4(sigma, sigmoidf_(v[0]), sigmoidf_(v[1]), sigmoidf_(v[2]));
}

// Tensor memory and barriers of a forward block: 64 TMEM columns (one 128 x 64 FP32
// accumulator), an MMA barrier and a drain barrier per group.
template <int NG>
__device__ __forceinline__ uint32_t fwd_block_setup(uint32_t* tslot, uint64_t* bar, uint64_t* drain_bar) {
    if ((threadIdx.x >> 5) == 0) tmem_alloc(tslot, fwd_cols(NG));
    if (threadIdx.x == 0) {
        for (int g = 0; g < NG; ++g) {
            mbar_init(bar + g, 1);
            mbar_init(drain_bar + g, 1);
        }
        mbar_fence_init();
    }
    to_tensor();
    return *tslot;
}

// End of a forward block: after a timeout, drain each group's issued MMAs; free the TMEM.
template <int NG>
__device__ __forceinline__ void fwd_block_finish(uint32_t tmem, uint64_t* drain_bar, bool timed_out) {
    fence_before_sync();
    const bool any_timeout = __syncthreads_or(timed_out) != 0;
    fence_after_sync();
    if (any_timeout) {
        const uint32_t warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
        if ((warp & 3u) == 0u && elect_one()) drain_mma(drain_bar + (warp >> 2));
        fence_before_sync();
        __syncthreads();
        fence_after_sync();
    }
    if ((threadIdx.x >> 5) == 0) tmem_dealloc(tmem, fwd_cols(NG));
}

template <bool BF16, bool kSel = false, bool kSplit = false>
__global__ void __launch_bounds__(128 * kFwdGroups, 1) k_field_fwd_tc(DevCfg c, const float* __restrict__ params,
                                                      const float* __restrict__ rays, uint32_t cap,
                                                      const uint32_t* __restrict__ n_total,
                                                      const uint32_t* __restrict__ ray_id,
                                                      const float* __restrict__ ts, float4* __restrict__ sig_rgb,
                                                      uint4* __restrict__ feat_out, float feat_scale,
                                                      uint32_t* __restrict__ err,
                                                      const uint32_t* __restrict__ sel = nullptr,
                                                      const uint32_t* __restrict__ fine = nullptr,
                                                      size_t fine_stride = 0) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t bar[kFwdGroups], drain_bar[kFwdGroups];
    __shared__ uint32_t tslot;
    const uint32_t n = *n_total;
    if (blockIdx.x * 128u >= n) return;
    load_weight_tiles<BF16, 128 * kFwdGroups>(params + (size_t)c.L * c.T * 2, smem, threadIdx.x);
    const uint32_t tmem = fwd_block_setup<kFwdGroups>(&tslot, bar, drain_bar);
    const uint32_t n_tiles = (n + 127) / 128;
    const float2* tables = reinterpret_cast<const float2*>(params);
    uint32_t phase = 0;
    bool timed_out = false;
    const int group = __shfl_sync(0xffffffffu, threadIdx.x >> 7, 0);
    // a group's tiles; the first of every block before the second of any
    for (uint32_t tile = group * gridDim.x + blockIdx.x; tile < n_tiles; tile += kFwdGroups * gridDim.x) {
        const uint32_t i0 = tile * 128;
        fwd_tile<BF16, kSel, kSplit>(c, tables, rays, cap, ray_id, ts, sig_rgb, feat_out, feat_scale, i0, n, smem,
                                     tmem + 64u * group, bar + group, phase, timed_out, sel, fine, fine_stride);
        fence_before_sync();
        if (nb_or(1 + group, 128, timed_out)) {
            timed_out = true;
            if ((threadIdx.x & 127) == 0) atomicOr(err, kErrTimeout);
            break;
        }
        fence_after_sync();
    }
    fwd_block_finish<kFwdGroups>(tmem, drain_bar, timed_out);
}

// ------------------------------------------------------------------ level by level
// A map whose tables do not fit the L2 (levels_split) takes its finest levels, up to 8,
// one after the other over all samples, so that each level's table (or its gradient) stays
// in the L2 while it is used: k_gather_levels before the forward, k_scatter_levels after
// the backward.  The features (MLP type) and dL/dfeat (FP32) of these levels travel
// through the half of the encoding buffer that 16-bit rows leave free.  The work items are
// taken in order of level, tile by tile.  For the floor workload (2^22 entries per
// level, 83.6 M samples) the forward takes 17.3 ms instead of 25.1 and the backward 26.5
// instead of 44.9, whose random sectors come from the HBM.

// x of sample i (0 for i >= n).
__device__ __forceinline__ float3 position_of(const DevCfg& c, const float* __restrict__ rays, uint32_t cap,
                                              const uint32_t* __restrict__ ray_id, const float* __restrict__ ts,
                                              uint32_t i, uint32_t n) {
    float3 d;
    if (i >= n) return make_float3(0.f, 0.f, 0.f);
    return sample_pos_tc(c, rays, cap, __ldcs(ray_id + i), __ldcs(ts + i), d);
}

template <bool BF16>
__global__ void __launch_bounds__(256) k_gather_levels(DevCfg c, const float* __restrict__ params,
                                                       const float* __restrict__ rays, uint32_t cap,
                                                       const uint32_t* __restrict__ n_total,
                                                       const uint32_t* __restrict__ ray_id,
                                                       const float* __restrict__ ts, float feat_scale,
                                                       uint32_t* __restrict__ fine, size_t fine_stride) {
    const uint32_t n = *n_total, n_tiles = (n + 255u) / 256u, l0 = split_level(c.L);
    const uint64_t n_items = (uint64_t)n_tiles * (c.L - l0);
    const float2* tables = reinterpret_cast<const float2*>(params);
    for (uint64_t it = blockIdx.x; it < n_items; it += gridDim.x) {
        const uint32_t k = (uint32_t)(it / n_tiles), tile = (uint32_t)(it - (uint64_t)k * n_tiles);
        const uint32_t i = tile * 256u + (threadIdx.x & ~31u) + pair_sample(threadIdx.x & 31u);
        float f[2];
        encode_level(c, tables, position_of(c, rays, cap, ray_id, ts, i, n), (int)(l0 + k), f);
        if (i < n) __stcs(fine + k * fine_stride + i, pack2<BF16>(f[0] * feat_scale, f[1] * feat_scale));
    }
}

// One item: 2048 samples at one level, 128 walks of 16 samples for each x parity
// (scatter_walk); the positions and dL/dfeat are staged in shared memory.
constexpr uint32_t kScatterTile = 2048;
constexpr int kScatterSmem = kScatterTile * (16 + 8);
__global__ void __launch_bounds__(256) k_scatter_levels(DevCfg c, float* __restrict__ grads,
                                                        const float* __restrict__ rays, uint32_t cap,
                                                        const uint32_t* __restrict__ n_total,
                                                        const uint32_t* __restrict__ ray_id,
                                                        const float* __restrict__ ts,
                                                        const float2* __restrict__ dfine, size_t fine_stride) {
    extern __shared__ __align__(128) uint8_t smem[];
    float4* pos = reinterpret_cast<float4*>(smem);
    float2* df = reinterpret_cast<float2*>(smem + kScatterTile * 16);
    const uint32_t n = *n_total, n_tiles = (n + kScatterTile - 1) / kScatterTile, l0 = split_level(c.L);
    const uint64_t n_items = (uint64_t)n_tiles * (c.L - l0);
    const uint32_t group = threadIdx.x >> 1;
    for (uint64_t it = blockIdx.x; it < n_items; it += gridDim.x) {
        const uint32_t k = (uint32_t)(it / n_tiles), tile = (uint32_t)(it - (uint64_t)k * n_tiles);
        const uint32_t level = l0 + k, i0 = tile * kScatterTile;
#pragma unroll 4
        for (uint32_t r = threadIdx.x; r < kScatterTile; r += 256u) {
            const float3 x = position_of(c, rays, cap, ray_id, ts, i0 + r, n);
            pos[tile_row<16>(r)] = make_float4(x.x, x.y, x.z, 0.f);
            df[tile_row<16>(r) ^ (((r >> 7) & 1u) << 3)] =
                i0 + r < n ? __ldcs(dfine + k * fine_stride + i0 + r) : make_float2(0.f, 0.f);
        }
        __syncthreads();
        ScatterRole s;
        set_level(c, level, s);
        s.p = threadIdx.x & 1u;
        s.r0 = s.rd = 16u * group;
        s.swz = group & 7u;
        s.dx = ((group >> 3) & 1u) << 3;
        const uint32_t left = n - i0;
        const uint32_t m = s.r0 < left ? min(16u, left - s.r0) : 0u;
        float2* gtab = reinterpret_cast<float2*>(grads) + (size_t)level * c.T;
        if (m > 0) {
            if (!unit_box(c)) scatter_walk<2, false>(s, gtab, c.T - 1, pos, df, m);
            else if (s.dense) scatter_walk<1, true>(s, gtab, c.T - 1, pos, df, m);
            else scatter_walk<0, true>(s, gtab, c.T - 1, pos, df, m);
        }
        __syncthreads();
    }
}

// Grouped forward (render of several views of several scenes): the batch's tiles
// are those of its pieces in order (a tile never mixes two pieces); a persistent
// block takes tiles i, i + grid, ...; where a tile belongs to another piece than the
// block's previous one, the block copies that piece's configuration into shared
// memory and, if the scene differs, rounds that scene's weights into the operand
// tiles.  Each tile is then exactly the single-view forward's tile.
// kSel: the pieces' runs s0 .. s0 + n_s - 1 index the selection sel (a render pass).
template <bool BF16, bool kSel = false>
__global__ void __launch_bounds__(128, 4) k_group_fwd_tc(const GroupItem* __restrict__ items, uint32_t n_items,
                                                      const uint32_t* __restrict__ n_tiles_total,
                                                      const float* __restrict__ rays, uint32_t cap,
                                                      const uint32_t* __restrict__ ray_id,
                                                      const float* __restrict__ ts, float4* __restrict__ sig_rgb,
                                                      float feat_scale, uint32_t* __restrict__ err,
                                                      const uint32_t* __restrict__ sel = nullptr) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t bar, drain_bar;
    __shared__ uint32_t tslot;
    __shared__ DevCfg cfg_s;
    __shared__ uint32_t tile0_s[kGroupMaxItems + 1];
    const uint32_t total = *n_tiles_total;
    if (blockIdx.x >= total) return;
    const uint32_t tmem = fwd_block_setup<1>(&tslot, &bar, &drain_bar);
    if (threadIdx.x < n_items) tile0_s[threadIdx.x] = items[threadIdx.x].tile0;
    if (threadIdx.x == 0) tile0_s[n_items] = total;
    __syncthreads();
    const float* cur_params = nullptr;
    uint32_t cur = n_items;  // no piece yet
    uint32_t phase = 0;
    bool timed_out = false;
    for (uint32_t tile = blockIdx.x; tile < total; tile += gridDim.x) {
        uint32_t j = 0;
        while (j + 1 < n_items && tile0_s[j + 1] <= tile) ++j;
        const GroupItem& it = items[j];
        if (j != cur) {
            __syncthreads();  // every thread is done with the previous tile's configuration
            const uint32_t* src = reinterpret_cast<const uint32_t*>(&it.c);
            uint32_t* dst = reinterpret_cast<uint32_t*>(&cfg_s);
            for (uint32_t w = threadIdx.x; w < sizeof(DevCfg) / 4; w += blockDim.x) dst[w] = src[w];
            if (it.params != cur_params)
                load_weight_tiles<BF16, 128>(it.params + (size_t)it.c.L * it.c.T * 2, smem, threadIdx.x);
            cur_params = it.params;
            cur = j;
            to_tensor();      // the weights to the tensor core, the configuration to every thread
        }
        const uint32_t k = (tile - tile0_s[j]) * 128;
        fwd_tile<BF16, kSel>(cfg_s, reinterpret_cast<const float2*>(it.params), rays, cap, ray_id, ts, sig_rgb,
                             nullptr, feat_scale, it.s0 + k, it.s0 + it.n_s, smem, tmem, &bar, phase, timed_out, sel);
        fence_before_sync();
        if (__syncthreads_or(timed_out)) {
            if (threadIdx.x == 0) atomicOr(err, kErrTimeout);
            break;
        }
    }
    fwd_block_finish<1>(tmem, &drain_bar, timed_out);
}

// ------------------------------------------------------------------ backward
// Warp-specialised in three warpgroups: warps 0-3 (the "MLP" group, thread r =
// sample row r = TMEM lane r) run the layer chain on the tensor cores; warps 4-7
// (the "IO" group, thread 128 + r serves row r) load each tile's inputs one tile
// ahead; warps 4-11 (IO and the "SC" group) scatter each finished tile's encoding
// gradient into the tables, by level (scatter_tile), while the MLP group runs the next
// tile.  For 19.5 M samples the chain alone takes 2.3 ms and the scatter alone 4.3,
// as long as both together: the scatter sets the pace, by its issue slots and its reductions.
// Registers are split with setmaxnreg: the block is launched with 80 per thread (two
// blocks of 384 threads per SM), the MLP group takes 96 (its epilogues hold 16 columns
// at a time), the IO group 80 and the SC group 64, which is 240 = 3 x 80; 104 / 80 / 56
// measured 4.34 ms, 104 / 72 / 64 4.39, 128 / 64 / 48 4.62.
// The groups hand tiles over through named barriers:
//   kBarIn      IO -> MLP        the tile's encodings (X0) and row data are in place
//   kBarDfReady MLP -> IO, SC    the chain is done (X0 free) and dL/dfeat is in smem
//   kBarDfFree  IO, SC -> MLP    both scatters of the tile are done (dL/dfeat read)
// All groups walk the same tile list and meet every barrier, whatever happens to
// an MMA wait (a timed-out wait only skips waiting), so no barrier can block.
//
// TMEM columns: [0,64) layer chain, [64,128) dW4, [128,160) dW3, [160,192) dW1,
// [192,208) dW2^T, [208,224) dW5^T.  The weight gradients are M=64 products: row m
// of such an accumulator is TMEM lane 32*(m/16) + m%16.
constexpr uint32_t kColW4 = 64, kColW3 = 128, kColW1 = 160, kColW2T = 192, kColW5T = 208;
constexpr int kBarMlp = 1, kBarIn = 2, kBarDfReady = 3, kBarDfFree = 4;
constexpr int kBwdThreads = 384;            // MLP, IO and SC warpgroups
constexpr uint32_t kRegMlp = 96, kRegIo = 80, kRegSc = 64;
static_assert(128 * (kRegMlp + kRegIo + kRegSc) == kBwdThreads * 80,
              "the setmaxnreg split must add up to the launch allocation (80 registers per thread)");
constexpr int kDfBytes = 128 * 32 * 4;      // dL/dfeat, [level][row] float2
constexpr int kRowBytes = 128 * 32;         // row data: {d.xyz, valid}, {dz0, dz1, dz2, dL/dsigma}
constexpr int kXBytes = 2 * 128 * 16;       // sample positions (x, valid) of the tiles, by parity
constexpr int kBwdSmem = kWB + kT32 + kT64 + kT32 + kT64 + kT64 + kT16 + kDfBytes + kRowBytes + kXBytes;  // 114688

namespace {

// ReLU branches of 32 consecutive columns in one word: bit 15 - j is column 2 j's,
// bit 31 - j column 2 j + 1's.
//
// 64 accumulator columns -> relu(scale * a) into a 64-column tile; the branch of each
// column (a * scale > 0) is returned in two words.  n = 0 - scale * a has its sign bit
// set exactly where the branch is taken (a zero of either sign gives +0), so each
// branch is one funnel shift; the columns come 16 at a time, as more do not fit the
// chain's registers.
template <bool BF16>
__device__ __forceinline__ void relu_epilogue(uint32_t trow, uint8_t* tile, int r, float scale, uint32_t* m) {
    float v[16];
    uint32_t me = 0, mo = 0;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        ld_cols<16>(trow, 16 * h, v);
#pragma unroll
        for (int k = 0; k < 16; k += 2) {
            const float ne = fmaf(v[k], -scale, 0.f), no = fmaf(v[k + 1], -scale, 0.f);
            me = __funnelshift_l(__float_as_uint(ne), me, 1);
            mo = __funnelshift_l(__float_as_uint(no), mo, 1);
            v[k] = -ne;
            v[k + 1] = -no;
        }
        store_row_at<BF16, 16, true>(tile, r, 16 * h, v);
        if (h & 1) m[h >> 1] = __byte_perm(me, mo, 0x5410);
    }
}

// 0xffff in each half of the word whose top bit is set (prmt's sign replication of bytes
// 1 and 3).
__device__ __forceinline__ uint32_t sign_halves(uint32_t x) {
    uint32_t d;
    asm("prmt.b32 %0, %1, 0, 0xBB99;" : "=r"(d) : "r"(x));
    return d;
}

// 64 accumulator columns masked by the ReLU branches into a 64-column tile: the packed
// pair's mask is the sign of two bytes of the shifted word.
template <bool BF16>
__device__ __forceinline__ void mask_epilogue(uint32_t trow, uint8_t* tile, int r, const uint32_t* m) {
    float v[16];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        ld_cols<16>(trow, 16 * h, v);
        uint32_t q[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            q[j] = pack2<BF16>(v[2 * j], v[2 * j + 1]) & sign_halves(m[h >> 1] * (1u << (8 * (h & 1) + j)));
#pragma unroll
        for (int g = 0; g < 2; ++g)
            *reinterpret_cast<uint4*>(tile + tile_offset(r, 16 * h + 8 * g, 128)) =
                make_uint4(q[4 * g], q[4 * g + 1], q[4 * g + 2], q[4 * g + 3]);
    }
}

// dL/dp (world position) through the levels l0, l0 + 2, ... of a tile's samples, by the 128
// threads r of a warpgroup, to out[stride * sample].
__device__ __forceinline__ void pose_terms(const DevCfg& c, const float* __restrict__ params, const float4* pos,
                                           const float2* df, int r, int l0, uint32_t i0, uint32_t n,
                                           float4* __restrict__ out, uint32_t stride) {
    const uint32_t row = (r & ~31) + pair_sample(r & 31);
    const float4 x = pos[tile_row<16>(row)];
    const float3 g = hash_grad_x(c, reinterpret_cast<const float2*>(params), make_float3(x.x, x.y, x.z),
                                 [&](int l) { return df[tile_df<16>(row, l)]; }, l0);
    if (i0 + row < n)
        out[stride * (size_t)(i0 + row)] = make_float4(g.x * c.inv_size, g.y * c.inv_size, g.z * c.inv_size, 0.f);
}

}  // namespace

// kPose: also writes, per sample, dL/dp (world position) through the even levels (IO
// group) into pose_s[2 i] and through the odd ones (SC group) into pose_odd[i], and the
// view-direction gradient through the SH encoding (MLP group) into pose_s[2 i + 1].
// G: samples per scatter walk (8: at most 8 levels scattered here).  kSplit: the levels
// from split_level(c.L) on go to dfine instead, for k_scatter_levels.
template <bool BF16, bool kPose, int G, bool kSplit>
__global__ void __launch_bounds__(kBwdThreads, 2) k_field_bwd_tc(DevCfg c, const float* __restrict__ params,
                                                         float* __restrict__ grads, const float* __restrict__ rays,
                                                         uint32_t cap, const uint32_t* __restrict__ n_total,
                                                         const uint32_t* __restrict__ ray_id,
                                                         const float* __restrict__ ts, const uint4* __restrict__ feat,
                                                         const float4* __restrict__ sig_rgb,
                                                         const float4* __restrict__ dsig_rgb, float feat_scale,
                                                         const float* __restrict__ seed_max,
                                                         float4* __restrict__ pose_s, float4* __restrict__ pose_odd,
                                                         float2* __restrict__ dfine, size_t fine_stride,
                                                         uint32_t* __restrict__ err) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t bar, drain_bar;
    __shared__ uint32_t tslot;
    uint8_t* tX0 = smem + kWB;   // 128 x 32, written by the IO group
    uint8_t* tH1 = tX0 + kT32;   // 128 x 64  (later G1)
    uint8_t* tX3 = tH1 + kT64;   // 128 x 32  (later G2 in columns 0..15)
    uint8_t* tH3 = tX3 + kT32;   // 128 x 64  (later G3)
    uint8_t* tH4 = tH3 + kT64;   // 128 x 64  (later G4)
    uint8_t* tG5 = tH4 + kT64;   // 128 x 16
    uint8_t* sDf = tG5 + kT16;   // dL/dfeat: [16 levels][128 rows] float2
    float4* sRow = reinterpret_cast<float4*>(sDf + kDfBytes);  // [128][2]
    float4* sX = sRow + 2 * 128;                                // [2][128]: (x, valid) of tile k at k & 1
    const float2* sDf2 = reinterpret_cast<const float2*>(sDf);

    constexpr uint32_t kOX0 = kWB, kOH1 = kOX0 + kT32, kOX3 = kOH1 + kT64, kOH3 = kOX3 + kT32, kOH4 = kOH3 + kT64,
                       kOG5 = kOH4 + kT64;
    using X0K = KMaj<kOX0, 128>;
    using H1K = KMaj<kOH1, 128>;
    using X3K = KMaj<kOX3, 128>;
    using H3K = KMaj<kOH3, 128>;
    using H4K = KMaj<kOH4, 128>;
    using G5K = KMaj<kOG5, 128>;
    using X0M = MnMaj<kOX0, 128>;
    using H1M = MnMaj<kOH1, 128>;
    using X3M = MnMaj<kOX3, 128>;
    using H3M = MnMaj<kOH3, 128>;
    using H4M = MnMaj<kOH4, 128>;
    using G5M = MnMaj<kOG5, 128>;

    const uint32_t n = *n_total;
    if (blockIdx.x * 128u >= n) return;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), r = tid & 127;
    load_weight_tiles<BF16, kBwdThreads>(params + (size_t)c.L * c.T * 2, smem, tid);
    if (warp == 0) tmem_alloc(&tslot, 256);
    if (tid == 0) {
        mbar_init(&bar, 1);
        mbar_init(&drain_bar, 1);
        mbar_fence_init();
    }
    to_tensor();
    const uint32_t tmem = tslot;
    const uint32_t n_tiles = (n + 127) / 128;
    const uint32_t n_mine = blockIdx.x < n_tiles ? (n_tiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    const float gm_d = seed_max[1], gm_c = seed_max[2];
    const float gm_dc = fmaxf(gm_d, gm_c);
    const float S = gm_dc > 0.f ? exp2f(fminf(fmaxf(floorf(log2f(kGradTarget / gm_dc)), -100.f), 100.f)) : 1.f;
    const float Sc = gm_c > 0.f ? exp2f(fminf(fmaxf(floorf(log2f(kGradTarget / gm_c)), -100.f), 100.f)) : S;
    const float inv_S = 1.f / S, inv_Sc = 1.f / Sc;
    const float c_to_d = S * inv_Sc;  // power of two: exact
    const uint32_t n_lev = kSplit ? split_level(c.L) : c.L;  // levels scattered here
    static_assert(!kPose || G == 16, "the pose terms read dL/dfeat in the order of G = 16");
    bool timed_out = false;

    if (warp < 4) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(kRegMlp));
        // ======================= MLP group: the layer chain on the tensor cores
        const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
        const float inv_fs = 1.f / feat_scale;
        uint32_t phase = 0;
        const uint32_t base4 = smem_u32(smem) >> 4;
        for (uint32_t k = 0; k < n_mine; ++k) {
            nb_sync(kBarIn, 256);
            const float4 rd = sRow[2 * r], rz = sRow[2 * r + 1];
            const bool valid = rd.w != 0.f;
            float v[32];
            uint32_t m1[2], m3[2], m4[2];
            // ---- forward recompute (same arithmetic as the forward kernel)
            to_tensor_group(kBarMlp);
            if (warp == 0 && elect_one()) {
                gemm<BF16, 128, 64, X0K, W1K, 2>(tmem, base4, base4, false);
                mma_commit(&bar);
            }
            wait_mma(&bar, phase, timed_out, c.wait_polls);
            relu_epilogue<BF16>(trow, tH1, r, inv_fs, m1);
            to_tensor_group(kBarMlp);
            if (warp == 0 && elect_one()) {
                gemm<BF16, 128, 16, H1K, W2K, 4>(tmem, base4, base4, false);
                mma_commit(&bar);
            }
            wait_mma(&bar, phase, timed_out, c.wait_polls);
            float y[32];
            ld_cols<16>(trow, 0, y);
            const float sigma = expf(fminf(y[0], kSigmaHMax));
            const float sig_grad = y[0] < kSigmaHMax ? sigma : 0.f;
            if (valid) sh16(rd.x, rd.y, rd.z, y + kGeo);
            else {
#pragma unroll
                for (int q = kGeo; q < 32; ++q) y[q] = 0.f;
            }
            store_row_at<BF16, 32>(tX3, r, 0, y);
            to_tensor_group(kBarMlp);
            if (warp == 0 && elect_one()) {
                gemm<BF16, 128, 64, X3K, W3K, 2>(tmem, base4, base4, false);
                mma_commit(&bar);
            }
            wait_mma(&bar, phase, timed_out, c.wait_polls);
            relu_epilogue<BF16>(trow, tH3, r, 1.f, m3);
            to_tensor_group(kBarMlp);
            if (warp == 0 && elect_one()) {
                gemm<BF16, 128, 64, H3K, W4K, 4>(tmem, base4, base4, false);
                mma_commit(&bar);
            }
            wait_mma(&bar, phase, timed_out, c.wait_polls);
            relu_epilogue<BF16>(trow, tH4, r, 1.f, m4);
            // the colours' gradient seed dz (FP32, scaled by S) comes from the IO group
            v[0] = rz.x;
            v[1] = rz.y;
            v[2] = rz.z;
#pragma unroll
            for (int q = 3; q < 16; ++q) v[q] = 0.f;
            store_row_at<BF16, 16>(tG5, r, 0, v);
            // ---- backward: dW5^T += H4^T G5 ; dH4 = G5 W5
            to_tensor_group(kBarMlp);
            if (warp == 0 && elect_one()) {
                gemm<BF16, 64, 16, H4M, G5M, 8>(tmem + kColW5T, base4, base4, k > 0);
                gemm<BF16, 128, 64, G5K, W5M, 1>(tmem, base4, base4, false);
                mma_commit(&bar);
            }
            wait_mma(&bar, phase, timed_out, c.wait_polls);
            mask_epilogue<BF16>(trow, tH4, r, m4);                 // G4
            // dW4 += G4^T H3 ; dH3 = G4 W4
            to_tensor_group(kBarMlp);
            if (warp == 0 && elect_one()) {
                gemm<BF16, 64, 64, H4M, H3M, 8>(tmem + kColW4, base4, base4, k > 0);
                gemm<BF16, 128, 64, H4K, W4M, 4>(tmem, base4, base4, false);
                mma_commit(&bar);
            }
            wait_mma(&bar, phase, timed_out, c.wait_polls);
            mask_epilogue<BF16>(trow, tH3, r, m3);                 // G3
            // dW3 += G3^T X3 ; dX3 = G3 W3
            to_tensor_group(kBarMlp);
            if (warp == 0 && elect_one()) {
                gemm<BF16, 64, 32, H3M, X3M, 8>(tmem + kColW3, base4, base4, k > 0);
                gemm<BF16, 128, 32, H3K, W3M, 4>(tmem, base4, base4, false);
                mma_commit(&bar);
            }
            wait_mma(&bar, phase, timed_out, c.wait_polls);
            if (kPose) {
                // the SH inputs' gradient (columns 16..31, colour scale) -> view direction
                ld_cols<16>(trow, 16, v);
#pragma unroll
                for (int q = 0; q < 16; ++q) v[q] *= inv_Sc;
                const float3 gd = sh16_vjp(rd.x, rd.y, rd.z, v);
                const uint32_t i = (blockIdx.x + k * gridDim.x) * 128 + r;
                if (valid) pose_s[2 * (size_t)i + 1] = make_float4(gd.x, gd.y, gd.z, 0.f);
            }
            ld_cols<16>(trow, 0, v);
#pragma unroll
            for (int q = 0; q < 16; ++q) v[q] *= c_to_d;                // colour scale -> density scale
            v[0] += S * rz.w * sig_grad;                                 // dL/dh_0 += dL/dsigma * dsigma/dh_0
            store_row_at<BF16, 16>(tX3, r, 0, v);                        // G2 (columns 0..15)
            // dW2^T += H1^T G2 ; dH1 = G2 W2
            to_tensor_group(kBarMlp);
            if (warp == 0 && elect_one()) {
                gemm<BF16, 64, 16, H1M, X3M, 8>(tmem + kColW2T, base4, base4, k > 0);
                gemm<BF16, 128, 64, X3K, W2M, 1>(tmem, base4, base4, false);
                mma_commit(&bar);
            }
            wait_mma(&bar, phase, timed_out, c.wait_polls);
            mask_epilogue<BF16>(trow, tH1, r, m1);                 // G1
            // dW1 += G1^T X0 ; dF = G1 W1
            to_tensor_group(kBarMlp);
            if (warp == 0 && elect_one()) {
                gemm<BF16, 64, 32, H1M, X0M, 8>(tmem + kColW1, base4, base4, k > 0);
                gemm<BF16, 128, 32, H1K, W1M, 4>(tmem, base4, base4, false);
                mma_commit(&bar);
            }
            wait_mma(&bar, phase, timed_out, c.wait_polls);
            ld_cols<32>(trow, 0, v);
            fence_before_sync();
            if (k > 0) nb_sync(kBarDfFree, kBwdThreads);  // both scatters of the previous tile are done
#pragma unroll
            for (int q = 0; q < 16; ++q)
                if (!kSplit || q < 8)
                    reinterpret_cast<float2*>(sDf)[tile_df<G>(r, q)] = make_float2(v[2 * q] * inv_S, v[2 * q + 1] * inv_S);
            if constexpr (kSplit) {
                const uint32_t i = (blockIdx.x + k * gridDim.x) * 128 + r;
                const int l0 = (int)split_level(c.L);
                if (i < n) {
#pragma unroll
                    for (int q = 0; q < 16; ++q)
                        if (q >= l0 && q < (int)c.L)
                            __stcs(dfine + (size_t)(q - l0) * fine_stride + i,
                                   make_float2(v[2 * q] * inv_S, v[2 * q + 1] * inv_S));
                }
            }
            nb_arrive(kBarDfReady, kBwdThreads);          // also: X0 and the row data are free
        }
        // ---- flush the weight gradients (lane 32*(m/16) + m%16 holds row m)
        const bool any_timeout = __syncthreads_or(timed_out) != 0;  // all three groups take part
        fence_after_sync();
        if (any_timeout && warp == 0 && elect_one()) drain_mma(&drain_bar);  // the thread that issued every MMA
        if (n_mine > 0 && !any_timeout) {
            float* gm_ = grads + (size_t)c.L * c.T * 2;
            const int lane = tid & 31;
            const int m = warp * 16 + lane;
            const bool has = lane < 16;
            float w[32];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                ld_cols<32>(trow, kColW4 + 32 * h, w);
                if (has)
                    for (int q = 0; q < 32; ++q) atomicAdd(gm_ + kOffW4 + m * 64 + 32 * h + q, w[q] * inv_Sc);
            }
            ld_cols<32>(trow, kColW3, w);
            if (has)
                for (int q = 0; q < 32; ++q) atomicAdd(gm_ + kOffW3 + m * 32 + q, w[q] * inv_Sc);
            ld_cols<32>(trow, kColW1, w);
            if (has)
                for (int q = 0; q < 32; ++q) atomicAdd(gm_ + kOffW1 + m * 32 + q, w[q] * inv_S * inv_fs);
            ld_cols<16>(trow, kColW2T, w);
            if (has)
                for (int q = 0; q < 16; ++q) atomicAdd(gm_ + kOffW2 + q * 64 + m, w[q] * inv_S);
            ld_cols<16>(trow, kColW5T, w);
            if (has)
                for (int q = 0; q < 3; ++q) atomicAdd(gm_ + kOffW5 + q * 64 + m, w[q] * inv_Sc);
        }
        if (any_timeout && tid == 0) atomicOr(err, kErrTimeout);
    } else if (warp >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kRegSc));
        // ======================= SC group: its half of the levels' gradient scatter
        const uint32_t level = G == 16 ? scatter_level(c, 128u + r) : 0u;
        for (uint32_t k = 0; k < n_mine; ++k) {
            nb_sync(kBarDfReady, kBwdThreads);
            const uint32_t i0 = (blockIdx.x + k * gridDim.x) * 128;
            const float4* pos = sX + (k & 1u) * 128;
            scatter_tile<G>(c, reinterpret_cast<float2*>(grads), 128u + r, level, n_lev, pos, sDf2, n - i0);
            if (kPose) pose_terms(c, params, pos, sDf2, r, 1, i0, n, pose_odd, 1);
            if (k + 1 < n_mine) nb_arrive(kBarDfFree, kBwdThreads);
        }
        __syncthreads_or(false);                      // pairs with the MLP group's flush barrier
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kRegIo));
        // ======================= IO group: tile inputs one tile ahead, its half of the scatter
        const uint32_t level = G == 16 ? scatter_level(c, r) : 0u;
        float3 x_next = make_float3(0.f, 0.f, 0.f);
        bool valid_next = false;
        uint4 f_next[4];
        float4 rd_next, rz_next;
        // inputs of this block's k-th tile for row r, into registers
        auto load = [&](uint32_t k) {
            const uint32_t i = (blockIdx.x + k * gridDim.x) * 128 + r;
            valid_next = i < n;
            float3 d = make_float3(0.f, 0.f, 0.f);
            x_next = make_float3(0.f, 0.f, 0.f);
            rd_next = make_float4(0.f, 0.f, 0.f, 0.f);
            rz_next = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int q = 0; q < 4; ++q) f_next[q] = make_uint4(0u, 0u, 0u, 0u);
            if (valid_next) {
                x_next = sample_pos_tc(c, rays, cap, ray_id[i], ts[i], d);
                const float4 g = dsig_rgb[i], col = sig_rgb[i];
#pragma unroll
                for (int q = 0; q < 4; ++q) f_next[q] = feat[(size_t)i * 4 + q];
                rd_next = make_float4(d.x, d.y, d.z, 1.f);
                rz_next = make_float4(Sc * g.y * col.y * (1.f - col.y), Sc * g.z * col.z * (1.f - col.z),
                                      Sc * g.w * col.w * (1.f - col.w), g.x);
            }
        };
        // the inputs of tile kk into the operand tile and the row data (and its sample
        // positions for the SC group)
        auto publish = [&](uint32_t kk) {
            sX[(kk & 1u) * 128 + tile_row<G>(r)] = make_float4(x_next.x, x_next.y, x_next.z, valid_next ? 1.f : 0.f);
#pragma unroll
            for (int q = 0; q < 4; ++q) *reinterpret_cast<uint4*>(tX0 + tile_offset(r, 8 * q, 128)) = f_next[q];
            sRow[2 * r] = rd_next;
            sRow[2 * r + 1] = rz_next;
            fence_proxy_async();                      // X0 is read by the tensor core
            nb_arrive(kBarIn, 256);
        };
        if (n_mine > 0) {
            load(0);
            publish(0);
        }
        for (uint32_t k = 0; k < n_mine; ++k) {
            if (k + 1 < n_mine) load(k + 1);          // global loads in flight during the chain
            nb_sync(kBarDfReady, kBwdThreads);
            if (k + 1 < n_mine) publish(k + 1);       // next tile's inputs; the MLP group starts on it
            const uint32_t i0 = (blockIdx.x + k * gridDim.x) * 128;
            const float4* pos = sX + (k & 1u) * 128;
            scatter_tile<G>(c, reinterpret_cast<float2*>(grads), r, level, n_lev, pos, sDf2, n - i0);
            if (kPose) pose_terms(c, params, pos, sDf2, r, 0, i0, n, pose_s, 2);
            if (k + 1 < n_mine) nb_arrive(kBarDfFree, kBwdThreads);  // dL/dfeat read: the MLP group may overwrite it
        }
        __syncthreads_or(false);                      // pairs with the MLP group's flush barrier
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == 0) tmem_dealloc(tmem, 256);
}

// ------------------------------------------------------------------ launchers

// Whether a step's finest levels are taken level by level: where the tables are larger than
// the L2.  131 k rays (10 M samples), forward + backward: at 16 levels of 2^20 entries
// 2.1 + 2.3 ms as they are, 1.9 + 3.3 level by level; at 2^21 2.7 + 3.8 and 2.0 + 3.3, at
// 2^22 3.2 + 5.6 and 2.2 + 3.5.  Small batches stay as they are: their two more launches
// cost what they save (at 2^22, 81 k samples: 0.047 + 0.104 and 0.043 + 0.108; 322 k:
// 0.121 + 0.208 and 0.094 + 0.223; 653 k: 0.221 + 0.364 and 0.158 + 0.340).
bool levels_split(const DevCfg& c, uint32_t n_rays) {
    int dev = 0, l2 = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
    return (uint64_t)c.L * c.T * sizeof(float2) > (uint64_t)l2 && (uint64_t)n_rays * c.max_samples >= (1u << 19);
}

// The half of the encoding buffer that 16-bit rows leave free: 64 bytes per sample.
static void* fine_buffer(const StepBufs& b) { return b.feat + 16 * b.cap_samples; }

template <bool BF16>
static void fwd_tc(const DevCfg& c, const float* params, uint32_t n_rays, const StepBufs& b, bool store_feat,
                   int n_sm, cudaStream_t s) {
    const float fs = BF16 ? 1.f : 256.f;
    uint4* feat = store_feat ? reinterpret_cast<uint4*>(b.feat) : nullptr;
    // per call: the attribute belongs to the current device (cheap next to the kernel)
    if (store_feat && levels_split(c, n_rays)) {
        uint32_t* fine = static_cast<uint32_t*>(fine_buffer(b));
        k_gather_levels<BF16><<<n_sm * 6, 256, 0, s>>>(c, params, b.rays, b.cap_rays, b.offsets + n_rays, b.ray_id, b.t,
                                                       fs, fine, b.cap_samples);
        cudaFuncSetAttribute(k_field_fwd_tc<BF16, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmemN);
        k_field_fwd_tc<BF16, false, true><<<n_sm, 128 * kFwdGroups, kFwdSmemN, s>>>(
            c, params, b.rays, b.cap_rays, b.offsets + n_rays, b.ray_id, b.t, b.sig_rgb, feat, fs, b.err, nullptr, fine,
            b.cap_samples);
        return;
    }
    cudaFuncSetAttribute(k_field_fwd_tc<BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmemN);
    k_field_fwd_tc<BF16><<<n_sm, 128 * kFwdGroups, kFwdSmemN, s>>>(c, params, b.rays, b.cap_rays, b.offsets + n_rays,
                                                          b.ray_id, b.t, b.sig_rgb, feat, fs, b.err);
}

template <bool BF16, bool kPose, int G, bool kSplit>
static void bwd_launch(const DevCfg& c, const float* params, float* grads, uint32_t n_rays, const StepBufs& b, int n_sm,
                       cudaStream_t s) {
    // per call: the attribute belongs to the current device (cheap next to the kernel)
    cudaFuncSetAttribute(k_field_bwd_tc<BF16, kPose, G, kSplit>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwdSmem);
    const float fs = BF16 ? 1.f : 256.f;
    k_field_bwd_tc<BF16, kPose, G, kSplit><<<n_sm * 2, kBwdThreads, kBwdSmem, s>>>(
        c, params, grads, b.rays, b.cap_rays, b.offsets + n_rays, b.ray_id, b.t, reinterpret_cast<const uint4*>(b.feat),
        b.sig_rgb, b.dsig_rgb, fs, b.loss, kPose ? b.pose_s : nullptr, kPose ? b.pose_odd : nullptr,
        kSplit ? static_cast<float2*>(fine_buffer(b)) : nullptr, b.cap_samples, b.err);
}

template <bool BF16, bool kPose>
static void bwd_tc(const DevCfg& c, const float* params, float* grads, uint32_t n_rays, const StepBufs& b, int n_sm,
                   cudaStream_t s) {
    if constexpr (kPose) {
        bwd_launch<BF16, true, 16, false>(c, params, grads, n_rays, b, n_sm, s);
    } else if (levels_split(c, n_rays)) {
        bwd_launch<BF16, false, 8, true>(c, params, grads, n_rays, b, n_sm, s);
        cudaFuncSetAttribute(k_scatter_levels, cudaFuncAttributeMaxDynamicSharedMemorySize, kScatterSmem);
        k_scatter_levels<<<n_sm * 4, 256, kScatterSmem, s>>>(c, grads, b.rays, b.cap_rays, b.offsets + n_rays, b.ray_id,
                                                             b.t, static_cast<const float2*>(fine_buffer(b)),
                                                             b.cap_samples);
    } else if (c.L <= 8) {
        bwd_launch<BF16, false, 8, false>(c, params, grads, n_rays, b, n_sm, s);
    } else {
        bwd_launch<BF16, false, 16, false>(c, params, grads, n_rays, b, n_sm, s);
    }
}

template <bool BF16>
static void fwd_tc_sel(const DevCfg& c, const float* params, const uint32_t* sel, const uint32_t* n_sel,
                       const StepBufs& b, int n_sm, cudaStream_t s) {
    cudaFuncSetAttribute(k_field_fwd_tc<BF16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmemN);
    const float fs = BF16 ? 1.f : 256.f;
    k_field_fwd_tc<BF16, true><<<n_sm, 128 * kFwdGroups, kFwdSmemN, s>>>(c, params, b.rays, b.cap_rays, n_sel, b.ray_id, b.t,
                                                                b.sig_rgb, nullptr, fs, b.err, sel);
}

void launch_field_fwd_tc_sel(const DevCfg& c, const float* params, const uint32_t* sel, const uint32_t* n_sel,
                             const StepBufs& b, bool bf16, int n_sm, cudaStream_t s) {
    if (bf16) fwd_tc_sel<true>(c, params, sel, n_sel, b, n_sm, s);
    else fwd_tc_sel<false>(c, params, sel, n_sel, b, n_sm, s);
}

void launch_field_fwd_tc(const DevCfg& c, const float* params, uint32_t n_rays, const StepBufs& b, bool store_feat,
                         bool bf16, int n_sm, cudaStream_t s) {
    if (bf16) fwd_tc<true>(c, params, n_rays, b, store_feat, n_sm, s);
    else fwd_tc<false>(c, params, n_rays, b, store_feat, n_sm, s);
}

template <bool BF16, bool kSel>
static void group_fwd(const GroupItem* items, uint32_t n_items, const uint32_t* n_tiles, const StepBufs& b,
                      const uint32_t* sel, int n_sm, cudaStream_t s) {
    cudaFuncSetAttribute(k_group_fwd_tc<BF16, kSel>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem);
    k_group_fwd_tc<BF16, kSel><<<n_sm * 4, 128, kFwdSmem, s>>>(items, n_items, n_tiles, b.rays, b.cap_rays, b.ray_id,
                                                                b.t, b.sig_rgb, BF16 ? 1.f : 256.f, b.err, sel);
}

void launch_group_fwd_tc(const GroupItem* items, uint32_t n_items, const uint32_t* n_tiles, const StepBufs& b,
                         bool bf16, int n_sm, cudaStream_t s, const uint32_t* sel) {
    if (sel) {
        if (bf16) group_fwd<true, true>(items, n_items, n_tiles, b, sel, n_sm, s);
        else group_fwd<false, true>(items, n_items, n_tiles, b, sel, n_sm, s);
    } else {
        if (bf16) group_fwd<true, false>(items, n_items, n_tiles, b, sel, n_sm, s);
        else group_fwd<false, false>(items, n_items, n_tiles, b, sel, n_sm, s);
    }
}

void launch_field_bwd_tc(const DevCfg& c, const float* params, float* grads, uint32_t n_rays, const StepBufs& b,
                         bool bf16, int n_sm, cudaStream_t s, bool pose) {
    if (pose) {
        if (bf16) bwd_tc<true, true>(c, params, grads, n_rays, b, n_sm, s);
        else bwd_tc<false, true>(c, params, grads, n_rays, b, n_sm, s);
    } else {
        if (bf16) bwd_tc<true, false>(c, params, grads, n_rays, b, n_sm, s);
        else bwd_tc<false, false>(c, params, grads, n_rays, b, n_sm, s);
    }
}

}  // namespace nm
