// encoding.cuh - multiresolution hash-grid encoding and its gradient scatter
// (step a3 / a11).  The grid is the Instant-NGP encoding the paper uses as its map
// (Sec. 3.4): per level l, the sample's cell at resolution N_l, the 8 corner slots
// (dense index or spatial hash), and trilinear interpolation of 2 FP32 features.
#pragma once

#include "common.cuh"

namespace nm {

// Trilinear corner weight of corner k = bx + 2 by + 4 bz.
__device__ __forceinline__ float corner_weight(int k, float wx, float wy, float wz) {
    return ((k & 1) ? wx : 1.f - wx) * ((k & 2) ? wy : 1.f - wy) * ((k & 4) ? wz : 1.f - wz);
}

// The sample of a warp's 32 that lane `lane` encodes: lanes 2 i and 2 i + 1 have samples i
// and 16 + i (encode_level's loads then cover 16 consecutive samples each).
__device__ __forceinline__ uint32_t pair_sample(uint32_t lane) { return (lane >> 1) + 16u * (lane & 1u); }

// Table values around grid position x at level l, the 4 (y, z) pairs of this lane's corners
// (lower and upper in x), and the offsets w; called by all 32 lanes, whose positions follow
// pair_sample.  tables: [L][T] float2.  The gathers are bound by the
// 128-byte lines their instructions touch in the L1 (39.5 wavefronts per sample at 73 % of
// the data pipe when every lane read its own corners, odd x pairs in two instructions).
// Corners k and k + 1 (k even) differ only in x and share a line 15 times in 16, so one
// instruction reads both: the even lane the lower corner of its own sample and, in a second
// instruction, the upper one of its neighbour's; the odd lane likewise.  Each then gets
// its upper corner by a shuffle.  That is 27.7 lines per sample on the room workload's
// rays instead of 43.7 (counted on the host); forward of 19.5 M samples 3.36 ms,
// 3.66 before (2.82 with the groups that share the weights).
__device__ __forceinline__ void level_corners(const DevCfg& c, const float2* __restrict__ tables, float3 x, int l,
                                              float2* lo, float2* up, float* w) {
    const uint32_t N = c.res[l], Tmask = c.T - 1;
    const bool dense = (c.dense_mask >> l) & 1u;
    const bool odd = threadIdx.x & 1u;
    const uint32_t m1 = dense ? N + 1u : 2654435761u, m2 = dense ? (N + 1u) * (N + 1u) : 805459861u;
    uint32_t cx, cy, cz;
    level_cell(x.x, N, cx, w[0]);
    level_cell(x.y, N, cy, w[1]);
    level_cell(x.z, N, cz, w[2]);
    const uint32_t ya = cy * m1, za = cz * m2;
    const uint32_t xn = __shfl_xor_sync(0xffffffffu, cx, 1), yn = __shfl_xor_sync(0xffffffffu, ya, 1),
                   zn = __shfl_xor_sync(0xffffffffu, za, 1);
    // instruction 0: the even lane's sample, 1: the odd lane's
    const uint32_t X[2] = {odd ? xn + 1u : cx, odd ? cx : xn + 1u};
    const uint32_t Y[2] = {odd ? yn : ya, odd ? ya : yn}, Z[2] = {odd ? zn : za, odd ? za : zn};
    const float2* tab = tables + (size_t)l * c.T;
    float2 v[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t a = Y[i] + (j & 1) * m1, b = Z[i] + (j >> 1) * m2;
            const uint32_t s = dense ? X[i] + a + b : (X[i] ^ a ^ b) & Tmask;
            v[i][j] = __ldg(tab + s);
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 snd = odd ? v[0][j] : v[1][j];
        lo[j] = odd ? v[1][j] : v[0][j];
        up[j] = make_float2(__shfl_xor_sync(0xffffffffu, snd.x, 1), __shfl_xor_sync(0xffffffffu, snd.y, 1));
    }
}

// Features of level l of grid position x into f[0], f[1] (whole warps, pair_sample order):
// the corners in the order k = 0 .. 7, each times its weight.
__device__ __forceinline__ void encode_level(const DevCfg& c, const float2* __restrict__ tables, float3 x, int l,
                                             float* f) {
    float2 lo[4], up[4];
    float w[3];
    level_corners(c, tables, x, l, lo, up, w);
    float a0 = 0.f, a1 = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float w0 = corner_weight(2 * j, w[0], w[1], w[2]);
        const float w1 = corner_weight(2 * j + 1, w[0], w[1], w[2]);
        a0 += w0 * lo[j].x;
        a1 += w0 * lo[j].y;
        a0 += w1 * up[j].x;
        a1 += w1 * up[j].y;
    }
    f[0] = a0;
    f[1] = a1;
}

// Features of levels l0 .. l0 + kGatherGroup - 1 into f[0 .. 2 kGatherGroup) (zero for
// levels >= L), one level after the other: loads of 4 or 2 levels in flight spilled
// registers in the tensor-core forward (3.18 and 3.08 ms against 3.03).
constexpr int kGatherGroup = 4;

__device__ __forceinline__ void encode_group(const DevCfg& c, const float2* __restrict__ tables, float3 x,
                                             int l0, float* f) {
#pragma unroll
    for (int g = 0; g < kGatherGroup; ++g) {
        if (l0 + g < (int)c.L) {
            encode_level(c, tables, x, l0 + g, f + 2 * g);
        } else {
            f[2 * g] = 0.f;
            f[2 * g + 1] = 0.f;
        }
    }
}

// Encodes grid position x into f[0 .. 2L) (f[2L .. 32) set to zero).
__device__ __forceinline__ void hash_encode(const DevCfg& c, const float2* __restrict__ tables,
                                            float3 x, float* f) {
#pragma unroll
    for (int l0 = 0; l0 < kEnc / 2; l0 += kGatherGroup) encode_group(c, tables, x, l0, f + 2 * l0);
}

// ---------------------------------------------------------------- tile scatter
// dL/dtable of a 128-sample tile (both backward kernels): 256 threads, thread st
// walks the 16 consecutive samples 16 g .. 16 g + 15 of the tile at one level, for the
// vertices whose x coordinate has parity p.  Consecutive samples lie on a ray, so they
// share vertices: at the coarse levels the whole cell, and where a step crosses one
// face still 4 of its 8 vertices.  Each sample's cell has exactly one vertex per parity
// of (x, y, z), so a vertex keeps its accumulator (parity of y and z) and its lane
// (parity of x) for as long as the samples touch it; the sum leaves with one 8-byte
// reduction when the ray moves on.  Two lanes p = 0, 1 side by side flush x-adjacent
// vertices in one instruction, which share a 32-byte sector 3 times in 4.
// Per sample this issues 48.4 reductions in 33.3 sectors on the room workload's rays
// (counted on the host), against 61.4 in 52.2 for sums over runs of equal cells within
// a warp, and needs no shuffle at all: the backward of 19.5 M samples takes 4.29 ms
// instead of 6.74.  It issues in 0.62 of the cycles, with the integer pipe at 0.43.
// Walks of G = 16 samples: 8 groups and 2 parities per level, two levels per warp.  With at
// most 8 levels to scatter (G = 8): 16 groups of 8 samples, one level per warp.
struct ScatterRole {
    uint32_t N, m1, m2, p;      // resolution, y and z strides (or hash primes), x parity
    uint32_t r0, rd, swz, dx;   // first sample row; first dL/dfeat place; permutation of the walk's rows (and of dL/dfeat's)
    bool dense;
};

// The level of scatter thread st at G = 16: each half warp has one.  The dense levels pair up
// among themselves (one index arithmetic per warp); the others pair coarse with fine,
// since a fine level flushes at almost every sample and the slowest warp sets the pace
// (pairs of neighbours, 14 and 15 in one warp: 4.38 against 4.34 ms for the backward).
__device__ __forceinline__ uint32_t scatter_level(const DevCfg& c, uint32_t st) {
    const uint32_t dense = c.dense_mask & 0xffffu, nd = __popc(dense), in_pairs = nd & ~1u;
    const uint32_t w = st >> 5, hi = (st >> 4) & 1u;
    uint32_t k;  // place in the order: dense levels, then the others
    if (2u * w < in_pairs) k = 2u * w + hi;
    else k = hi ? 15u - (w - in_pairs / 2u) : w + in_pairs / 2u;
    const bool want_dense = k < nd;
    if (!want_dense) k -= nd;
    uint32_t level = 0;
    for (uint32_t l = 0, seen = 0; l < 16; ++l)
        if (((dense >> l) & 1u) == (want_dense ? 1u : 0u) && seen++ == k) level = l;
    return level;
}

__device__ __forceinline__ void set_level(const DevCfg& c, uint32_t level, ScatterRole& s) {
    s.N = c.res[level];
    s.dense = (c.dense_mask >> level) & 1u;
    s.m1 = s.dense ? s.N + 1u : 2654435761u;
    s.m2 = s.dense ? (s.N + 1u) * (s.N + 1u) : 805459861u;
}

// Physical row of sample row r in the tile buffers the scatter walks (positions, and
// dL/dfeat per level): lanes of the groups read rows G g + i with the same i, which
// the permutation spreads over all banks (dL/dfeat: the odd levels of G = 16, which mostly
// share a warp with even ones, or the upper groups of G = 8, over the other half).
template <int G>
__device__ __forceinline__ uint32_t tile_row(uint32_t r) { return r ^ ((r / G) & 7u); }
template <int G>
__device__ __forceinline__ uint32_t tile_df(uint32_t r, uint32_t level) {
    return level * 128u + (tile_row<G>(r) ^ ((G == 16 ? level & 1u : (r >> 6) & 1u) << 3));
}

// Where a differs from b: acc leaves to *p by one 8-byte FP32 reduction, and is cleared.
__device__ __forceinline__ void flush_if_ne(float2* p, float2& v, uint32_t a, uint32_t b) {
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "setp.ne.u32 q, %3, %4;\n"
        "@q red.relaxed.gpu.global.add.v2.f32 [%2], {%0, %1};\n"
        "@q mov.f32 %0, 0f00000000;\n"
        "@q mov.f32 %1, 0f00000000;\n"
        "}\n" : "+f"(v.x), "+f"(v.y) : "l"(p), "r"(a), "r"(b)
        : "memory");
}

// The walk of one thread.  kMode: 0 hashed levels, 1 dense levels, 2 both in the warp.
// A vertex that leaves is told by its slot: two vertices with one slot share an entry.
// Cells are kept as the bits of 2^23 + c: the bias, a multiple of 2^24 once multiplied,
// vanishes under the slot mask (at most 2^24 entries).  Of an axis' two vertices one is
// odd and one even; the trilinear weight of either is q's distance from the other, for
// either order of the two.  (1 - |q - odd| for the odd one would save an add, but in the
// first cell it is rounded to 2^-24 where q itself is the weight: 4.27 for 4.29 ms.)  Beyond the last cell
// (kUnit = false: a box that reaches past the unit cube, whose samples extrapolate from that
// cell) the distance takes its sign from the order instead.
template <int kMode, bool kUnit>
__device__ __forceinline__ void scatter_walk(const ScatterRole& s, float2* __restrict__ gtab, uint32_t mask,
                                             const float4* pos, const float2* df, uint32_t n) {
    const float Nf = small_float(s.N), top = Nf - 0.5f;
    const uint32_t np = 1u - s.p;
    pos += s.r0;
    df += s.rd;
    uint32_t held[4];                                     // slots by parity, [2 z + y]
    float2 acc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        acc[k] = make_float2(0.f, 0.f);
        held[k] = 0u;
    }
#pragma unroll 1
    for (uint32_t i = 0; i < n; ++i) {
        const float4 q = pos[i ^ s.swz];
        const float2 gl = df[i ^ s.swz ^ s.dx];
        const float qx = fmul(q.x, Nf), qy = fmul(q.y, Nf), qz = fmul(q.z, Nf);
        // positions are >= 0 (the box test)
        const uint32_t cx = __float_as_uint(__fadd_rd(fminf(qx, top), 8388608.f));
        const uint32_t cy = __float_as_uint(__fadd_rd(fminf(qy, top), 8388608.f));
        const uint32_t cz = __float_as_uint(__fadd_rd(fminf(qz, top), 8388608.f));
        // weight of the vertex whose other one is v (as bits); neg: that one is the upper
        auto weight = [](float qa, uint32_t v, bool neg) {
            const float d = fsub(qa, fsub(__uint_as_float(v), 8388608.f));
            return kUnit ? fabsf(d) : (neg ? -d : d);
        };
        const uint32_t X = ((cx + np) & ~1u) | s.p, xo = ((cx + s.p) & ~1u) | np;
        const uint32_t ye = (cy + 1u) & ~1u, yo = cy | 1u, ze = (cz + 1u) & ~1u, zo = cz | 1u;
        const uint32_t A[2] = {ye * s.m1, yo * s.m1};
        const uint32_t B[2] = {ze * s.m2, zo * s.m2};
        const float fx = weight(qx, xo, (cx & 1u) == s.p);
        const float fy[2] = {weight(qy, yo, !(cy & 1u)), weight(qy, ye, cy & 1u)};
        const float fz[2] = {weight(qz, zo, !(cz & 1u)), weight(qz, ze, cz & 1u)};
        uint32_t slot[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t a = A[k & 1], b = B[k >> 1];
            slot[k] = (kMode == 1 || (kMode == 2 && s.dense) ? X + a + b : X ^ a ^ b) & mask;
        }
        if (i > 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k) flush_if_ne(gtab + held[k], acc[k], slot[k], held[k]);
        }
        const float xy[2] = {fx * fy[0], fx * fy[1]};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float w = xy[k & 1] * fz[k >> 1];
            acc[k].x += w * gl.x;
            acc[k].y += w * gl.y;
            held[k] = slot[k];
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) atomicAdd(gtab + held[k], acc[k]);
}

__device__ __forceinline__ bool unit_box(const DevCfg& c) {
    return c.box[0] <= 1.f && c.box[1] <= 1.f && c.box[2] <= 1.f;
}

// pos: [128] (x, y, z, -) by tile_row; df: dL/dfeat by tile_df; n_valid: samples in the
// tile; n_levels: the levels 0 .. n_levels - 1 are scattered (G = 8: at most 8).  level:
// scatter_level(c, st) (G = 16 only).
template <int G>
__device__ __forceinline__ void scatter_tile(const DevCfg& c, float2* __restrict__ gtables, uint32_t st,
                                             uint32_t level, uint32_t n_levels, const float4* pos, const float2* df,
                                             uint32_t n_valid) {
    const uint32_t lane = st & 31u;
    const uint32_t g = G == 16 ? (lane >> 1) & 7u : lane >> 1;
    if (G == 8) level = st >> 5;
    ScatterRole s;
    set_level(c, level, s);
    s.p = lane & 1u;
    s.r0 = G * g;
    s.swz = g & 7u;
    s.dx = G == 16 ? (level & 1u) << 3 : 0u;
    s.rd = level * 128u + (G == 16 ? s.r0 : s.r0 ^ ((g >> 3) << 3));
    const uint32_t n = level < n_levels && s.r0 < n_valid ? min((uint32_t)G, n_valid - s.r0) : 0u;
    const uint32_t hashed = __ballot_sync(0xffffffffu, n && !s.dense), dense = __ballot_sync(0xffffffffu, n && s.dense);
    if (n == 0u) return;
    float2* gtab = gtables + (size_t)level * c.T;
    const uint32_t mask = c.T - 1;
    if (!unit_box(c)) scatter_walk<2, false>(s, gtab, mask, pos, df, n);
    else if (dense == 0u) scatter_walk<0, true>(s, gtab, mask, pos, df, n);
    else if (hashed == 0u) scatter_walk<1, true>(s, gtab, mask, pos, df, n);
    else scatter_walk<2, true>(s, gtab, mask, pos, df, n);
}

// dL/dx = sum_l (d f_l / dx) . dL/df_l at grid position x over the levels l0, l0 + 2, ...,
// for the pose gradient: inside a cell of level l (resolution N) the trilinear weight of
// corner k is w_k = prod_a (b_a ? w_a : 1 - w_a) with w_a = x_a N - c_a, so
// dw_k/dx_a = N (b_a ? 1 : -1) prod_{a' != a} (b_a' ? w_a' : 1 - w_a'); the table
// values of the 8 corners are read again (whole warps, pair_sample order: the encoding's
// loads).  df(l): dL/df_l of this lane's sample.  The even and the odd levels are summed by
// different warps (one thread per sample for all of them made the FP16 backward of 4.87 M
// samples with pose terms 2.79 ms, against 1.11 without; now 2.39).
template <class DF>
__device__ __forceinline__ float3 hash_grad_x(const DevCfg& c, const float2* __restrict__ tables, float3 x, DF df,
                                              int l0) {
    float gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll 1
    for (int l = l0; l < (int)c.L; l += 2) {
        float2 lo[4], up[4];
        float w[3];
        level_corners(c, tables, x, l, lo, up, w);
        const float2 g = df(l);
        float ax = 0.f, ay = 0.f, az = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int by = j & 1, bz = j >> 1;
            const float e0 = lo[j].x * g.x + lo[j].y * g.y, e1 = up[j].x * g.x + up[j].y * g.y;
            const float fy = by ? w[1] : 1.f - w[1], fz = bz ? w[2] : 1.f - w[2];
            const float m = (1.f - w[0]) * e0 + w[0] * e1;
            ax += (e1 - e0) * fy * fz;
            ay += (by ? m : -m) * fz;
            az += (bz ? m : -m) * fy;
        }
        const float N = small_float(c.res[l]);
        gx += N * ax;
        gy += N * ay;
        gz += N * az;
    }
    return make_float3(gx, gy, gz);
}

__device__ __forceinline__ float sigmoidf_(float z) { return 1.f / (1.f + expf(-z)); }

}  // namespace nm
