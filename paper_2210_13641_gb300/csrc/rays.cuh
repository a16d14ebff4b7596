// rays.cuh - pinhole ray casting and the ray batch's structure-of-arrays store,
// shared by the mapping step's ray draw, the render's view rays and the grouped
// render of several views (step a1).
#pragma once

#include "internal.h"

namespace nm {

// Back-projection of the pixel centre, rotation to world, normalisation; exact
// FP32 operation order (the same integer decisions follow from these values).
__device__ __forceinline__ void cast_ray(const float* c2w, const float* K, uint32_t u,
                                         uint32_t v, float3& o, float3& d) {
    const float dx = fdiv(fsub(fadd((float)u, 0.5f), K[2]), K[0]);
    const float dy = fdiv(fsub(fadd((float)v, 0.5f), K[3]), K[1]);
    const float wx = fadd(fadd(fmul(c2w[0], dx), fmul(c2w[1], dy)), c2w[2]);
    const float wy = fadd(fadd(fmul(c2w[4], dx), fmul(c2w[5], dy)), c2w[6]);
    const float wz = fadd(fadd(fmul(c2w[8], dx), fmul(c2w[9], dy)), c2w[10]);
    const float n = __fsqrt_rn(fadd(fadd(fmul(wx, wx), fmul(wy, wy)), fmul(wz, wz)));
    d = make_float3(fdiv(wx, n), fdiv(wy, n), fdiv(wz, n));
    o = make_float3(c2w[3], c2w[7], c2w[11]);
}

__device__ __forceinline__ void store_ray(float* rays, uint32_t cap, uint32_t r, float3 o,
                                          float3 d, float4 t0, float V, uint32_t kf) {
    rays[kOx * cap + r] = o.x;
    rays[kOy * cap + r] = o.y;
    rays[kOz * cap + r] = o.z;
    rays[kDx * cap + r] = d.x;
    rays[kDy * cap + r] = d.y;
    rays[kDz * cap + r] = d.z;
    rays[kIr * cap + r] = t0.x;
    rays[kIg * cap + r] = t0.y;
    rays[kIb * cap + r] = t0.z;
    rays[kD * cap + r] = t0.w;
    rays[kV * cap + r] = V;
    rays[kKf * cap + r] = __uint_as_float(kf);
}

// Totals of the rays' sample counts per tile of kScanTile rays, from which k_compact and
// k_select find where a ray's samples go: all samples, the first kRenderFirst of each ray,
// the samples a render's second pass still evaluates.  The ray generation clears them
// (first, live: nullptr in a step), k_march and the compositing add to them.
struct TileTotals {
    uint32_t *all, *first, *live;
};
inline TileTotals tile_totals(const StepBufs& b, bool render) {
    // a render does not use the partials of the training compositing
    uint32_t* p = reinterpret_cast<uint32_t*>(b.partials);
    return TileTotals{b.block_sums, render ? p : nullptr, render ? p + kCompositeMaxBlocks : nullptr};
}
static_assert(ray_tiles(1u << 24) <= kCompositeMaxBlocks, "the totals of the largest batch fit the partials");

// Whether thread i of a batch's ray generation clears the totals of tile i.  The tiles are
// counted, not i * kScanTile compared with n_rays: that product wraps from thread 2^20 on.
__host__ __device__ __forceinline__ bool clears_tile(uint32_t i, uint32_t n_rays) { return i < ray_tiles(n_rays); }

__device__ __forceinline__ void clear_totals(const TileTotals& t, uint32_t i, uint32_t n_rays) {
    if (!clears_tile(i, n_rays)) return;
    t.all[i] = 0u;
    if (t.first) t.first[i] = 0u;
    if (t.live) t.live[i] = 0u;
}

// The march of one ray by one warp: retained steps to row (max_samples at most), their
// number returned to all lanes.
__device__ __forceinline__ uint32_t march_ray(const DevCfg& c, const uint32_t* __restrict__ bits,
                                              const float* __restrict__ rays, uint32_t cap, uint32_t r, float* row) {
    const uint32_t lane = threadIdx.x & 31u;
    const float3 o = make_float3(rays[kOx * cap + r], rays[kOy * cap + r], rays[kOz * cap + r]);
    const float3 d = make_float3(rays[kDx * cap + r], rays[kDy * cap + r], rays[kDz * cap + r]);
    const uint32_t max_samples = c.max_samples;
    uint32_t i_lo, i_hi;
    box_step_range(c, o, d, i_lo, i_hi);
    uint32_t n = 0;
    for (uint32_t i0 = i_lo; i0 < i_hi && n < max_samples; i0 += 32) {
        const uint32_t i = i0 + lane;
        bool keep = false;
        float t = 0.f;
        if (i < i_hi) {
            t = sample_t(c, i);
            const float3 x = grid_pos(c, o, d, t);
            keep = in_box(c, x) && occupied(c, bits, x);
        }
        const uint32_t m = __ballot_sync(0xffffffffu, keep);
        const uint32_t pos = n + __popc(m & ((1u << lane) - 1u));
        if (keep && pos < max_samples) row[pos] = t;
        n += __popc(m);
    }
    return n < max_samples ? n : max_samples;
}

// Count n of the warp's ray r to counts, and the block's 8 rays (of one tile) to the totals.
__device__ __forceinline__ void ray_totals(const TileTotals& t, uint32_t r, uint32_t n, uint32_t n_rays,
                                           uint32_t* __restrict__ counts) {
    __shared__ uint32_t cnt[8];
    const uint32_t w = threadIdx.x >> 5;
    if ((threadIdx.x & 31u) == 0u) {
        cnt[w] = n;
        if (r < n_rays) counts[r] = n;
    }
    __syncthreads();
    if (threadIdx.x != 0u) return;
    uint32_t all = 0, first = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        all += cnt[k];
        first += min(cnt[k], kRenderFirst);
    }
    if (all == 0u) return;
    atomicAdd(t.all + r / kScanTile, all);
    if (t.first) atomicAdd(t.first + r / kScanTile, first);
}

}  // namespace nm
