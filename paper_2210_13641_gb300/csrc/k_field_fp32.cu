// k_field_fp32.cu - the field on FP32 CUDA cores (the plain form): hash encoding,
// density MLP (sigma = exp(h_0)), SH view encoding and colour MLP (sigmoid) forward
// (steps a3-a6), and the recomputing backward pass (steps a10-a11).
//
// Both work on tiles of 128 samples whose activations sit in shared memory.
#include "encoding.cuh"
#include "internal.h"

namespace nm {

// 16-byte loads, several in flight (each launch pays this once per block).
__device__ __forceinline__ void load_weights(float* W, const float* __restrict__ mlp) {
#pragma unroll 5
    for (int i = threadIdx.x; i < kMlpParams / 4; i += blockDim.x)
        reinterpret_cast<float4*>(W)[i] = __ldg(reinterpret_cast<const float4*>(mlp) + i);
}

__device__ __forceinline__ float3 sample_pos(const DevCfg& c, const float* __restrict__ rays,
                                             uint32_t cap, uint32_t r, float t, float3& d) {
    const float3 o = make_float3(rays[kOx * cap + r], rays[kOy * cap + r], rays[kOz * cap + r]);
    d = make_float3(rays[kDx * cap + r], rays[kDy * cap + r], rays[kDz * cap + r]);
    return grid_pos(c, o, d, t);
}

constexpr int kTile = 128;          // samples of a tile
constexpr int kFieldThreads = 256;  // threads of a block, forward and backward

// o[n][q] += sum_k W[n][k] x_q[k] for NO outputs and 4 samples (rows of ROW floats: x, 32 rows
// on, ...) over K inputs, k ascending.
template <int K, int NO, int ROW>
__device__ __forceinline__ void dot_rows(const float* __restrict__ W, const float* x, float (*o)[4]) {
#pragma unroll 1
    for (int k = 0; k < K; k += 4) {
        float4 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = *reinterpret_cast<const float4*>(x + 32 * q * ROW + k);
#pragma unroll
        for (int n = 0; n < NO; ++n) {
            const float4 w = *reinterpret_cast<const float4*>(W + n * K + k);
#pragma unroll
            for (int q = 0; q < 4; ++q) o[n][q] = fmaf(w.x, v[q].x, o[n][q]);
#pragma unroll
            for (int q = 0; q < 4; ++q) o[n][q] = fmaf(w.y, v[q].y, o[n][q]);
#pragma unroll
            for (int q = 0; q < 4; ++q) o[n][q] = fmaf(w.z, v[q].z, o[n][q]);
#pragma unroll
            for (int q = 0; q < 4; ++q) o[n][q] = fmaf(w.w, v[q].w, o[n][q]);
        }
    }
}

template <int N>
__device__ __forceinline__ void zero(float* v) {
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = 0.f;
}

// Output n of sample q, N of them (a multiple of 4, or 2), to the samples' rows.
template <int N, bool RELU, int ROW>
__device__ __forceinline__ void put(float* dst, const float (*o)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float v[N];
#pragma unroll
        for (int n = 0; n < N; ++n) v[n] = RELU ? fmaxf(o[n][q], 0.f) : o[n][q];
        float* d = dst + 32 * q * ROW;
        if constexpr (N % 4 == 0) {
#pragma unroll
            for (int n = 0; n < N; n += 4)
                *reinterpret_cast<float4*>(d + n) = make_float4(v[n], v[n + 1], v[n + 2], v[n + 3]);
        } else {
            *reinterpret_cast<float2*>(d) = make_float2(v[0], v[1]);
        }
    }
}

// ------------------------------------------------------------------ forward
// Tiles of 128 samples, two 256-thread blocks per SM: two threads encode each sample (half
// the levels each), then every layer is a phase over 4 samples x 8 outputs per thread
// (dot_rows) on activations in shared memory.  Bound by the multiply-adds (9.4 k per
// sample: 1.2 ms for 4.87 M samples) and the loads that feed them, and the gathers.  One
// thread per sample, all weights read again for each, took 3.31 ms there; this form
// 2.91.
constexpr int kFRow = 132;  // row: f[0,32) x3[32,64) h1, then h3 [64,128); h4 over f and x3
constexpr int kFx3 = 32, kFh = 64;

struct alignas(16) SmemFwd {
    float W[kMlpParams];        // plain (out, in) layout as in the parameter buffer
    float act[kTile * kFRow];
};

// kSel: the samples sel[0 .. *n_total) of the batch instead of 0 .. *n_total (a
// render's passes); the encodings are not stored then.
template <bool kSel>
__global__ void __launch_bounds__(kFieldThreads, 2) k_field_fwd_fp32(DevCfg c, const float* __restrict__ params,
                                                        const float* __restrict__ rays, uint32_t cap,
                                                        const uint32_t* __restrict__ n_total,
                                                        const uint32_t* __restrict__ ray_id,
                                                        const float* __restrict__ ts,
                                                        float4* __restrict__ sig_rgb,
                                                        float* __restrict__ feat_out,
                                                        const uint32_t* __restrict__ sel) {
    extern __shared__ __align__(16) float smem_raw[];
    SmemFwd& s = *reinterpret_cast<SmemFwd*>(smem_raw);
    const uint32_t n = *n_total;
    if (blockIdx.x * (uint32_t)kTile >= n) return;
    load_weights(s.W, params + (size_t)c.L * c.T * 2);
    const float* W5 = s.W + kOffW5;
    const float2* tables = reinterpret_cast<const float2*>(params);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float* const row0 = s.act + lane * kFRow;                   // layer products: samples lane, lane + 32, ...
    const int part = tid >> 7;                                   // encoding: levels 8 part .. 8 part + 7
    const uint32_t er = (tid & 96) + pair_sample(tid & 31);      // of this sample (whole warps)
    float* const erow = s.act + er * kFRow;
    float* const trow = s.act + (tid & 127) * kFRow;
    for (uint32_t i0 = blockIdx.x * (uint32_t)kTile; i0 < n; i0 += gridDim.x * (uint32_t)kTile) {
        {
            const uint32_t j = i0 + er;
            const bool valid = j < n;
            const uint32_t i = valid ? (kSel ? sel[j] : j) : 0u;
            float3 d = make_float3(0.f, 0.f, 0.f), x = d;
            if (valid) x = sample_pos(c, rays, cap, ray_id[i], ts[i], d);
            if (part) {
                float sh[16];
                sh16(d.x, d.y, d.z, sh);
#pragma unroll
                for (int k = 0; k < 16; k += 4)
                    *reinterpret_cast<float4*>(erow + kFx3 + kGeo + k) = make_float4(sh[k], sh[k + 1], sh[k + 2], sh[k + 3]);
            }
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int l = 8 * part + 2 * h;
                float f[4] = {0.f, 0.f, 0.f, 0.f};
                if (l < (int)c.L) encode_level(c, tables, x, l, f);
                if (l + 1 < (int)c.L) encode_level(c, tables, x, l + 1, f + 2);
                const float4 q = make_float4(f[0], f[1], f[2], f[3]);
                *reinterpret_cast<float4*>(erow + 2 * l) = q;
                if (!kSel && feat_out && valid) *reinterpret_cast<float4*>(feat_out + (size_t)i * kEnc + 2 * l) = q;
            }
        }
        __syncthreads();
        float o[8][4];
        zero<32>(&o[0][0]);
        dot_rows<kEnc, 8, kFRow>(s.W + kOffW1 + 8 * warp * kEnc, row0, o);
        put<8, true, kFRow>(row0 + kFh + 8 * warp, o);
        __syncthreads();
        zero<8>(&o[0][0]);
        dot_rows<kHid, 2, kFRow>(s.W + kOffW2 + 2 * warp * kHid, row0 + kFh, o);
        put<2, false, kFRow>(row0 + kFx3 + 2 * warp, o);
        __syncthreads();
        const float sigma = expf(fminf(trow[kFx3], kSigmaHMax));
        zero<32>(&o[0][0]);
        dot_rows<32, 8, kFRow>(s.W + kOffW3 + 8 * warp * 32, row0 + kFx3, o);
        put<8, true, kFRow>(row0 + kFh + 8 * warp, o);
        __syncthreads();
        zero<32>(&o[0][0]);
        dot_rows<kHid, 8, kFRow>(s.W + kOffW4 + 8 * warp * kHid, row0 + kFh, o);
        put<8, true, kFRow>(row0 + 8 * warp, o);
        __syncthreads();
        if (tid < kTile && i0 + tid < n) {
            float z[3] = {0.f, 0.f, 0.f};
#pragma unroll 4
            for (int q = 0; q < kHid; q += 4) {
                const float4 h = *reinterpret_cast<const float4*>(trow + q);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float4 w = *reinterpret_cast<const float4*>(W5 + k * kHid + q);
                    z[k] = fmaf(w.x, h.x, z[k]);
                    z[k] = fmaf(w.y, h.y, z[k]);
                    z[k] = fmaf(w.z, h.z, z[k]);
                    z[k] = fmaf(w.w, h.w, z[k]);
                }
            }
            sig_rgb[kSel ? sel[i0 + tid] : i0 + tid] = make_float4(sigma, sigmoidf_(z[0]), sigmoidf_(z[1]), sigmoidf_(z[2]));
        }
        __syncthreads();  // the next tile overwrites the rows
    }
}

template <bool kSel>
static void fwd_fp32(const DevCfg& c, const float* params, const uint32_t* n, const uint32_t* sel, const StepBufs& b,
                     float* feat, int n_sm, cudaStream_t st) {
    const int smem = (int)sizeof(SmemFwd);
    // per call: the attribute belongs to the current device (cheap next to the kernel)
    cudaFuncSetAttribute(k_field_fwd_fp32<kSel>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    k_field_fwd_fp32<kSel><<<n_sm * 2, kFieldThreads, smem, st>>>(c, params, b.rays, b.cap_rays, n, b.ray_id, b.t,
                                                                  b.sig_rgb, feat, sel);
}

void launch_field_fwd_fp32(const DevCfg& c, const float* params, uint32_t n_rays, const StepBufs& b,
                           bool store_feat, int n_sm, cudaStream_t st) {
    fwd_fp32<false>(c, params, b.offsets + n_rays, nullptr, b, store_feat ? b.feat : nullptr, n_sm, st);
}

void launch_field_fwd_fp32_sel(const DevCfg& c, const float* params, const uint32_t* sel, const uint32_t* n_sel,
                               const StepBufs& b, int n_sm, cudaStream_t st) {
    fwd_fp32<true>(c, params, n_sel, sel, b, nullptr, n_sm, st);
}

// ------------------------------------------------------------------ backward
// A 256-thread block per SM walks tiles of 128 samples.  A tile's activations sit in
// shared memory, one row of 260 floats per sample, and every layer is a phase between
// block barriers:
//  - layer products (forward recompute and data gradients): a thread takes 4 samples and
//    an eighth of the outputs (4 x 8 sums in registers), 4 inputs at a time: 4 16-byte
//    loads of activations and 8 of weights, which all lanes share, for 128 multiply-adds.
//    The recompute sums in the forward kernel's order, so its ReLU branches are the
//    forward's, bit for bit;
//  - weight gradients: a thread owns 8 rows and 4 columns of each weight matrix for a part
//    of the samples (3 16-byte loads for 32 multiply-adds).  A matrix has 2, 4 or 8 such
//    parts, of 64, 32 or 16 samples of a tile; in turn, one part per tile adds its registers
//    to the block's sums in shared memory and clears them.  So no FP32 sum runs over more
//    than 128 products, nor over more than the block's tiles after that, and no two parts
//    meet at an entry.  Registers kept over all tiles took 7.92 instead of 8.05 ms, but a
//    flat sum over the 13.8 k equal products of a thread's 215 tiles is off by 1e-4 of
//    itself (this one: 2e-6);
//  - the encoding gradient goes through shared memory to the tile scatter.
// The multiply-adds (28 k per sample: 3.6 ms for 4.87 M samples at the FP32 cores' rate)
// and the shared-memory loads that feed them bound it.  One thread per sample with 128
// threads per SM, whose weight-gradient products took 8 4-byte loads for 16 multiply-adds,
// needed 14.2 ms there; this form 8.05 ms (with 2 samples x 16 outputs per thread it took 0.7 more).
constexpr int kRow = 260;  // 16-byte rows; consecutive rows start 16 bytes apart modulo the banks
// Row layout: f[0,32) h1[32,96) x3[96,128) h3[128,192) h4[192,256), then the colour
// seeds (dL/dc, later dL/dz) and dL/dsigma (later dL/dsigma * dsigma/dh_0)
constexpr int kRf = 0, kRh1 = 32, kRx3 = 96, kRh3 = 128, kRh4 = 192, kRdz = 256, kRds = 259;

struct SmemBwd {
    float W[kMlpParams];          // plain (out, in) layout as in the parameter buffer
    float dW[kMlpParams];         // the block's weight gradients
    float act[kTile * kRow];
    float2 df[kTile * 16];        // dL/dfeat by tile_df
    float4 pos[2][kTile];         // sample positions by tile_row, by tile parity
};
static_assert(kMlpParams % 4 == 0, "rows of 16 bytes behind the weights");

// o[k][q] += sum_n W[n][k] g_q[n] for NO consecutive k over N rows of length LD.
template <int N, int LD, int NO>
__device__ __forceinline__ void dot_cols(const float* __restrict__ W, const float* g, float (*o)[4]) {
#pragma unroll 1
    for (int n = 0; n < N; n += 4) {
        float v[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 t = *reinterpret_cast<const float4*>(g + 32 * q * kRow + n);
            v[0][q] = t.x;
            v[1][q] = t.y;
            v[2][q] = t.z;
            v[3][q] = t.w;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float w[NO];
            if constexpr (NO % 4 == 0) {
#pragma unroll
                for (int k = 0; k < NO; k += 4) {
                    const float4 t = *reinterpret_cast<const float4*>(W + (n + i) * LD + k);
                    w[k] = t.x;
                    w[k + 1] = t.y;
                    w[k + 2] = t.z;
                    w[k + 3] = t.w;
                }
            } else {
                const float2 t = *reinterpret_cast<const float2*>(W + (n + i) * LD);
                w[0] = t.x;
                w[1] = t.y;
            }
#pragma unroll
            for (int k = 0; k < NO; ++k)
#pragma unroll
                for (int q = 0; q < 4; ++q) o[k][q] = fmaf(w[k], v[i][q], o[k][q]);
        }
    }
}

// acc[4 n + j] += sum_s g[s][n] x[s][j] over samples s0 .. s0 + ns - 1, 8 rows n and 4
// columns j (g, x: the thread's first row and column in the activation rows).
__device__ __forceinline__ void outer_sum(const float* g, const float* x, int s0, int ns, float* acc) {
    g += s0 * kRow;
    x += s0 * kRow;
#pragma unroll 2
    for (int s = 0; s < ns; ++s, g += kRow, x += kRow) {
        const float4 xv = *reinterpret_cast<const float4*>(x);
#pragma unroll
        for (int n = 0; n < 8; n += 4) {
            const float4 gv = *reinterpret_cast<const float4*>(g + n);
            const float gn[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                acc[4 * (n + m)] = fmaf(gn[m], xv.x, acc[4 * (n + m)]);
                acc[4 * (n + m) + 1] = fmaf(gn[m], xv.y, acc[4 * (n + m) + 1]);
                acc[4 * (n + m) + 2] = fmaf(gn[m], xv.z, acc[4 * (n + m) + 2]);
                acc[4 * (n + m) + 3] = fmaf(gn[m], xv.w, acc[4 * (n + m) + 3]);
            }
        }
    }
}

// 8 gradients of 4 samples over their activations (masked by the ReLU branches those tell).
__device__ __forceinline__ void put_masked(float* act, const float (*o)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int n = 0; n < 8; n += 4) {
            float4* a = reinterpret_cast<float4*>(act + 32 * q * kRow + n);
            const float4 h = *a;
            *a = make_float4(h.x > 0.f ? o[n][q] : 0.f, h.y > 0.f ? o[n + 1][q] : 0.f,
                             h.z > 0.f ? o[n + 2][q] : 0.f, h.w > 0.f ? o[n + 3][q] : 0.f);
        }
}

// kPose: also writes, per sample, dL/dp (world position) through the even levels into
// pose_s[2 i] and through the odd ones into pose_odd[8 i] (over the sample's row of feat,
// which its tile has read), and the view-direction gradient through the SH encoding into
// pose_s[2 i + 1].
template <bool kPose>
__global__ void __launch_bounds__(kFieldThreads) k_field_bwd_fp32(DevCfg c, const float* __restrict__ params,
                                                          float* __restrict__ grads,
                                                          const float* __restrict__ rays, uint32_t cap,
                                                          const uint32_t* __restrict__ n_total,
                                                          const uint32_t* __restrict__ ray_id,
                                                          const float* __restrict__ ts,
                                                          const float* feat,
                                                          const float4* __restrict__ dsig_rgb,
                                                          float4* __restrict__ pose_s, float4* pose_odd) {
    extern __shared__ __align__(16) float smem_raw[];
    SmemBwd& s = *reinterpret_cast<SmemBwd*>(smem_raw);
    const uint32_t n = *n_total;
    if (blockIdx.x * (uint32_t)kTile >= n) return;
    const float* mlp = params + (size_t)c.L * c.T * 2;
    load_weights(s.W, mlp);
    const float* W1 = s.W + kOffW1;
    const float* W2 = s.W + kOffW2;
    const float* W3 = s.W + kOffW3;
    const float* W4 = s.W + kOffW4;
    const float* W5 = s.W + kOffW5;
    float2* gtables = reinterpret_cast<float2*>(grads);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // layer products: samples lane, lane + 32, ..., the warp's eighth of the outputs
    float* const row0 = s.act + lane * kRow;
    // weight gradients: 4 columns and 8 rows per thread.  64 columns are 16 lanes (a half
    // warp each other samples or rows), 32 columns 8 lanes.
    const int c16 = 4 * (lane & 15), c8 = 4 * (lane & 7), half = lane >> 4, quart = lane >> 3, e0 = warp * 16;
    const uint32_t level = scatter_level(c, tid);
    for (int i = tid; i < kMlpParams; i += kFieldThreads) s.dW[i] = 0.f;  // added to many barriers later
    float g1[32], g2[32], g3[32], g4[32], g5[6];
    zero<32>(g1);
    zero<32>(g2);
    zero<32>(g3);
    zero<32>(g4);
    zero<6>(g5);
    auto add = [&](int off, int ld, float* g) {
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            float4* p = reinterpret_cast<float4*>(s.dW + off + n * ld);
            const float4 v = *p;
            *p = make_float4(v.x + g[4 * n], v.y + g[4 * n + 1], v.z + g[4 * n + 2], v.w + g[4 * n + 3]);
        }
        zero<32>(g);
    };
    // the sums of part p4 (of W4), p3 (W3, W1) and p2 (W2, W5) into dW
    auto add_part = [&](int p4, int p3, int p2) {
        if (half == p4) add(kOffW4 + 8 * warp * kHid + c16, kHid, g4);
        if (quart == p3) {
            add(kOffW3 + 8 * warp * 32 + c8, 32, g3);
            add(kOffW1 + 8 * warp * kEnc + c8, kEnc, g1);
        }
        if (warp == p2) {
            add(kOffW2 + 8 * half * kHid + c16, kHid, g2);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                float2* p = reinterpret_cast<float2*>(s.dW + kOffW5 + k * kHid + 2 * lane);
                const float2 v = *p;
                *p = make_float2(v.x + g5[2 * k], v.y + g5[2 * k + 1]);
            }
            zero<6>(g5);
        }
    };
    const uint32_t n_tiles = (n + kTile - 1) / kTile;
    int turn = 0;  // the block's tiles, counted
    for (uint32_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++turn) {
        const uint32_t i0 = tile * kTile, parity = turn & 1;
        {   // inputs: two threads per sample
            const int r = tid & 127, part = tid >> 7;
            const uint32_t i = i0 + r;
            const bool valid = i < n;
            float* row = s.act + r * kRow;
            float4 v[4];
            const float4* fi = reinterpret_cast<const float4*>(feat + (size_t)i * kEnc) + 4 * part;
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = valid ? fi[k] : make_float4(0.f, 0.f, 0.f, 0.f);
            if (part == 0) {
                float3 x = make_float3(0.f, 0.f, 0.f), d = x;
                float sh[16];
                zero<16>(sh);
                if (valid) {
                    x = sample_pos(c, rays, cap, ray_id[i], ts[i], d);
                    sh16(d.x, d.y, d.z, sh);
                }
                s.pos[parity][tile_row<16>(r)] = make_float4(x.x, x.y, x.z, 0.f);
                #pragma unroll
                for (int k = 0; k < 16; k += 4)
                    *reinterpret_cast<float4*>(row + kRx3 + kGeo + k) = make_float4(sh[k], sh[k + 1], sh[k + 2], sh[k + 3]);
            } else {
                const float4 g = valid ? dsig_rgb[i] : make_float4(0.f, 0.f, 0.f, 0.f);
                *reinterpret_cast<float4*>(row + kRdz) = make_float4(g.y, g.z, g.w, g.x);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) *reinterpret_cast<float4*>(row + kRf + 16 * part + 4 * k) = v[k];
        }
        __syncthreads();
        float o[8][4];
        // ---- forward recompute
        zero<32>(&o[0][0]);
        dot_rows<kEnc, 8, kRow>(W1 + 8 * warp * kEnc, row0 + kRf, o);
        put<8, true, kRow>(row0 + kRh1 + 8 * warp, o);
        __syncthreads();
        zero<8>(&o[0][0]);
        dot_rows<kHid, 2, kRow>(W2 + 2 * warp * kHid, row0 + kRh1, o);
        put<2, false, kRow>(row0 + kRx3 + 2 * warp, o);
        __syncthreads();
        zero<32>(&o[0][0]);
        dot_rows<32, 8, kRow>(W3 + 8 * warp * 32, row0 + kRx3, o);
        put<8, true, kRow>(row0 + kRh3 + 8 * warp, o);
        __syncthreads();
        zero<32>(&o[0][0]);
        dot_rows<kHid, 8, kRow>(W4 + 8 * warp * kHid, row0 + kRh3, o);
        put<8, true, kRow>(row0 + kRh4 + 8 * warp, o);
        __syncthreads();
        if (tid < kTile) {  // colours: dL/dz; the density's seed
            float* row = s.act + tid * kRow;
            float z[3] = {0.f, 0.f, 0.f};
#pragma unroll 4
            for (int q = 0; q < kHid; ++q) {
                const float h = row[kRh4 + q];
#pragma unroll
                for (int k = 0; k < 3; ++k) z[k] = fmaf(W5[k * kHid + q], h, z[k]);
            }
            float4 g = *reinterpret_cast<const float4*>(row + kRdz);
            const float c0 = sigmoidf_(z[0]), c1 = sigmoidf_(z[1]), c2 = sigmoidf_(z[2]);
            const float y0 = row[kRx3];
            g.x = g.x * c0 * (1.f - c0);
            g.y = g.y * c1 * (1.f - c1);
            g.z = g.z * c2 * (1.f - c2);
            g.w = y0 < kSigmaHMax ? g.w * expf(fminf(y0, kSigmaHMax)) : 0.f;
            *reinterpret_cast<float4*>(row + kRdz) = g;
        }
        __syncthreads();
        // ---- backward.  dW5 += dz^T h4
#pragma unroll 4
        for (int q = e0; q < e0 + 16; ++q) {
            const float4 g = *reinterpret_cast<const float4*>(s.act + q * kRow + kRdz);
            const float2 h = *reinterpret_cast<const float2*>(s.act + q * kRow + kRh4 + 2 * lane);
            g5[0] = fmaf(g.x, h.x, g5[0]);
            g5[1] = fmaf(g.x, h.y, g5[1]);
            g5[2] = fmaf(g.y, h.x, g5[2]);
            g5[3] = fmaf(g.y, h.y, g5[3]);
            g5[4] = fmaf(g.z, h.x, g5[4]);
            g5[5] = fmaf(g.z, h.y, g5[5]);
        }
        // dA4 = (W5^T dz) [h4 > 0]
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 p = *reinterpret_cast<const float4*>(row0 + 32 * q * kRow + kRdz);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                o[k][q] = W5[8 * warp + k] * p.x + W5[kHid + 8 * warp + k] * p.y + W5[2 * kHid + 8 * warp + k] * p.z;
        }
        __syncthreads();
        put_masked(row0 + kRh4 + 8 * warp, o);
        __syncthreads();
        // dW4 += dA4^T h3;  dA3 = (W4^T dA4) [h3 > 0]
        outer_sum(s.act + kRh4 + 8 * warp, s.act + kRh3 + c16, 64 * half, 64, g4);
        zero<32>(&o[0][0]);
        dot_cols<kHid, kHid, 8>(W4 + 8 * warp, row0 + kRh4, o);
        __syncthreads();
        put_masked(row0 + kRh3 + 8 * warp, o);
        __syncthreads();
        // dW3 += dA3^T x3;  dy = (W3^T dA3)[0:16], dy_0 += the density's seed
        outer_sum(s.act + kRh3 + 8 * warp, s.act + kRx3 + c8, 32 * quart, 32, g3);
        if (kPose && tid < kTile && i0 + tid < n) {
            // the SH inputs' gradient (W3^T dA3)[16:32] -> the view-direction gradient
            const float* row = s.act + tid * kRow;
            float dsh[kSH];
            zero<kSH>(dsh);
#pragma unroll 4
            for (int nn = 0; nn < kHid; ++nn) {
                const float gg = row[kRh3 + nn];
#pragma unroll
                for (int m = 0; m < kSH; ++m) dsh[m] += W3[nn * 32 + kGeo + m] * gg;
            }
            const uint32_t r = ray_id[i0 + tid];
            const float3 gd = sh16_vjp(rays[kDx * cap + r], rays[kDy * cap + r], rays[kDz * cap + r], dsh);
            pose_s[2 * (size_t)(i0 + tid) + 1] = make_float4(gd.x, gd.y, gd.z, 0.f);
        }
        zero<8>(&o[0][0]);
        dot_cols<kHid, 32, 2>(W3 + 2 * warp, row0 + kRh3, o);
        if (warp == 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) o[0][q] += row0[32 * q * kRow + kRds];
        }
        __syncthreads();
        put<2, false, kRow>(row0 + kRx3 + 2 * warp, o);
        __syncthreads();
        // dW2 += dy^T h1;  dA1 = (W2^T dy) [h1 > 0]
        outer_sum(s.act + kRx3 + 8 * half, s.act + kRh1 + c16, e0, 16, g2);
        zero<32>(&o[0][0]);
        dot_cols<kGeo, kHid, 8>(W2 + 8 * warp, row0 + kRx3, o);
        __syncthreads();
        put_masked(row0 + kRh1 + 8 * warp, o);
        __syncthreads();
        // dW1 += dA1^T f;  df = W1^T dA1, scattered into the tables
        outer_sum(s.act + kRh1 + 8 * warp, s.act + kRf + c8, 32 * quart, 32, g1);
        zero<16>(&o[0][0]);
        dot_cols<kHid, kEnc, 4>(W1 + 4 * warp, row0 + kRh1, o);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            s.df[tile_df<16>(lane + 32 * q, 2 * warp)] = make_float2(o[0][q], o[1][q]);
            s.df[tile_df<16>(lane + 32 * q, 2 * warp + 1)] = make_float2(o[2][q], o[3][q]);
        }
        __syncthreads();
        add_part(turn & 1, turn & 3, turn & 7);  // the next part's turn is behind the next tile's barriers
        scatter_tile<16>(c, gtables, tid, level, c.L, s.pos[parity], s.df, n - i0);
        if (kPose) {  // dL/dp: warps 0-3 the even levels, 4-7 the odd ones
            const int odd = tid >> 7;
            const uint32_t row = (tid & 96) + pair_sample(lane);
            const float4 x = s.pos[parity][tile_row<16>(row)];
            const float3 g = hash_grad_x(c, reinterpret_cast<const float2*>(params), make_float3(x.x, x.y, x.z),
                                         [&](int l) { return s.df[tile_df<16>(row, l)]; }, odd);
            if (i0 + row < n)
                (odd ? pose_odd + 8 * (size_t)(i0 + row) : pose_s + 2 * (size_t)(i0 + row))[0] =
                    make_float4(g.x * c.inv_size, g.y * c.inv_size, g.z * c.inv_size, 0.f);
        }
        // the next tile's inputs go to rows that nobody reads any more, and to the other
        // position buffer; dL/dfeat is written again many barriers later
    }
    // ---- what each part has left, one after the other
    for (int part = 0; part < 8; ++part) {
        __syncthreads();
        add_part(part, part, part);
    }
    __syncthreads();
    float* gmlp = grads + (size_t)c.L * c.T * 2;
    for (int e = tid; e < kMlpParams; e += kFieldThreads) {
        const float v = s.dW[e];
        if (v != 0.f) atomicAdd(gmlp + e, v);
    }
}

void launch_field_bwd_fp32(const DevCfg& c, const float* params, float* grads, uint32_t n_rays,
                           const StepBufs& b, int n_sm, cudaStream_t st, bool pose) {
    const size_t smem = sizeof(SmemBwd);
    // per call: the attribute belongs to the current device (cheap next to the kernel)
    cudaFuncSetAttribute(k_field_bwd_fp32<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_field_bwd_fp32<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (pose)
        k_field_bwd_fp32<true><<<n_sm, kFieldThreads, smem, st>>>(c, params, grads, b.rays, b.cap_rays,
                                                                 b.offsets + n_rays, b.ray_id, b.t, b.feat, b.dsig_rgb,
                                                                 b.pose_s, b.pose_odd);
    else
        k_field_bwd_fp32<false><<<n_sm, kFieldThreads, smem, st>>>(c, params, grads, b.rays, b.cap_rays,
                                                                  b.offsets + n_rays, b.ray_id, b.t, b.feat,
                                                                  b.dsig_rgb, nullptr, nullptr);
}

}  // namespace nm
