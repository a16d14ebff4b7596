// k_cov.cu - marginal covariances of the tracking frontend's dense bundle
// adjustment, the producer of the per-pixel depth variances Sigma_D that weight the
// mapping loss (Sec. 3.1, Eq. cov).  The BA Hessian has the cameras/depths arrow
// structure H = [[C, E], [E^T, P]] (Eq. hessian): C the 6K x 6K camera block, P
// diagonal (one inverse depth per pixel), E block-sparse (per pixel, the 6-vectors
// of the few poses its flow residuals involve).  Then
//   H_T = C - E P^-1 E^T = L L^T,   Sigma_T = (L L^T)^-1,
//   Sigma_d = diag(P^-1 + P^-T E^T Sigma_T E P^-1).
// FP64 throughout: the reduced camera matrix of a bundle adjustment is badly
// conditioned, and the work is small (the camera block of a keyframe window has at
// most kCovMaxC rows).
// The FP64 units are what there is little of (about 2 multiply-adds per clock and SM):
// every product is taken once (the symmetric halves are not computed twice), and what
// need not be one block is spread over the SMs.
//   k_cov_schur   pixels -> sum_q e_a e_b^T / P_q into a shared-memory copy of the
//                 c x c matrix per block, flushed with FP64 atomics;
//   k_cov_chol    one block: C - that sum, Cholesky in shared memory;
//   k_cov_inv     L^-1, one warp per column;
//   k_cov_gram    Sigma_T = L^-T L^-1, one thread per element of its lower triangle;
//   k_cov_depth   one thread per pixel: 1/P + (E P^-1)_q^T Sigma_T (E P^-1)_q.
// 20 keyframes, 96 k pixels, 4 blocks per pixel: the call takes 0.67 ms on device arrays
// (2.45 before: one block for everything after the sum, with index decoding by square
// roots and one thread per column of the inverse, 1.83 ms; sums by a shared atomic per
// product, 0.344; the full squares in k_cov_depth, 0.136).
#include <cstdint>
#include <cstring>
#include <string>

#include <cuda_runtime.h>

#include "nerfmap.h"
#include "internal.h"

namespace nm {

namespace {

constexpr uint32_t kCovMaxC = 144;  // 24 keyframes
constexpr uint32_t kCovMaxB = 8;
constexpr int kCovThreads = 512;

void set_cov_error(const char* msg) { set_global_error(msg); }

__device__ __forceinline__ uint32_t tri(uint32_t i, uint32_t j) { return i * (i + 1) / 2 + j; }  // i >= j

// Column-major packed lower triangle of order c: column k starts at its diagonal.
__device__ __forceinline__ uint32_t col(uint32_t c, uint32_t k) { return k * c - k * (k - 1) / 2 - k; }  // + i

// Each warp takes a run of consecutive pixels.  Consecutive pixels mostly belong to one
// keyframe and touch the same poses, so the products e_a e_b^T / P_q of the pairs a >= b
// are summed in the lanes' registers (entry t = lane + 32 m of the pairs' 36 products)
// while the poses stay the same, and leave for the block's shared copy of the packed
// lower triangle when they change.
template <int B>
__global__ void __launch_bounds__(256) k_cov_schur(uint32_t c, const double* __restrict__ P, uint32_t p,
                                                   const int32_t* __restrict__ blk, const double* __restrict__ e,
                                                   double* __restrict__ acc, uint32_t* __restrict__ flag) {
    constexpr int kEntries = B * (B + 1) / 2 * 36, kM = (kEntries + 31) / 32;
    extern __shared__ double sh[];
    __shared__ double se[8][2][B * 6];  // per warp: e and e / P of the pixel
    __shared__ int32_t sk[8][B];        // per warp: the poses the sums belong to
    const uint32_t n_tri = c * (c + 1) / 2;
    for (uint32_t i = threadIdx.x; i < n_tri; i += blockDim.x) sh[i] = 0.0;
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    if (lane < B) sk[w][lane] = -1;
    __syncthreads();
    double sum[kM];
    uint32_t at[kM];                    // the lane's entries: 6 a + r in the low half, 6 b + col above
#pragma unroll
    for (int m = 0; m < kM; ++m) {
        const uint32_t t = lane + 32u * m, pair = t / 36u, rc = t % 36u;
        uint32_t a = 0;
        while ((a + 1) * (a + 2) / 2 <= pair) ++a;
        at[m] = (6u * a + rc / 6u) | ((6u * (pair - a * (a + 1) / 2) + rc % 6u) << 16);
        sum[m] = 0.0;
    }
    auto flush = [&]() {
#pragma unroll
        for (int m = 0; m < kM; ++m) {
            if ((int)(lane + 32u * m) >= kEntries) continue;
            uint32_t t = at[m];
            asm volatile("" : "+r"(t));  // decoded here, not kept decoded in registers for every entry
            const uint32_t ia = t & 0xffffu, ib = t >> 16;
            const uint32_t a = ia / 6u, b = ib / 6u, r = ia % 6u, cc = ib % 6u;
            const int32_t ka = sk[w][a], kb = sk[w][b];
            if (ka < 0 || kb < 0) continue;
            uint32_t i = 6u * (uint32_t)ka + r, j = 6u * (uint32_t)kb + cc;
            double v = sum[m];
            if (a == b && r < cc) continue;                     // the mirrored product of the same block
            if (a != b && ka == kb && r == cc) v += v;           // (a, b) and (b, a) meet on the diagonal
            if (i < j) {
                const uint32_t x = i;
                i = j;
                j = x;
            }
            if (i < c) atomicAdd(&sh[tri(i, j)], v);
        }
#pragma unroll
        for (int m = 0; m < kM; ++m) sum[m] = 0.0;
    };
    const uint32_t n_warps = gridDim.x * 8u, chunk = (p + n_warps - 1) / n_warps;
    const uint32_t q0 = min(p, (blockIdx.x * 8u + w) * chunk), q1 = min(p, q0 + chunk);
    for (uint32_t q = q0; q < q1; ++q) {
        const double Pq = P[q];
        if (!(Pq > 0.0)) {
            if (lane == 0) atomicOr(flag, 1u);
            continue;
        }
        const int32_t k = lane < B ? blk[(size_t)q * B + lane] : 0;
        if (__ballot_sync(0xffffffffu, lane < B && k != sk[w][lane < B ? lane : 0])) {
            flush();
            __syncwarp();
            if (lane < B) sk[w][lane] = k;
        }
        const double inv = 1.0 / Pq;
        __syncwarp();
        for (uint32_t t = lane; t < B * 6; t += 32) {
            const double v = e[(size_t)q * B * 6 + t];
            se[w][0][t] = v;
            se[w][1][t] = v * inv;
        }
        __syncwarp();
#pragma unroll
        for (int m = 0; m < kM; ++m)
            if ((int)(lane + 32u * m) < kEntries) sum[m] = fma(se[w][0][at[m] & 0xffffu], se[w][1][at[m] >> 16], sum[m]);
    }
    __syncwarp();
    if (q1 > q0) flush();
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n_tri; i += blockDim.x)
        if (sh[i] != 0.0) atomicAdd(&acc[i], sh[i]);
}

// One block: H_T = C - acc, right-looking Cholesky (column-major packed).  While the other
// warps subtract column j's products from the columns beyond j + 1, warp 0 does that for
// column j + 1 and finishes it (pivot, scaling): one barrier per column.
__global__ void __launch_bounds__(kCovThreads) k_cov_chol(uint32_t c, const double* __restrict__ C,
                                                          const double* __restrict__ acc, double* __restrict__ L,
                                                          double* __restrict__ rinv, uint32_t* __restrict__ flag) {
    extern __shared__ double A[];
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (uint32_t i = w; i < c; i += nw)
        for (uint32_t j = lane; j <= i; j += 32) A[col(c, j) + i] = C[(size_t)i * c + j] - acc[tri(i, j)];
    __syncthreads();
    bool bad = false;
    auto finish = [&](uint32_t j) {  // warp 0: pivot and scaling of column j
        double* a = A + col(c, j);
        const double d = a[j];
        bad = bad || !(d > 0.0);
        const double l = d > 0.0 ? sqrt(d) : 1.0, r = 1.0 / l;
        __syncwarp();
        for (uint32_t i = j + 1 + lane; i < c; i += 32) a[i] *= r;
        if (lane == 0) {
            a[j] = l;
            rinv[j] = r;
        }
        __syncwarp();
    };
    if (w == 0) finish(0);
    __syncthreads();
    for (uint32_t j = 0; j + 1 < c; ++j) {
        const double* a = A + col(c, j);
        for (uint32_t k = w == 0 ? j + 1 : j + 1 + w; k < c; k += w == 0 ? c : nw - 1) {
            double* b = A + col(c, k);
            const double f = a[k];
            for (uint32_t i = k + lane; i < c; i += 32) b[i] -= a[i] * f;
        }
        if (w == 0) {
            __syncwarp();
            finish(j + 1);
        }
        __syncthreads();
    }
    for (uint32_t t = threadIdx.x; t < c * (c + 1) / 2; t += blockDim.x) L[t] = A[t];
    if (threadIdx.x == 0 && bad) atomicOr(flag, 2u);
}

// Y = L^-1 by columns (Y[j][i], zeros above the diagonal): one warp per column, lane i's
// rows i, i + 32, ...; each solved entry is subtracted from the rows below it.
constexpr int kCovRows = (kCovMaxC + 31) / 32;
__global__ void __launch_bounds__(128) k_cov_inv(uint32_t c, const double* __restrict__ L,
                                                 const double* __restrict__ rinv, double* __restrict__ Y) {
    extern __shared__ double A[];
    for (uint32_t t = threadIdx.x; t < c * (c + 1) / 2; t += blockDim.x) A[t] = L[t];
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31u, j = blockIdx.x * 4u + (threadIdx.x >> 5);
    if (j >= c) return;
    double b[kCovRows];
#pragma unroll
    for (int m = 0; m < kCovRows; ++m) b[m] = lane + 32u * m == j ? 1.0 : 0.0;
#pragma unroll
    for (int m = 0; m < kCovRows; ++m) {
        for (uint32_t kk = 0; kk < 32; ++kk) {
            const uint32_t k = 32u * m + kk;
            if (k < j) continue;  // warp-uniform
            if (k >= c) break;
            const double y = __shfl_sync(0xffffffffu, b[m], kk) * rinv[k];
            const double* a = A + col(c, k);
            if (lane == kk) b[m] = y;
#pragma unroll
            for (int q = m; q < kCovRows; ++q) {
                const uint32_t i = lane + 32u * q;
                if (i > k && i < c) b[q] -= a[i] * y;
            }
        }
    }
#pragma unroll
    for (int m = 0; m < kCovRows; ++m)
        if (lane + 32u * m < c) Y[(size_t)j * c + lane + 32u * m] = b[m];
}

// Sigma_T = Y^T Y: (i, j) = sum_{k >= i} Y[k][i] Y[k][j] for i >= j, and its mirror image.
__global__ void __launch_bounds__(256) k_cov_gram(uint32_t c, const double* __restrict__ Y, double* __restrict__ ST) {
    if (blockIdx.y > blockIdx.x) return;
    const uint32_t i = blockIdx.x * 16u + (threadIdx.x & 15u), j = blockIdx.y * 16u + (threadIdx.x >> 4);
    if (i >= c || j > i) return;
    const double *yi = Y + (size_t)i * c, *yj = Y + (size_t)j * c;
    double s = 0.0;
    for (uint32_t k = i; k < c; ++k) s = fma(yi[k], yj[k], s);
    ST[(size_t)i * c + j] = s;
    ST[(size_t)j * c + i] = s;
}

// Per pixel: Sigma_d = 1/P + (E P^-1)_q^T Sigma_T (E P^-1)_q over its blocks, each pair
// of blocks once (Sigma_T is symmetric).
__global__ void __launch_bounds__(256) k_cov_depth(uint32_t c, const double* __restrict__ P, uint32_t p,
                                                   const int32_t* __restrict__ blk, const double* __restrict__ e,
                                                   uint32_t B, const double* __restrict__ ST,
                                                   double* __restrict__ Sd) {
    const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= p) return;
    const double inv = 1.0 / P[q];
    double diag = 0.0, off = 0.0;  // off: half of the mirrored products
    for (uint32_t a = 0; a < B; ++a) {
        const int32_t ka = blk[(size_t)q * B + a];
        if (ka < 0 || 6u * (uint32_t)ka >= c) continue;
        double ea[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) ea[r] = e[((size_t)q * B + a) * 6 + r];
        const double* S = ST + (size_t)(6u * (uint32_t)ka) * c;
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            const double* row = S + (size_t)r * c + 6u * (uint32_t)ka;
            diag = fma(ea[r] * row[r], ea[r], diag);
            double t = 0.0;
#pragma unroll
            for (int k = 0; k < r; ++k) t = fma(row[k], ea[k], t);
            off = fma(ea[r], t, off);
        }
        for (uint32_t b = 0; b < a; ++b) {
            const int32_t kb = blk[(size_t)q * B + b];
            if (kb < 0 || 6u * (uint32_t)kb >= c) continue;
            double eb[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) eb[k] = e[((size_t)q * B + b) * 6 + k];
#pragma unroll
            for (int r = 0; r < 6; ++r) {
                const double* row = S + (size_t)r * c + 6u * (uint32_t)kb;
                double t = 0.0;
#pragma unroll
                for (int k = 0; k < 6; ++k) t = fma(row[k], eb[k], t);
                off = fma(ea[r], t, off);
            }
        }
    }
    Sd[q] = inv + (diag + 2.0 * off) * inv * inv;
}

template <int B>
void launch_schur(uint32_t grid, size_t sh, cudaStream_t s, uint32_t c, const double* P, uint32_t p,
                  const int32_t* blk, const double* e, double* acc, uint32_t* flag) {
    // per call: the attribute belongs to the current device (cheap next to the kernel)
    cudaFuncSetAttribute(k_cov_schur<B>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(kCovMaxC * (kCovMaxC + 1) / 2 * sizeof(double)));
    k_cov_schur<B><<<grid, 256, sh, s>>>(c, P, p, blk, e, acc, flag);
}

struct DevBuf {
    void* p = nullptr;
    ~DevBuf() {
        if (p) cudaFree(p);
    }
};

}  // namespace

}  // namespace nm

using namespace nm;

extern "C" int map_marginal_covariances(const double* C, uint32_t c, const double* P, uint32_t p,
                                        const int32_t* blk, const double* e, uint32_t B, double* sigma_T,
                                        double* sigma_d, int mem_kind, void* stream) {
    clear_global_error();
    if (!C || !P || !blk || !e || !sigma_T || !sigma_d) {
        set_cov_error("map_marginal_covariances: null argument");
        return MAP_EINVAL;
    }
    if (c == 0 || c % 6 != 0 || c > kCovMaxC || B == 0 || B > kCovMaxB || p == 0) {
        set_cov_error("map_marginal_covariances: need c = 6..144 (a multiple of 6), 1 <= B <= 8, p >= 1");
        return MAP_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const bool host = mem_kind != MAP_MEM_DEVICE;
    const size_t bC = (size_t)c * c * sizeof(double), bP = (size_t)p * sizeof(double);
    const size_t bBlk = (size_t)p * B * sizeof(int32_t), bE = (size_t)p * B * 6 * sizeof(double);
    const size_t n_tri = (size_t)c * (c + 1) / 2;
    DevBuf work, inputs;
    // work: acc (packed), flag, L (packed), 1 / diag(L), L^-1
    if (cudaMalloc(&work.p, (2 * n_tri + 2 + c + (size_t)c * c) * sizeof(double)) != cudaSuccess) {
        set_cov_error("map_marginal_covariances: cudaMalloc failed");
        return MAP_ENOMEM;
    }
    double* acc = static_cast<double*>(work.p);
    uint32_t* flag = reinterpret_cast<uint32_t*>(acc + n_tri);
    double* L = acc + n_tri + 2;
    double* rinv = L + n_tri;
    double* Y = rinv + c;
    const double *dC = C, *dP = P, *dE = e;
    const int32_t* dBlk = blk;
    double *dST = sigma_T, *dSd = sigma_d;
    if (host) {
        if (cudaMalloc(&inputs.p, bC + bP + bBlk + bE + bC + bP + 64) != cudaSuccess) {
            set_cov_error("map_marginal_covariances: cudaMalloc failed");
            return MAP_ENOMEM;
        }
        char* q = static_cast<char*>(inputs.p);
        double* hC = reinterpret_cast<double*>(q);
        double* hP = reinterpret_cast<double*>(q + bC);
        double* hE = reinterpret_cast<double*>(q + bC + bP);
        int32_t* hB = reinterpret_cast<int32_t*>(q + bC + bP + bE);
        double* hST = reinterpret_cast<double*>(q + bC + bP + bE + ((bBlk + 7) / 8) * 8);
        double* hSd = hST + (size_t)c * c;
        if (cudaMemcpyAsync(hC, C, bC, cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaMemcpyAsync(hP, P, bP, cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaMemcpyAsync(hE, e, bE, cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaMemcpyAsync(hB, blk, bBlk, cudaMemcpyHostToDevice, s) != cudaSuccess) {
            set_cov_error("map_marginal_covariances: copy to the device failed");
            return MAP_ECUDA;
        }
        dC = hC;
        dP = hP;
        dE = hE;
        dBlk = hB;
        dST = hST;
        dSd = hSd;
    }
    cudaMemsetAsync(work.p, 0, n_tri * sizeof(double) + 16, s);
    const size_t sh = n_tri * sizeof(double);
    const int sh_max = (int)(kCovMaxC * (kCovMaxC + 1) / 2 * sizeof(double));
    cudaFuncSetAttribute(k_cov_chol, cudaFuncAttributeMaxDynamicSharedMemorySize, sh_max);
    cudaFuncSetAttribute(k_cov_inv, cudaFuncAttributeMaxDynamicSharedMemorySize, sh_max);
    uint32_t grid = (p + 7) / 8;
    if (grid > 152u * 2u) grid = 152u * 2u;
    using Schur = void (*)(uint32_t, size_t, cudaStream_t, uint32_t, const double*, uint32_t, const int32_t*,
                           const double*, double*, uint32_t*);
    static const Schur schur[kCovMaxB] = {launch_schur<1>, launch_schur<2>, launch_schur<3>, launch_schur<4>,
                                          launch_schur<5>, launch_schur<6>, launch_schur<7>, launch_schur<8>};
    schur[B - 1](grid, sh, s, c, dP, p, dBlk, dE, acc, flag);
    k_cov_chol<<<1, kCovThreads, sh, s>>>(c, dC, acc, L, rinv, flag);
    k_cov_inv<<<(c + 3) / 4, 128, sh, s>>>(c, L, rinv, Y);
    const uint32_t tiles = (c + 15) / 16;
    k_cov_gram<<<dim3(tiles, tiles), 256, 0, s>>>(c, Y, dST);
    k_cov_depth<<<(p + 255) / 256, 256, 0, s>>>(c, dP, p, dBlk, dE, B, dST, dSd);
    if (cudaGetLastError() != cudaSuccess) {
        set_cov_error("map_marginal_covariances: kernel launch failed");
        return MAP_ECUDA;
    }
    uint32_t hflag = 0;
    if (host) {
        if (cudaMemcpyAsync(sigma_T, dST, bC, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(sigma_d, dSd, bP, cudaMemcpyDeviceToHost, s) != cudaSuccess) {
            set_cov_error("map_marginal_covariances: copy to the host failed");
            return MAP_ECUDA;
        }
    }
    if (cudaMemcpyAsync(&hflag, flag, sizeof(uint32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        set_cov_error("map_marginal_covariances: device error");
        return MAP_ECUDA;
    }
    if (hflag & 1u) {
        set_cov_error("map_marginal_covariances: a pixel's P entry is not positive");
        return MAP_EINVAL;
    }
    if (hflag & 2u) {
        set_cov_error("map_marginal_covariances: the reduced camera matrix is not positive definite");
        return MAP_EINVAL;
    }
    return MAP_OK;
}
