// Device pieces of a BOS reconstruction iteration (Sec. 2.4, Sec. 3.2, without the PINN
// terms): a minibatch of random pixels, L_BOS over that minibatch, and the AdaBelief
// update of the voxel temperatures.
//
//   sample_pixels_kernel -- k-th index = splitmix64 output (draw * npix + k + 1) for the seed,
//                           reduced to [0, n_pixels) by 128-bit multiply-high (uniform)
//   loss_pixels_kernel   -- loss = s sum_k (target[pix_k] - I_k)^2, dL/dI_k = -2 s (target[pix_k] - I_k)
//   counter_add_kernel   -- an on-device iteration counter (draw and step numbers of a
//                           captured CUDA graph)
//   sort_pixels_kernel   -- orders a minibatch by the Morton key of its pixels, so that each
//                           warp of the tracers gets neighbouring pixels (coherent rays)
//   adabelief_kernel     -- AdaBelief (Zhuang et al., NeurIPS 2020):
//                             m = b1 m + (1 - b1) g,  s = b2 s + (1 - b2) (g - m)^2 + eps,
//                             theta -= lr (m / (1 - b1^t)) / (sqrt(s / (1 - b2^t)) + eps)
#include <math.h>

#include "../../include/bos.h"
#include "bos_device.cuh"
#include "bos_internal.h"

namespace bos {

__global__ void sample_pixels_kernel(int32_t* __restrict__ pix, long long npix, unsigned long long n_pixels,
                                     unsigned long long seed, unsigned long long draw0,
                                     const unsigned long long* __restrict__ draw_dev) {
    const unsigned long long draw = draw0 + (draw_dev ? *draw_dev : 0ULL);
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < npix;
         k += (long long)gridDim.x * blockDim.x) {
        unsigned long long z = splitmix64_output(seed, draw * (unsigned long long)npix + (unsigned long long)k + 1ULL);
        pix[k] = (int32_t)__umul64hi(z, n_pixels);
    }
}

__global__ void loss_pixels_kernel(const float* __restrict__ I, const float* __restrict__ target,
                                   const int32_t* __restrict__ pix, long long npix, float scale, double* loss,
                                   float* __restrict__ dLdI) {
    double acc = 0.0;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < npix;
         k += (long long)gridDim.x * blockDim.x) {
        const float t = __ldg(target + pix[k]);
        const double r = (double)t - (double)I[k];
        acc += r * r;
        if (dLdI) dLdI[k] = (-2.0f * scale) * (t - I[k]);
    }
    for (int m = 16; m >= 1; m >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, m);
    __shared__ double part[32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += part[i];
        atomicAdd(loss, (double)scale * s);
    }
}

__global__ void adabelief_kernel(float* __restrict__ theta, const float* __restrict__ grad, float* __restrict__ m,
                                 float* __restrict__ s, long long n, float lr, float b1, float b2, float eps,
                                 long long step0, const unsigned long long* __restrict__ step_dev) {
    // bias corrections 1 / (1 - b^t) for step t (t >= 1)
    const float t = (float)(step0 + (long long)(step_dev ? *step_dev : 0ULL));
    const float c1 = 1.0f / (1.0f - powf(b1, t));
    const float c2 = 1.0f / (1.0f - powf(b2, t));
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float g = grad[i];
        const float mi = b1 * m[i] + (1.0f - b1) * g;
        const float d = g - mi;
        const float si = b2 * s[i] + (1.0f - b2) * d * d + eps;
        m[i] = mi;
        s[i] = si;
        theta[i] -= lr * (mi * c1) / (sqrtf(si * c2) + eps);
    }
}

__global__ void counter_add_kernel(unsigned long long* c, unsigned long long inc) { *c += inc; }

// Interleave the bits of x (even positions) and y (odd positions), 16 bits each.
__device__ __forceinline__ uint32_t morton2(uint32_t x, uint32_t y) {
    auto spread = [](uint32_t v) {
        v &= 0xffffu;
        v = (v | (v << 8)) & 0x00ff00ffu;
        v = (v | (v << 4)) & 0x0f0f0f0fu;
        v = (v | (v << 2)) & 0x33333333u;
        v = (v | (v << 1)) & 0x55555555u;
        return v;
    };
    return spread(x) | (spread(y) << 1);
}

// One block sorts a pixel list (n <= kSortMax) by the Morton key of (px, py): a least-significant
// digit radix sort, eight bits per pass, as many passes as the largest key has digits (two for
// a 100 x 100 image).  Warp w owns elements [32 w R, 32 (w + 1) R) in R rounds of a lane each; the
// lanes of a round that share a digit find one another with match.any, so ranks are stable and
// need no atomics.  Elements wait in registers while the block scatters them through shared
// memory.  What bounds it: the latency of its dependent steps on the one SM.  A reconstruction
// iteration of 5000 pixels (64^3 cells, 2 rays each): 528 us with the bitonic sort that stood
// here, whose 91 passes took 107 us, 436 us so.
// A warp's counters are a row of 257: counting (any digit) and the scan (8 digits x 4 groups of
// warps per warp) both spread over the banks.
constexpr int kSortMax = 16384;
constexpr int kSortThreads = 1024;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortRow = 257;

constexpr size_t sort_smem_bytes(int n) { return (2 * (size_t)n + kSortWarps * kSortRow) * sizeof(uint32_t); }

template <int ROUNDS>
__global__ void __launch_bounds__(kSortThreads) sort_pixels_kernel(int32_t* __restrict__ pix, int n, int width) {
    extern __shared__ uint32_t sh[];
    uint32_t* const keys = sh;
    uint32_t* const vals = sh + n;
    uint32_t* const hist = sh + 2 * n;
    __shared__ uint32_t wsum[kSortWarps], all_bits;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int R = (n + kSortThreads - 1) / kSortThreads;      // <= ROUNDS
    const int first = w * 32 * R + lane;
    uint32_t* const mine = hist + w * kSortRow;
    uint32_t key[ROUNDS], val[ROUNDS], rank[ROUNDS], bits = 0;
    if (threadIdx.x == 0) all_bits = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int e = first + 32 * r;
        key[r] = val[r] = rank[r] = 0;
        if (r < R && e < n) {
            val[r] = (uint32_t)pix[e];
            key[r] = morton2(val[r] % (uint32_t)width, val[r] / (uint32_t)width);
            bits |= key[r];
        }
    }
    bits = __reduce_or_sync(0xffffffffu, bits);
    if (lane == 0) atomicOr(&all_bits, bits);
    __syncthreads();
    bits = all_bits;
    for (int shift = 0; shift < 32 && (bits >> shift) != 0; shift += 8) {
        for (int i = threadIdx.x; i < kSortWarps * kSortRow; i += kSortThreads) hist[i] = 0;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r) {
            const bool on = r < R && first + 32 * r < n;
            const unsigned act = __ballot_sync(0xffffffffu, on);
            if (on) {
                const uint32_t d = (key[r] >> shift) & 255u;
                const unsigned peers = __match_any_sync(act, d);
                const uint32_t before = mine[d];
                rank[r] = before + __popc(peers & ((1u << lane) - 1u));
                __syncwarp(act);
                if (lane == __ffs(peers) - 1) mine[d] = before + __popc(peers);
            }
            __syncwarp();
        }
        __syncthreads();
        // exclusive prefix sums over (digit, warp): thread t takes digit t / 4 of warps 8 (t % 4) ..
        uint32_t c[8], sum = 0;
        uint32_t* const col = hist + (threadIdx.x & 3) * 8 * kSortRow + (threadIdx.x >> 2);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            c[k] = col[k * kSortRow];
            sum += c[k];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int m = 1; m < 32; m <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, incl, m);
            if (lane >= m) incl += o;
        }
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        uint32_t base = lane < w ? wsum[lane] : 0u;
        base = __reduce_add_sync(0xffffffffu, base) + incl - sum;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            col[k * kSortRow] = base;
            base += c[k];
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r)
            if (r < R && first + 32 * r < n) {
                const uint32_t at = mine[(key[r] >> shift) & 255u] + rank[r];
                keys[at] = key[r];
                vals[at] = val[r];
            }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r)
            if (r < R && first + 32 * r < n) {
                key[r] = keys[first + 32 * r];
                val[r] = vals[first + 32 * r];
            }
    }
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r)
        if (r < R && first + 32 * r < n) pix[first + 32 * r] = (int32_t)val[r];
}

template <int ROUNDS>
static cudaError_t launch_sort_pixels(int32_t* pix, int n, int width, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(sort_pixels_kernel<ROUNDS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sort_smem_bytes(ROUNDS * kSortThreads));
    if (e != cudaSuccess) return e;
    sort_pixels_kernel<ROUNDS><<<1, kSortThreads, sort_smem_bytes(n), st>>>(pix, n, width);
    return cudaGetLastError();
}

}  // namespace bos

namespace {
int sms_of_current() {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}
}  // namespace

extern "C" {

bos_status_t bos_sample_pixels(int32_t* pix_dev, int64_t npix, int64_t n_pixels, uint64_t seed, uint64_t draw,
                               const uint64_t* draw_dev, void* stream) {
    if (!pix_dev || npix <= 0 || n_pixels <= 0 || n_pixels > INT32_MAX) {
        bos::set_last_error("bos_sample_pixels: need npix > 0 and 0 < n_pixels <= 2^31 - 1");
        return BOS_ERR_INVALID_ARG;
    }
    bos::sample_pixels_kernel<<<sms_of_current() * 4, 256, 0, (cudaStream_t)stream>>>(
        pix_dev, npix, (unsigned long long)n_pixels, seed, draw, (const unsigned long long*)draw_dev);
    return cudaGetLastError() == cudaSuccess ? BOS_OK : BOS_ERR_CUDA;
}

bos_status_t bos_loss_l2_pixels(const float* I_dev, const float* target_dev, const int32_t* pix_dev, int64_t npix,
                                float scale, double* loss_dev, float* dLdI_dev, void* stream) {
    if (!I_dev || !target_dev || !pix_dev || !loss_dev || npix <= 0 || !(scale > 0.0f) || !isfinite(scale)) {
        bos::set_last_error("bos_loss_l2_pixels: bad argument");
        return BOS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(loss_dev, 0, sizeof(double), st) != cudaSuccess) return BOS_ERR_CUDA;
    bos::loss_pixels_kernel<<<sms_of_current() * 4, 256, 0, st>>>(I_dev, target_dev, pix_dev, npix, scale,
                                                                   loss_dev, dLdI_dev);
    return cudaGetLastError() == cudaSuccess ? BOS_OK : BOS_ERR_CUDA;
}

bos_status_t bos_adabelief_step(float* theta_dev, const float* grad_dev, float* m_dev, float* s_dev, int64_t n,
                                float lr, float beta1, float beta2, float eps, int64_t step, const uint64_t* step_dev,
                                void* stream) {
    if (!theta_dev || !grad_dev || !m_dev || !s_dev || n <= 0 || (step < 1 && !step_dev) || step < 0 ||
        !(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f)) {
        bos::set_last_error("bos_adabelief_step: bad argument");
        return BOS_ERR_INVALID_ARG;
    }
    bos::adabelief_kernel<<<sms_of_current() * 4, 256, 0, (cudaStream_t)stream>>>(
        theta_dev, grad_dev, m_dev, s_dev, n, lr, beta1, beta2, eps, (long long)step,
        (const unsigned long long*)step_dev);
    return cudaGetLastError() == cudaSuccess ? BOS_OK : BOS_ERR_CUDA;
}

bos_status_t bos_sort_pixels(int32_t* pix_dev, int64_t npix, int width, int height, void* stream) {
    if (!pix_dev || npix <= 0 || npix > bos::kSortMax || width <= 0 || height <= 0 || width > 65535 ||
        height > 65535) {
        bos::set_last_error("bos_sort_pixels: need 1 <= npix <= 16384 and an image of at most 65535 x 65535");
        return BOS_ERR_INVALID_ARG;
    }
    const int n = (int)npix;
    const cudaStream_t st = (cudaStream_t)stream;
    const cudaError_t e = n <= 2 * bos::kSortThreads   ? bos::launch_sort_pixels<2>(pix_dev, n, width, st)
                          : n <= 8 * bos::kSortThreads ? bos::launch_sort_pixels<8>(pix_dev, n, width, st)
                                                       : bos::launch_sort_pixels<16>(pix_dev, n, width, st);
    return e == cudaSuccess ? BOS_OK : BOS_ERR_CUDA;
}

bos_status_t bos_counter_add(uint64_t* counter_dev, uint64_t inc, void* stream) {
    if (!counter_dev) {
        bos::set_last_error("bos_counter_add: NULL counter");
        return BOS_ERR_INVALID_ARG;
    }
    bos::counter_add_kernel<<<1, 1, 0, (cudaStream_t)stream>>>((unsigned long long*)counter_dev, inc);
    return cudaGetLastError() == cudaSuccess ? BOS_OK : BOS_ERR_CUDA;
}

}  // extern "C"
