// Block-level reductions shared by the SIMT kernels and the adjoint's
// reduction kernel: a fixed-order block sum and the ordered FP64 reduction of
// the chi^2 tile partials and entropy partials into the objective scalars.
#pragma once

#include <cstdint>

#include "common.cuh"
#include "internal.h"
#include "logratio.cuh"

namespace msk {

// ---------------------------------------------------------------------------
// block reductions (fixed tree: deterministic)
// ---------------------------------------------------------------------------
template <int BLOCK>
__device__ __forceinline__ double block_sum(double x, double* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = x;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0) {
        for (int i = 0; i < BLOCK / 32; ++i) r += sh[i];
    }
    __syncthreads();
    return r;  // valid in thread 0
}

__device__ __forceinline__ int image_of(const DevData& d, int c) { return d.shared ? 0 : c; }

// A pixel's gradient from its chi^2 part, beam (t0 + t1) scale with scale a power
// of two, and the entropy's part, in FP64: any beam and sum that FP32 holds.  The
// pixel's FP64 operations bound this step on large images: with the scale divided
// out and the logarithm formed again the gradient reduction took 70 us at 1024 x
// 1024, with the inverse scale and the logarithm that the entropy left in lg 41 us
// (CUDA events around the launch).
__device__ __forceinline__ double pixel_gradient(const DevData& d, float beam, float t0, float t1, double scale,
                                                 double x, const double* lg) {
    const double g = (double)beam * ((double)t0 + (double)t1);
    if (d.lambda == 0.0) return g * scale;
    return fma(g, scale, fma(d.lambda, lg ? *lg : log_ratio(x, d.G, d.ginv), d.lambda));
}

// 1 / f of a power of two f, exactly, without a division.
__device__ __forceinline__ double pow2_inverse(float f) {
    return __hiloint2double((1023 + 127 - (int)(__float_as_uint(f) >> 23)) << 20, 0);
}

// The bound projection: a pixel at I = G (or below) does not move down.
__device__ __forceinline__ double project_pixel(const DevData& d, double x, double gr) {
    // (the bits of doubles order as they do, positive G; NaN is above)
    return __double_as_longlong(x) <= __double_as_longlong(d.G) && gr > 0.0 ? 0.0 : gr;
}

// x log(x/G) of the pixel at flat index q (value x); for a line-search probe,
// whose operand is the difference max(I + alpha d, G) - I, the change against
// the base image.
__device__ __forceinline__ double entropy_term(const DevData& d, const ImgSrc& src, double x, int64_t q) {
    const double l = log_ratio(x, d.G, d.ginv);
    if (src.lg) src.lg[q] = l;
    double e = x * l;
    if (src.diff) {
        const double x0 = src.f64[q];
        e -= x0 * log_ratio(x0, d.G, d.ginv);
    }
    return e;
}

// Sums of x and y over the block, the same order every time; valid in thread 0.
template <int BLOCK>
__device__ __forceinline__ void block_sum2(double& x, double& y, double (*sh)[2]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x += __shfl_down_sync(0xffffffffu, x, o);
        y += __shfl_down_sync(0xffffffffu, y, o);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
        sh[w][0] = x;
        sh[w][1] = y;
    }
    __syncthreads();
    if (w == 0) {
        x = l < BLOCK / 32 ? sh[l][0] : 0.0;
        y = l < BLOCK / 32 ? sh[l][1] : 0.0;
#pragma unroll
        for (int o = BLOCK / 64; o > 0; o >>= 1) {
            x += __shfl_down_sync(0xffffffffu, x, o);
            y += __shfl_down_sync(0xffffffffu, y, o);
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Ordered FP64 reductions of tile partials into per-image and total scalars.
// scal layout: [0..2] = Phi, chi^2, S totals; [3 + 3i ...] per image.
// ---------------------------------------------------------------------------
// sc.splits blocks per image (ScalarArgs); block (i, q) sums a contiguous share
// of image i's chi^2 partials and entropy partials in a fixed order; the last of
// the n_images x splits blocks to finish adds the shares in order.  One block
// per image and one image need no hand-over between blocks at all, which is
// most of the time where the partials are few: 128 x 128 with 60,001
// visibilities (1,880 + 64 partials) 9.8 us in 32 blocks, 7.9 us in one (CUDA
// events around the launch, about 5 us of which are theirs), and a 64 x 64 solve
// of five iterations (324 + 16 partials, 65 reductions) 1.81 -> 1.67 ms.

// img_tmp: 2 * SCAL_SPLIT * n_images partials, then the completion counter
// (zero between evaluations)
__device__ __host__ inline unsigned* scalars_counter(double* img_tmp, int n_images) {
    return (unsigned*)(img_tmp + 2 * SCAL_SPLIT * n_images);
}

// The finished scalars (and the status word) to the host.  Whole block.
__device__ __forceinline__ void scalars_to_host(const ScalarArgs& sc, int n_images) {
    if (!sc.host) return;
    __syncthreads();
    for (int k = threadIdx.x; k < 3 + 3 * n_images; k += blockDim.x) sc.host[1 + k] = __ldcg(sc.scal + k);
    if (threadIdx.x == 0) *(int*)sc.host = *sc.status;
}

// Every thread of the block (THREADS) calls this (block-wide barriers inside).
// Returns true in every thread of the one block that has all scalars in scal
// (__ldcg reads them).
template <int THREADS>
__device__ __forceinline__ bool scalars_block(const DevData& d, const ScalarArgs& sc, int i, int q) {
    __shared__ double sh[THREADS / 32][2];
    __shared__ bool last;
    const int splits = sc.splits;
    int c_lo = d.shared ? 0 : i, c_hi = d.shared ? d.C : i + 1;
    const int64_t t0 = 4LL * sc.tile_off[c_lo], t1 = 4LL * sc.tile_off[c_hi];  // channels are contiguous
    const int64_t len = t1 - t0;
    const int64_t a = t0 + len * q / splits, b = t0 + len * (q + 1) / splits;
    double x = 0.0, y = 0.0;
    {
        // four sums: four additions and loads in flight
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        int64_t t = a + threadIdx.x;
        for (; t + 3 * THREADS < b; t += 4 * THREADS)
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] += sc.chi_part[t + k * THREADS];
        for (; t < b; t += THREADS) v[0] += sc.chi_part[t];
        x = (v[0] + v[1]) + (v[2] + v[3]);
    }
    if (sc.with_entropy) {
        const int e0 = (int)((int64_t)sc.n_ent * q / splits), e1 = (int)((int64_t)sc.n_ent * (q + 1) / splits);
        for (int e = e0 + threadIdx.x; e < e1; e += THREADS) y += sc.ent_part[(int64_t)i * sc.n_ent + e];
    }
    block_sum2<THREADS>(x, y, sh);
    auto put = [&](int im, double chi, double S) {
        sc.scal[3 + 3 * im] = chi - d.lambda * S;
        sc.scal[4 + 3 * im] = chi;
        sc.scal[5 + 3 * im] = S;
    };
    const bool alone = d.n_images * splits == 1;
    if (threadIdx.x == 0) {
        if (splits == 1) {
            put(i, x, y);
            if (alone) {
                sc.scal[0] = x - d.lambda * y;
                sc.scal[1] = x;
                sc.scal[2] = y;
            }
        } else {
            sc.img_tmp[((int64_t)i * splits + q) * 2] = x;
            sc.img_tmp[((int64_t)i * splits + q) * 2 + 1] = y;
        }
        if (!alone) {
            // the last block to finish forms the totals
            __threadfence();
            last = atomicAdd(scalars_counter(sc.img_tmp, d.n_images), 1u) == (unsigned)(d.n_images * splits) - 1;
        }
    }
    __syncthreads();
    if (alone) {
        scalars_to_host(sc, d.n_images);
        return true;
    }
    if (!last) return false;
    __threadfence();
    // Stage 2 (last block): one warp per image adds its partials (read through
    // L2) in a fixed order; thread 0 then forms the totals in image order
    if (splits > 1) {
        static_assert(SCAL_SPLIT == 32, "one partial per lane");
        for (int im = threadIdx.x >> 5; im < d.n_images; im += THREADS / 32) {
            const double* p = sc.img_tmp + ((int64_t)im * splits + (threadIdx.x & 31)) * 2;
            double c2 = __ldcg(p), s2 = __ldcg(p + 1);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                c2 += __shfl_down_sync(0xffffffffu, c2, o);
                s2 += __shfl_down_sync(0xffffffffu, s2, o);
            }
            if ((threadIdx.x & 31) == 0) put(im, c2, s2);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double ta = 0, tb = 0, tc = 0;
        for (int im = 0; im < d.n_images; ++im) {
            ta += __ldcg(sc.scal + 3 + 3 * im);
            tb += __ldcg(sc.scal + 4 + 3 * im);
            tc += __ldcg(sc.scal + 5 + 3 * im);
        }
        sc.scal[0] = ta;
        sc.scal[1] = tb;
        sc.scal[2] = tc;
        *scalars_counter(sc.img_tmp, d.n_images) = 0;  // ready for the next evaluation
    }
    scalars_to_host(sc, d.n_images);
    return true;
}

}  // namespace msk
