// Operand preparation of the FP16X3 forward (the fold is defined in
// kernels_fold.cu): attenuation B = A I, the four mirror sums of every pixel
// quadruple, centring, scaling and splitting into FP16 hi and lo planes, and the
// image's entropy partials, in one launch.
//
// A strip is MEAN_L = 16 folded columns l of all four column types over all
// rows j.  Its means and its power-of-two operand scale need nothing outside
// it, so a cluster of up to eight CTAs, each with a share of the rows, forms
// them through distributed shared memory and no second launch has to wait for a
// whole image.  (Column means over the image with one scale per channel took a
// second launch and a completion counter: 23 + 8 us at 256 x 256 where this one
// takes 12 us, CUDA events around the launches.)
// Products and mirror sums are FP32 pairs, good to 2^-45: the 22 bits of the split are
// the same as from FP64 sums (error against 64-bit products on four kinds of images,
// 256 x 256: equal to the seven digits printed, 6.1e-9 rms of the strip's scale on
// random pixels).  The means only centre the operand, so plain FP32 sums in a fixed
// order serve.
//
// The entropy sum is independent of the strips: further CTAs of the same launch
// take 256 pixels per pass each, FP64 throughout.
#include <cooperative_groups.h>
#include <cstdint>

#include "common.cuh"
#include "internal.h"
#include "reduce.cuh"

namespace msk {

namespace {

constexpr int FP_THREADS = 256;  // 16 columns l x 16 rows j
constexpr int FP_KEEP = 4;       // row passes whose mirror sums stay in registers

// rows j per CTA are a multiple of 8 (the operand's core matrices)
int strip_cluster(int N) { return N / 16 < 8 ? N / 16 : 8; }

// a * x as a pair
__device__ __forceinline__ float2 pair_prod(float a, float x) {
    const float p = a * x;
    return make_float2(p, fmaf(a, x, -p));
}

// Attenuated value of pixel (n, m) as an FP32 pair.
__device__ __forceinline__ float2 operand_value(const DevData& d, const ImgSrc& src, int c, int i, int n, int m) {
    const int64_t NN = (int64_t)d.N * d.N, p = (int64_t)n * d.N + m;
    const float a = d.beam[(int64_t)c * NN + p];
    if (src.f32) return pair_prod(a, src.f32[(int64_t)i * NN + p]);
    double x = img_value(src, i, p, NN);
    if (src.diff) x -= src.f64[(int64_t)i * NN + p];
    x *= (double)a;
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
}

// The mirror sums ss, sa, as, aa of quadruple (j, l).
__device__ __forceinline__ void mirror_sums(const DevData& d, const ImgSrc& src, int c, int i, int j, int l,
                                            float2 (&f)[4]) {
    const int M = d.N / 2;
    const float2 pp = operand_value(d, src, c, i, M + j, M + l), pm = operand_value(d, src, c, i, M + j, M - 1 - l);
    const float2 mp = operand_value(d, src, c, i, M - 1 - j, M + l);
    const float2 mm = operand_value(d, src, c, i, M - 1 - j, M - 1 - l);
    const float2 s0 = df_add(pp.x, pp.y, mp.x, mp.y), s1 = df_add(pm.x, pm.y, mm.x, mm.y);
    const float2 d0 = df_add(pp.x, pp.y, -mp.x, -mp.y), d1 = df_add(pm.x, pm.y, -mm.x, -mm.y);
    f[0] = df_add(s0.x, s0.y, s1.x, s1.y);
    f[1] = df_add(s0.x, s0.y, -s1.x, -s1.y);
    f[2] = df_add(d0.x, d0.y, d1.x, d1.y);
    f[3] = df_add(d0.x, d0.y, -d1.x, -d1.y);
}

// KEEP: at most FP_KEEP row passes, their sums stay in registers; otherwise
// they are formed again for the second pass.
template <bool KEEP>
__global__ void __launch_bounds__(FP_THREADS) k_prep_fold(DevData d, ImgSrc src, int n_strip_ctas, int cluster,
                                                          uint16_t* __restrict__ planes, float4* __restrict__ cmean,
                                                          float* __restrict__ ymax_clear,
                                                          double* __restrict__ ent_part) {
    namespace cg = cooperative_groups;
    __shared__ __align__(16) uint16_t sp[4][2][16][16];  // column type, hi / lo, l, j
    __shared__ float red[FP_THREADS / 32][5], part[5];
    __shared__ double shd[FP_THREADS / 32];
    const int N = d.N, M = N / 2;
    const int64_t NN = (int64_t)N * N;
    chain_next();
    chain_wait();
    if ((int)blockIdx.x >= n_strip_ctas) {
        // ------------------------------------------------------ entropy
        const int n_ent = fold_ent_blocks(N), b = (int)blockIdx.x - n_strip_ctas;
        const int i = b / n_ent, e0 = b % n_ent;
        if (!ent_part || i >= d.n_images) return;  // (the grid is padded to whole clusters)
        double e = 0.0;
        for (int k = 0; k < fold_ent_pixels(N); k += FP_THREADS) {
            const int64_t p = (int64_t)e0 * fold_ent_pixels(N) + k + threadIdx.x;
            if (p < NN) e += entropy_term(d, src, img_value(src, i, p, NN), (int64_t)i * NN + p);
        }
        const double s = block_sum<FP_THREADS>(e, shd);
        if (threadIdx.x == 0) ent_part[b] = -s;
        return;
    }
    // -------------------------------------------------------------- strips
    cg::cluster_group cl = cg::this_cluster();
    const int rank = blockIdx.x % cluster, strip = (blockIdx.x / cluster) % (N / 32);
    const int c = blockIdx.x / cluster / (N / 32), i = image_of(d, c);
    // the residual maximum of the forward that follows starts at zero
    if (ymax_clear && blockIdx.x == 0 && threadIdx.x == 0) *ymax_clear = 0.f;
    const int rows = M / cluster, j0 = rank * rows, passes = (rows + 15) / 16;
    const int ll = threadIdx.x & 15, jl = threadIdx.x >> 4, l = strip * MEAN_L + ll;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float2 keep[KEEP ? FP_KEEP : 1][4];
    float acc[5] = {0.f, 0.f, 0.f, 0.f, 0.f};  // sums of the four types, max |f|
    auto take = [&](const float2 (&f)[4]) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            acc[k] += f[k].x;
            acc[4] = fmaxf(acc[4], fabsf(f[k].x));
        }
    };
    if (KEEP) {
#pragma unroll
        for (int q = 0; q < FP_KEEP; ++q)
            if (q < passes && q * 16 + jl < rows) {
                mirror_sums(d, src, c, i, j0 + q * 16 + jl, l, keep[q]);
                take(keep[q]);
            }
    } else {
        for (int q = 0; q < passes; ++q)
            if (q * 16 + jl < rows) {
                mirror_sums(d, src, c, i, j0 + q * 16 + jl, l, keep[0]);
                take(keep[0]);
            }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
        acc[4] = fmaxf(acc[4], __shfl_xor_sync(0xffffffffu, acc[4], o));
    }
    if (lane < 5) red[warp][lane] = lane == 0 ? acc[0] : lane == 1 ? acc[1] : lane == 2 ? acc[2] : lane == 3 ? acc[3] : acc[4];
    __syncthreads();
    if (threadIdx.x < 5) {
        float t = red[0][threadIdx.x];
        for (int w = 1; w < FP_THREADS / 32; ++w)
            t = threadIdx.x < 4 ? t + red[w][threadIdx.x] : fmaxf(t, red[w][threadIdx.x]);
        part[threadIdx.x] = t;
    }
    cl.sync();
    // every CTA of the cluster combines the shares in rank order
    if (threadIdx.x < 5) {
        float t = 0.f;
        for (int r = 0; r < cluster; ++r) {
            const float x = *cl.map_shared_rank(&part[threadIdx.x], r);
            t = threadIdx.x < 4 ? t + x : fmaxf(t, x);
        }
        red[0][threadIdx.x] = t;
    }
    __syncthreads();
    float mean[4], top = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        mean[k] = red[0][k] / (float)(M * MEAN_L);
        top = fmaxf(top, fabsf(mean[k]));
    }
    // The scale follows the strip down to 2^-113, where it is 2^127, the largest
    // power of two: fluxes in W/m^2/Hz (1 mJy = 1e-29) keep their 22 bits.
    const float sc = pow2_scale_for(fmaxf(red[0][4] + top, 9.62964972e-35f));
    if (rank == 0 && threadIdx.x < 2) {
        // (P mean, Q mean, 1 / scale) of the cosine and of the sine part
        cmean[((int64_t)c * 2 + threadIdx.x) * (N / 32) + strip] =
            threadIdx.x ? make_float4(mean[2], mean[3], 1.f / sc, 0.f) : make_float4(mean[0], mean[1], 1.f / sc, 0.f);
    }
    // Chunk layout of the planes: chunk (column block mb, part, row stage ks) of
    // BN columns x TC_BK rows, K-major interleaved 8 x 8 core matrices, hi plane
    // then lo plane.  A pass's values go through shared memory to 16-byte rows
    // (8 consecutive j of one column), one per thread.
    const int BN = d.fwd_bn, nk = M / TC_BK;
    const int t8 = threadIdx.x & 1, sl = (threadIdx.x >> 1) & 15, pl = (threadIdx.x >> 5) & 1, ty = threadIdx.x >> 6;
    const int col = fold_col(strip * MEAN_L + sl) + (ty & 1) * 8, mb = col / BN, r = col % BN;
    uint16_t* dst0 = planes + (int64_t)c * 2 * NN + (int64_t)pl * BN * TC_BK + (r / 8) * 64 + (r % 8) * 8;
    auto emit = [&](int q, const float2 (&f)[4]) {
        if (q * 16 + jl < rows) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 v = df_add(f[k].x, f[k].y, -mean[k], 0.f);
                uint32_t hi, lo;
                split_f16x2((v.x + v.y) * sc, 0.f, hi, lo);
                sp[k][0][ll][jl] = (uint16_t)hi;
                sp[k][1][ll][jl] = (uint16_t)lo;
            }
        }
        __syncthreads();
        const int jr = q * 16 + t8 * 8;  // first row of this thread's store
        if (jr < rows) {
            const int j = j0 + jr, ks = j / TC_BK, kk = j % TC_BK;
            const int64_t chunk = (int64_t)(2 * mb + (ty >> 1)) * nk + ks;
            *(uint4*)(dst0 + chunk * 2 * BN * TC_BK + (int64_t)(kk / 8) * (BN / 8) * 64) =
                *(const uint4*)&sp[ty][pl][sl][t8 * 8];
        }
        __syncthreads();
    };
    if (KEEP) {
#pragma unroll
        for (int q = 0; q < FP_KEEP; ++q)
            if (q < passes) emit(q, keep[q]);
    } else {
        for (int q = 0; q < passes; ++q) {
            if (q * 16 + jl < rows) mirror_sums(d, src, c, i, j0 + q * 16 + jl, l, keep[0]);
            emit(q, keep[0]);
        }
    }
    cl.sync();  // the shares stay until every CTA has read them
}

}  // namespace

void launch_prep_fold(const DevData& d, const ImgSrc& src, void* planes, float4* cmean, float* ymax_clear,
                      double* ent_part, cudaStream_t st) {
    const int cluster = strip_cluster(d.N), strips = d.N / 32 * d.C * cluster;
    const int ent = ent_part ? fold_ent_blocks(d.N) * d.n_images : 0;
    const bool keep = d.N / 2 / cluster <= 16 * FP_KEEP;
    launch_chained(keep ? k_prep_fold<true> : k_prep_fold<false>,
                   dim3((unsigned)(strips + (ent + cluster - 1) / cluster * cluster)), FP_THREADS, 0, st, d.chain,
                   cluster, d, src, strips, cluster, (uint16_t*)planes, cmean, ymax_clear, ent_part);
}

}  // namespace msk
