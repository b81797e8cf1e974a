// SIMT kernels of libmemsynth: per-visibility phase preparation, the
// BF16X3 and FP32 operand preparation, the plain direct-sum operator pair in
// FP32 (one exponential per visibility-pixel pair, the comparator of the
// tensor-core form), gradient assembly with the entropy term and positivity
// projection, ordered FP64 reductions and the CG vector updates.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "common.cuh"
#include "internal.h"
#include "logratio.cuh"
#include "reduce.cuh"

namespace msk {

// ---------------------------------------------------------------------------
// a1: per-visibility phase increments.  frac(u dx) reduced in FP64 and held as
// a 64-bit fixed-point fraction of a turn; pixel phases are then exact integer
// multiples (Eq. 1 on the grid x_m = (m - N/2) dx).
// ---------------------------------------------------------------------------
__global__ void k_phase_prep(int64_t Z, const double* __restrict__ u, const double* __restrict__ v,
                             double dx, double dy, uint64_t* __restrict__ pa,
                             uint64_t* __restrict__ pb) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Z) return;
    pa[k] = to_fixed_turns(u[k] * dx);
    pb[k] = to_fixed_turns(v[k] * dy);
}

void launch_phase_prep(int64_t Z, const double* u, const double* v, double dx, double dy,
                       uint64_t* pa, uint64_t* pb, cudaStream_t st) {
    if (Z <= 0) return;
    k_phase_prep<<<(unsigned)((Z + 255) / 256), 256, 0, st>>>(Z, u, v, dx, dy, pa, pb);
}

// ---------------------------------------------------------------------------
// a2, BF16X3: attenuation, centring and splitting of the forward's operand
// (FP16X3: kernels_fold_prep.cu).
// ---------------------------------------------------------------------------

// Column means c_m = (1/N) sum_n B[n][m] per channel (the operand of the
// tensor-core forward is centred column by column, see k_fwd_tc), in two
// stages with a fixed summation order.  Stage 1: block (column block of 32,
// row block rb of N/COL_RB rows, channel) -> partial sums per column.  Stage
// 2, run by the channel's last stage-1 block to finish (a completion counter
// per channel, which that block resets): c_m.
__global__ void __launch_bounds__(256) k_colsum(DevData d, ImgSrc src, double* __restrict__ psum,
                                                unsigned* __restrict__ count, float* __restrict__ cmean,
                                                double* __restrict__ ent_part) {
    __shared__ double sh[8][33];
    __shared__ bool last;
    chain_next();
    chain_wait();
    const int N = d.N;
    const int64_t NN = (int64_t)N * N;
    const int c = blockIdx.z, rb = blockIdx.y;
    const int i = image_of(d, c);
    const int lane = threadIdx.x & 31;
    const int m = blockIdx.x * 32 + lane;
    const int rg = threadIdx.x >> 5;
    const int n0 = (int)((int64_t)N * rb / COL_RB), n1 = (int)((int64_t)N * (rb + 1) / COL_RB);
    // the entropy partial of an image is formed by its first channel only
    // (the others would repeat it in the shared-image mode)
    const bool ent = ent_part && !(d.shared && c != 0);
    double acc = 0.0, e = 0.0;
    if (m < N) {
        for (int n = n0 + rg; n < n1; n += 8) {
            const int64_t p = (int64_t)n * N + m;
            double x = img_value(src, i, p, NN);
            if (ent) e += entropy_term(d, src, x, (int64_t)i * NN + p);
            if (src.diff) x -= src.f64[(int64_t)i * NN + p];
            acc += (double)d.beam[(int64_t)c * NN + p] * x;
        }
    }
    if (ent) {  // uniform over the block
        const double s = block_sum<256>(e, &sh[0][0]);
        if (threadIdx.x == 0)
            ent_part[(int64_t)i * gridDim.x * gridDim.y + (int64_t)rb * gridDim.x + blockIdx.x] = -s;
    }
    sh[rg][lane] = acc;
    __syncthreads();
    if (rg == 0 && m < N) {
        double t = 0.0;
        for (int k = 0; k < 8; ++k) t += sh[k][lane];
        psum[((int64_t)c * COL_RB + rb) * N + m] = t;
        __threadfence();  // each writer's partials visible device-wide before the count below
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&count[c], 1u) == gridDim.x * gridDim.y - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // stage 2: the partials of channel c in row-block order (read through L2)
    for (int mm = threadIdx.x; mm < N; mm += blockDim.x) {
        double t = 0.0;
#pragma unroll
        for (int r = 0; r < COL_RB; ++r) t += __ldcg(psum + ((int64_t)c * COL_RB + r) * N + mm);
        cmean[(int64_t)c * N + mm] = (float)(t / N);
    }
    if (threadIdx.x == 0) count[c] = 0;  // ready for the next evaluation
}

void launch_colmean(const DevData& d, const ImgSrc& src, float* cmean, double* psum, unsigned* count,
                    double* ent_part, cudaStream_t st) {
    launch_chained(k_colsum, dim3((d.N + 31) / 32, COL_RB, d.C), 256, 0, st, d.chain, 1, d, src, psum, count, cmean,
                   ent_part);
}

int colmean_tmp_count(int N, int C) { return COL_RB * N * C; }

// BF16X3: B - c_m as hi / lo planes, per channel chunks (m-block mb, n-stage
// ks) of BN x BK elements, K-major interleaved 8x8 core matrices, hi plane then
// lo plane.
__device__ __forceinline__ int64_t tc_plane_index(int n, int m, int N, int BN) {
    int nk = N / TC_BK;
    int mb = m / BN, r = m % BN, ks = n / TC_BK, k = n % TC_BK;
    int64_t chunk = (int64_t)mb * nk + ks;
    int64_t chunk_elems = (int64_t)2 * BN * TC_BK;  // hi + lo
    int64_t off = ((int64_t)(k / 8) * (BN / 8) + r / 8) * 64 + (r % 8) * 8 + (k % 8);
    return chunk * chunk_elems + off;  // in bf16 elements; lo at + BN*BK
}

__global__ void __launch_bounds__(256) k_planes(DevData d, ImgSrc src, __nv_bfloat16* __restrict__ planes,
                                                const float* cmean) {
    chain_next();
    chain_wait();
    const int N = d.N, BN = d.fwd_bn;
    const int64_t NN = (int64_t)N * N;
    const int c = blockIdx.y;
    const int i = image_of(d, c);
    const int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (p >= NN) return;
    double x = img_value(src, i, p, NN);
    if (src.diff) x -= src.f64[(int64_t)i * NN + p];
    const int n = (int)(p / N), m = (int)(p % N);
    const double b = (double)d.beam[(int64_t)c * NN + p] * x;
    const float bf = (float)(b - (double)cmean[(int64_t)c * N + m]);
    const __nv_bfloat16 hi = __float2bfloat16_rn(bf);
    __nv_bfloat16* base = planes + (int64_t)c * 2 * NN + tc_plane_index(n, m, N, BN);
    base[0] = hi;
    base[(int64_t)BN * TC_BK] = __float2bfloat16_rn(bf - __bfloat162float(hi));
}

void launch_planes(const DevData& d, const ImgSrc& src, void* planes, const float* cmean, cudaStream_t st) {
    launch_chained(k_planes, dim3(prep_blocks(d.N), d.C), 256, 0, st, d.chain, 1, d, src, (__nv_bfloat16*)planes, cmean);
}

// The maximum of every block's mx (of 256 threads) into ymax[0]: count[0] holds
// the running maximum (non-negative floats order as their bits), count[1] the
// blocks that have added theirs; the last one hands over and leaves both zero.
__device__ __forceinline__ void max_over_blocks(float mx, unsigned* count, float* ymax) {
    __shared__ float sh[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int k = 0; k < 8; ++k) mx = fmaxf(mx, sh[k]);
    atomicMax(count, __float_as_uint(mx));
    __threadfence();
    if (atomicAdd(count + 1, 1u) != gridDim.x - 1) return;
    __threadfence();
    ymax[0] = __uint_as_float(atomicExch(count, 0u));
    count[1] = 0;
}

// max |y| over n floats.
__global__ void __launch_bounds__(256) k_absmax(int64_t n, const float2* y, unsigned* count,
                                                float* ymax) {
    chain_next();
    chain_wait();
    float mx = 0.f;
    for (int64_t k = (int64_t)blockIdx.x * 256 + threadIdx.x; k < n; k += (int64_t)gridDim.x * 256) {
        const float2 v = y[k];
        mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
    max_over_blocks(mx, count, ymax);
}

// blocks of a pass over Z visibilities: one wave of four per SM at most
static unsigned vis_blocks(int64_t Z, int num_sms) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((Z + 255) / 256, 4 * num_sms));
}

void launch_absmax(int64_t Z, const float2* y, int num_sms, unsigned* count, float* ymax, cudaStream_t st) {
    launch_chained(k_absmax, dim3(vis_blocks(Z, num_sms)), 256, 0, st, 1, 1, Z, y, count, ymax);
}

// a2, FP32 direct form: B_c = A_c I.
__global__ void __launch_bounds__(256) k_prep(DevData d, ImgSrc src, float* __restrict__ bout, double* ent_part) {
    __shared__ double sh[8];
    const int N = d.N;
    const int64_t NN = (int64_t)N * N;
    const int c = blockIdx.y;
    const int i = image_of(d, c);
    const int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const bool ent = ent_part && !(d.shared && c != 0);  // as in k_colsum
    double e = 0.0;
    if (p < NN) {
        double x = img_value(src, i, p, NN);
        double xb = x;
        if (src.diff) {
            const double x0 = src.f64[(int64_t)i * NN + p];
            xb = x - x0;
            if (ent) e = x * log(x / src.G) - x0 * log(x0 / src.G);
        } else if (ent) {
            e = x * log(x / src.G);
        }
        bout[(int64_t)c * NN + p] = (float)((double)d.beam[(int64_t)c * NN + p] * xb);
    }
    if (ent) {  // uniform over the block (one channel per block row)
        double s = block_sum<256>(e, sh);
        if (threadIdx.x == 0) ent_part[(int64_t)i * gridDim.x + blockIdx.x] = -s;
    }
}

void launch_prep(const DevData& d, const ImgSrc& src, float* bout, double* ent_part, cudaStream_t st) {
    k_prep<<<dim3(prep_blocks(d.N), d.C), 256, 0, st>>>(d, src, bout, ent_part);
}

// ---------------------------------------------------------------------------
// a12: direct-sum forward, one thread per visibility, one exponential per
// (visibility, pixel) pair.  Image rows are staged in shared memory; each row's
// sum is formed in the working precision and added to an FP64 accumulator.
// Fused epilogue (Algorithm 2 + the reduction of Algorithm 1): residual,
// weight, chi^2 tile partial.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cis_minus(uint64_t p, float& c, float& s) {
    __sincosf(phase_to_angle_f32(p), &s, &c);
}

__global__ void __launch_bounds__(128) k_fwd_direct(DevData d, const VisTile* __restrict__ tiles,
                                                    const float* __restrict__ B, int mode, float2* yout,
                                                    double* __restrict__ chi_part) {
    extern __shared__ __align__(16) unsigned char smraw[];
    float* row = (float*)smraw;
    const VisTile t = tiles[blockIdx.x];
    const int N = d.N, c0 = N / 2;
    const int64_t NN = (int64_t)N * N;
    const bool valid = (int)threadIdx.x < t.count;
    const int64_t j = t.start + (valid ? threadIdx.x : 0);
    const uint64_t a = d.pa[j], b = d.pb[j];
    const float* Bc = B + (int64_t)t.chan * NN;
    double re = 0.0, im = 0.0;
    const uint64_t pstart = phase_mul(-c0, a);
    for (int n = 0; n < N; ++n) {
        __syncthreads();
        for (int m = threadIdx.x; m < N; m += 128) row[m] = Bc[(int64_t)n * N + m];
        __syncthreads();
        uint64_t p = pstart + phase_mul(n - c0, b);
        float rr = 0, ri = 0;
        for (int m = 0; m < N; ++m) {
            float cs, sn;
            cis_minus(p, cs, sn);
            float bv = row[m];
            rr += bv * cs;
            ri -= bv * sn;
            p += a;
        }
        re += (double)rr;
        im += (double)ri;
    }
    double chi = 0.0;
    if (valid) {
        if (mode == FWD_VIS) {
            yout[j] = make_float2((float)re, (float)im);
        } else if (mode == FWD_DCHI) {
            const float2 q = yout[j];
            chi = (double)q.x * re + (double)q.y * im + 0.5 * d.w[j] * (re * re + im * im);
        } else {
            double rr = re, ri = im;
            if (mode != FWD_CURV) { rr -= d.vo[j].x; ri -= d.vo[j].y; }
            double w = d.w[j];
            chi = 0.5 * w * (rr * rr + ri * ri);
            if (mode == FWD_RESID) {
                yout[j] = make_float2((float)(w * rr), (float)(w * ri));
            }
        }
    }
    if (mode != FWD_VIS) {
        // one partial per warp (32 visibilities), summed later in a fixed order
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) chi += __shfl_down_sync(0xffffffffu, chi, o);
        if ((threadIdx.x & 31) == 0) chi_part[(int64_t)blockIdx.x * 4 + (threadIdx.x >> 5)] = chi;
    }
}

void launch_fwd_direct(const DevData& d, const VisTile* tiles, int n_tiles, const float* B, int mode, float2* yout,
                       double* chi_part, cudaStream_t st) {
    if (n_tiles <= 0) return;
    k_fwd_direct<<<n_tiles, 128, d.N * sizeof(float), st>>>(d, tiles, B, mode, yout, chi_part);
}

// ---------------------------------------------------------------------------
// a12: direct-sum adjoint (the gradient kernel of Section 2.5): each thread
// owns ADJ_PPT adjacent pixels of a row and loops over a slice of the
// channel's visibilities staged in shared memory; slices (blockIdx.z) are
// summed later in a fixed order.  Sixteen pixels per thread share each
// visibility's phase set-up (two 64-bit products) among sixteen pairs, which
// leaves the FP32 form bound by its two SFU operations per pair (2 -> 16:
// 43 -> 31 ms per launch at 256^2 with 999,600 visibilities).
// ---------------------------------------------------------------------------
constexpr int ADJ_PPT = 16;
constexpr int ADJ_CHUNK = 256;

__global__ void __launch_bounds__(128) k_adj_direct(DevData d, const float2* __restrict__ y,
                                                    double* __restrict__ gsum, int ks) {
    __shared__ uint64_t sa[ADJ_CHUNK], sb[ADJ_CHUNK];
    __shared__ float syr[ADJ_CHUNK], syi[ADJ_CHUNK];
    const int N = d.N, c0 = N / 2;
    const int64_t NN = (int64_t)N * N;
    const int c = blockIdx.y;
    const int64_t pix = ((int64_t)blockIdx.x * 128 + threadIdx.x) * ADJ_PPT;
    const bool valid = pix < NN;
    const int n = valid ? (int)(pix / N) : 0, m0 = valid ? (int)(pix % N) : 0;
    const int64_t v0 = d.off[c], v1 = d.off[c + 1];
    const int64_t len = v1 - v0;
    const int64_t k0 = v0 + len * blockIdx.z / ks, k1 = v0 + len * (blockIdx.z + 1) / ks;
    double acc[ADJ_PPT];
#pragma unroll
    for (int q = 0; q < ADJ_PPT; ++q) acc[q] = 0.0;
    for (int64_t base = k0; base < k1; base += ADJ_CHUNK) {
        int cnt = (int)((k1 - base) < ADJ_CHUNK ? (k1 - base) : ADJ_CHUNK);
        __syncthreads();
        for (int q = threadIdx.x; q < cnt; q += 128) {
            sa[q] = d.pa[base + q];
            sb[q] = d.pb[base + q];
            float2 yy = y[base + q];
            syr[q] = yy.x;
            syi[q] = yy.y;
        }
        __syncthreads();
        float part[ADJ_PPT];
#pragma unroll
        for (int q = 0; q < ADJ_PPT; ++q) part[q] = 0;
        for (int k = 0; k < cnt; ++k) {
            uint64_t p = phase_mul(m0 - c0, sa[k]) + phase_mul(n - c0, sb[k]);
            float yr = syr[k], yi = syi[k];
#pragma unroll
            for (int q = 0; q < ADJ_PPT; ++q) {
                float cs, sn;
                cis_minus(p, cs, sn);
                // Re(y e^{+i theta}) = yr cos - yi sin
                part[q] += yr * cs - yi * sn;
                p += sa[k];
            }
        }
#pragma unroll
        for (int q = 0; q < ADJ_PPT; ++q) acc[q] += (double)part[q];
    }
    if (valid) {
        double* out = gsum + ((int64_t)blockIdx.z * d.C + c) * NN + pix;
#pragma unroll
        for (int q = 0; q < ADJ_PPT; ++q) out[q] = acc[q];
    }
}

int adj_direct_splits(const DevData& d, int num_sms) {
    int64_t NN = (int64_t)d.N * d.N;
    int64_t blocks = (NN / ADJ_PPT + 127) / 128 * d.C;
    int64_t want = 4LL * num_sms;
    int ks = (int)((want + blocks - 1) / blocks);
    if (ks < 1) ks = 1;
    if (ks > 64) ks = 64;
    return ks;
}

void launch_adj_direct(const DevData& d, const float2* y, double* gsum, int ks, cudaStream_t st) {
    int64_t NN = (int64_t)d.N * d.N;
    dim3 grid((unsigned)((NN / ADJ_PPT + 127) / 128), d.C, ks);
    k_adj_direct<<<grid, 128, 0, st>>>(d, y, gsum, ks);
}

// ---------------------------------------------------------------------------
// a7: gradient assembly.  grad chi^2 of image i is the sum over its channels
// of A_c times the channel's adjoint sum (Eq. chi2gradient with the beam
// factor; Eq. chi2-multi for a shared image), plus lambda (1 + log(I/G))
// (Eq. Sgradient), then the positive projection at the bound I = G.
// ---------------------------------------------------------------------------
// SPLIT threads per pixel: group g sums the g-th part of the ks shares, and the
// groups' sums are added in order.  One thread per pixel would wait for its 152
// loads and additions in turn (64 x 64, FP64 form: 28.7 -> 12.3 us, CUDA events).
constexpr int FIN_SPLIT = 8;
template <bool FAST_LOG, int SPLIT>
__global__ void __launch_bounds__(256) k_finalize(DevData d, ImgSrc src, const double* gsum, int ks,
                                                  int projected, float* out32, double* full64,
                                                  double* proj64) {
    constexpr int PIX = 256 / SPLIT;
    __shared__ double sh[SPLIT][PIX];
    chain_next();
    chain_wait();
    const int N = d.N;
    const int64_t NN = (int64_t)N * N;
    const int i = blockIdx.y;
    const int el = threadIdx.x % PIX, grp = threadIdx.x / PIX;
    const int64_t p = (int64_t)blockIdx.x * PIX + el;
    int c_lo = d.shared ? 0 : i, c_hi = d.shared ? d.C : i + 1;
    double g = 0.0;
    if (p < NN) {
        const int ka = ks * grp / SPLIT, kb = ks * (grp + 1) / SPLIT;
        for (int c = c_lo; c < c_hi; ++c) {
            double s = 0.0;
#pragma unroll 4
            for (int k = ka; k < kb; ++k) s += gsum[((int64_t)k * d.C + c) * NN + p];
            g += (double)d.beam[(int64_t)c * NN + p] * s;
        }
    }
    if (SPLIT > 1) {
        sh[grp][el] = g;
        __syncthreads();
        if (grp != 0) return;
        for (int k = 1; k < SPLIT; ++k) g += sh[k][el];
    }
    if (p >= NN) return;
    double x = img_value(src, i, p, NN);
    if (d.lambda != 0.0) g += d.lambda * (1.0 + (FAST_LOG ? log_ratio(x, d.G, d.ginv) : log(x / d.G)));
    double gp = (x <= d.G && g > 0.0) ? 0.0 : g;
    if (full64) full64[(int64_t)i * NN + p] = g;
    if (proj64) proj64[(int64_t)i * NN + p] = gp;
    if (out32) out32[(int64_t)i * NN + p] = (float)(projected ? gp : g);
}

void launch_finalize(const DevData& d, const ImgSrc& src, int fast_log, const double* gsum, int ks, int projected,
                     float* out32, double* full64, double* proj64, cudaStream_t st) {
    const bool split = ks >= FIN_SPLIT;
    const int pix = split ? 256 / FIN_SPLIT : 256;
    auto kernel = fast_log ? k_finalize<true, 1> : split ? k_finalize<false, FIN_SPLIT> : k_finalize<false, 1>;
    launch_chained(kernel, dim3((unsigned)(((int64_t)d.N * d.N + pix - 1) / pix), d.n_images), 256, 0, st, d.chain, 1, d,
                   src, gsum, ks, projected, out32, full64, proj64);
}

// ---------------------------------------------------------------------------
// Ordered FP64 reductions of tile partials into per-image and total scalars.
// scal layout: [0..2] = Phi, chi^2, S totals; [3 + 3i ...] per image.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_scalars(DevData d, ScalarArgs sc) {
    chain_next();
    chain_wait();
    scalars_block<256>(d, sc, blockIdx.x, blockIdx.y);
}

void launch_scalars(const DevData& d, const ScalarArgs& sc, cudaStream_t st) {
    launch_chained(k_scalars, dim3(d.n_images, sc.splits), 256, 0, st, d.chain, 1, d, sc);
}

int scalars_tmp_doubles(int n_images) { return 2 * SCAL_SPLIT * n_images + 1; }

// I = max(I + alpha_i d, G) for images with alpha_i > 0; g_prev = g.
__global__ void __launch_bounds__(256) k_cg_step(DevData d, double* I, const double* __restrict__ dir,
                                                 const double* __restrict__ alpha, const double* __restrict__ g,
                                                 double* __restrict__ g_prev) {
    const int64_t NN = (int64_t)d.N * d.N;
    const int i = blockIdx.y;
    const int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (p >= NN) return;
    const int64_t q = (int64_t)i * NN + p;
    g_prev[q] = g[q];
    if (alpha[i] > 0.0) I[q] = fmax(I[q] + alpha[i] * dir[q], d.G);
}

void launch_cg_step(const DevData& d, double* I, const double* dir, const double* alpha, const double* g,
                    double* g_prev, cudaStream_t st) {
    k_cg_step<<<dim3(prep_blocks(d.N), d.n_images), 256, 0, st>>>(d, I, dir, alpha, g, g_prev);
}

__global__ void k_clip_f32_to_f64(int64_t n, const float* __restrict__ in, double* __restrict__ out,
                                  double G) {
    int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (p < n) out[p] = fmax((double)in[p], G);
}

void launch_clip_f32_to_f64(const DevData& d, const float* in, double* out, cudaStream_t st) {
    int64_t n = (int64_t)d.n_images * d.N * d.N;
    k_clip_f32_to_f64<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, in, out, d.G);
}

__global__ void k_f64_to_f32(int64_t n, const double* __restrict__ in, float* __restrict__ out) {
    int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (p < n) out[p] = (float)in[p];
}

void launch_f64_to_f32(int64_t n, const double* in, float* out, cudaStream_t st) {
    if (n <= 0) return;
    k_f64_to_f32<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, in, out);
}

}  // namespace msk

namespace msk {

// ---------------------------------------------------------------------------
// Dirty image and PSF (Appendix A, Eq. dirty and Eq. PSF): the adjoint of
// y_k = omega_k V_k (or omega_k), omega_k = w_k / (sum of w over the channel);
// the sum of the adjoint's splits per channel, without the primary beam.
// ---------------------------------------------------------------------------
// what: 0 measured visibilities, 1 PSF (V = 1), 2 residuals V° - V, with the
// model V read from y64 (FP64 form) or y32 at the same index it overwrites.
// ymax (nullable): receives the result's maximum |component|, which the FP16X3
// adjoint scales by; here it costs no pass of its own (100,003
// visibilities: three launches of 16 us together, now one of 7).
__global__ void __launch_bounds__(256) k_dirty_y(DevData d, const double* __restrict__ wsum, int what,
                                                 int64_t z_total, float2* y32, double2* y64, unsigned* count, float* ymax) {
    chain_next();
    chain_wait();
    float mx = 0.f;
    for (int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x; j < z_total; j += (int64_t)gridDim.x * 256) {
        int lo = 0, hi = d.C;
        while (hi - lo > 1) {
            const int mid = (lo + hi) / 2;
            if (d.off[mid] <= j) lo = mid;
            else hi = mid;
        }
        const double om = d.w[j] / wsum[lo];
        double2 v = what == 1 ? make_double2(1.0, 0.0) : d.vo[j];
        if (what == 2) {
            const double2 m = y64 ? y64[j] : make_double2((double)y32[j].x, (double)y32[j].y);
            v.x -= m.x;
            v.y -= m.y;
        }
        const float2 o = make_float2((float)(om * v.x), (float)(om * v.y));
        y32[j] = o;
        if (y64) y64[j] = make_double2(om * v.x, om * v.y);
        mx = fmaxf(mx, fmaxf(fabsf(o.x), fabsf(o.y)));
    }
    if (ymax) max_over_blocks(mx, count, ymax);
}

__global__ void __launch_bounds__(256) k_dirty_out(DevData d, const double* __restrict__ gsum, int ks,
                                                   float* __restrict__ out) {
    const int64_t NN = (int64_t)d.N * d.N;
    const int c = blockIdx.y;
    const int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (p >= NN) return;
    double s = 0.0;
    for (int k = 0; k < ks; ++k) s += gsum[((int64_t)k * d.C + c) * NN + p];
    out[(int64_t)c * NN + p] = (float)s;
}

void launch_dirty_y(const DevData& d, const double* wsum, int what, int64_t z_total, float2* y32, double2* y64,
                    int num_sms, unsigned* count, float* ymax, cudaStream_t st) {
    launch_chained(k_dirty_y, dim3(vis_blocks(z_total, num_sms)), 256, 0, st, d.chain, 1, d, wsum, what, z_total, y32, y64,
                   count, ymax);
}

void launch_dirty_out(const DevData& d, const double* gsum, int ks, float* out, cudaStream_t st) {
    dim3 grid(prep_blocks(d.N), d.C);
    k_dirty_out<<<grid, 256, 0, st>>>(d, gsum, ks, out);
}

}  // namespace msk
