// The FP64 operator pair on the folded image (the fold is defined in
// kernels_fold.cu): the same sums as Eq. (1) and its adjoint, every product and
// sum in FP64.
//
// A visibility's phase factors separate into row and column factors, which a few
// sincospi and complex products generate, and mirror pixels share them: N^2
// multiply-adds a visibility and operator pass, where one FP64 exponential per
// (visibility, pixel) pair takes about fifty operations a pair.  The FP64 units
// (1.7 operations a clock and SM) bound both kernels; everything else hides
// behind them.  64 x 64 with 10,260 visibilities, objective and gradient: 8.0 ms
// with an exponential per pair, 0.31 ms now.
#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "internal.h"
#include "reduce.cuh"

namespace msk {

namespace {

constexpr double TWO_M64 = 5.421010862427522e-20;

struct __align__(16) D4 {
    double x, y, z, w;
};

// (cos, -sin)(2 pi p / 2^64), all 64 bits of the phase
struct cd2 {
    double x, y;
};
__device__ __forceinline__ cd2 cis_neg64(uint64_t p) {
    double s, c;
    sincospi((double)(int64_t)p * (2.0 * TWO_M64), &s, &c);
    return {c, -s};
}
__device__ __forceinline__ cd2 cmul64(cd2 a, cd2 b) {
    return {fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x)};
}
// (k + 1/2) p for half-pixel coordinates: (2 k + 1) (p / 2), p signed
__device__ __forceinline__ uint64_t half_phase(int k, uint64_t p) {
    return phase_mul(2 * k + 1, (uint64_t)((int64_t)p >> 1));
}

// ---------------------------------------------------------------------------
// Operand: the four mirror sums per (j, l), [channel][l / F_LB][j][l % F_LB][4],
// columns beyond N/2 zero; an entropy partial per block.
// ---------------------------------------------------------------------------
constexpr int F_LB = 16;  // columns l per block of the forward
constexpr int F_JC = 16;  // rows j per work unit
constexpr int F_TH = 128; // visibilities per tile

__host__ __device__ inline int f64_lblocks(int N) { return (N / 2 + F_LB - 1) / F_LB; }

// A block takes f64_prep_threads(N) quadruples: a pixel's FP64 operations, about
// fifty with the entropy's logarithm, bound the kernel, so an image whose blocks of
// 256 would not fill the SMs several times over spreads in blocks of 32: 64 x 64 13.4
// us against 19.6, 256 x 256 14.2 against 19.9, 512 x 512 (256 blocks of 256) 30.1
// against 33.8; 1024 x 1024 98.9 against 98.6, where more partials cost the scalar
// reduction 2 us (CUDA events).
__host__ __device__ inline int f64_prep_threads(int N) { return N <= 512 ? 32 : 256; }
template <int THREADS>
__global__ void __launch_bounds__(THREADS) k_prep_f64(DevData d, ImgSrc src, double* __restrict__ B,
                                                  double* __restrict__ ent_part) {
    __shared__ double sh[THREADS / 32];
    const int N = d.N, M = N / 2, LP = f64_lblocks(N) * F_LB;
    const int64_t NN = (int64_t)N * N;
    const int c = blockIdx.y, i = image_of(d, c);
    const int64_t q = (int64_t)blockIdx.x * THREADS + threadIdx.x;
    const bool ent = ent_part && !(d.shared && c != 0);
    double e = 0.0;
    if (q < (int64_t)M * LP) {
        const int j = (int)(q / LP), l = (int)(q % LP);
        double f[4] = {0.0, 0.0, 0.0, 0.0};
        if (l < M) {
            double v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int n = (k & 2) ? M - 1 - j : M + j, m = (k & 1) ? M - 1 - l : M + l;
                const int64_t p = (int64_t)n * N + m;
                double x = img_value(src, i, p, NN), xb = x;
                if (src.diff) {
                    // line-search probe: the operand and the entropy term are
                    // differences from the base image
                    const double x0 = src.f64[(int64_t)i * NN + p];
                    xb = x - x0;
                    if (ent) e += x * log(x / src.G) - x0 * log(x0 / src.G);
                } else if (ent) {
                    e += x * log(x / src.G);
                }
                v[k] = (double)d.beam[(int64_t)c * NN + p] * xb;
            }
            const double sp = v[0] + v[2], sm = v[1] + v[3], dp = v[0] - v[2], dm = v[1] - v[3];
            f[0] = sp + sm;
            f[1] = sp - sm;
            f[2] = dp + dm;
            f[3] = dp - dm;
        }
        double2* out = (double2*)(B + ((((int64_t)c * f64_lblocks(N) + l / F_LB) * M + j) * F_LB + l % F_LB) * 4);
        out[0] = make_double2(f[0], f[1]);
        out[1] = make_double2(f[2], f[3]);
    }
    if (ent) {
        const double s = block_sum<THREADS>(e, sh);
        if (threadIdx.x == 0) ent_part[(int64_t)i * gridDim.x + blockIdx.x] = -s;
    }
}

// The last steps of one visibility: W turned to V = exp(i pi (a + b)) W, then
// the forward mode.  Returns the chi^2 term.
__device__ __forceinline__ double finish64(const DevData& d, int64_t j, cd2 w, int mode, double2* yout) {
    const cd2 r = cis_neg64((uint64_t)((int64_t)d.pa[j] >> 1) + (uint64_t)((int64_t)d.pb[j] >> 1));
    double re = fma(w.x, r.x, w.y * r.y), im = fma(w.y, r.x, -w.x * r.y);  // W conj(r)
    if (mode == FWD_VIS) {
        yout[j] = make_double2(re, im);
        return 0.0;
    }
    const double wt = d.w[j];
    if (mode == FWD_DCHI) {
        const double2 y = yout[j];
        return y.x * re + y.y * im + 0.5 * wt * (re * re + im * im);
    }
    if (mode != FWD_CURV) {
        re -= d.vo[j].x;
        im -= d.vo[j].y;
    }
    if (mode == FWD_RESID) yout[j] = make_double2(wt * re, wt * im);
    return 0.5 * wt * (re * re + im * im);
}

__device__ __forceinline__ void chi_warp(double chi, int mode, double* slot) {
    if (mode == FWD_VIS) return;
    // one partial per warp (32 visibilities), summed later in a fixed order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) chi += __shfl_down_sync(0xffffffffu, chi, o);
    if ((threadIdx.x & 31) == 0) *slot = chi;
}

// Forward: one thread per visibility of a tile; work units are (column block,
// F_JC rows), cut into gridDim.y contiguous shares so that a short observation
// still gives every SM eight warps.  A share's operand rows pass through shared
// memory (broadcast reads); sums per row, then over rows.
__global__ void __launch_bounds__(F_TH) k_fwd_f64(DevData d, const VisTile* __restrict__ tiles,
                                                  const double* __restrict__ B, int mode,
                                                  double2* __restrict__ yout, double* __restrict__ chi_part,
                                                  double2* __restrict__ wpart, int64_t z_total) {
    __shared__ D4 sb[F_JC][F_LB];
    const VisTile t = tiles[blockIdx.x];
    const int M = d.N / 2, jch = (M + F_JC - 1) / F_JC, units = f64_lblocks(d.N) * jch;
    const int u0 = units * blockIdx.y / gridDim.y, u1 = units * (blockIdx.y + 1) / gridDim.y;
    const bool valid = (int)threadIdx.x < t.count;
    const int64_t k = t.start + (valid ? threadIdx.x : 0);
    const uint64_t a = d.pa[k], b = d.pb[k];
    const cd2 sa = cis_neg64(a), sbv = cis_neg64(b);
    cd2 w = {0.0, 0.0};
    double cx[F_LB], yx[F_LB];
    cd2 ey = {1.0, 0.0};
    for (int u = u0; u < u1; ++u) {
        const int lb = u / jch, j0 = (u % jch) * F_JC, nj = min(F_JC, M - j0);
        __syncthreads();
        const D4* src = (const D4*)(B + (((int64_t)t.chan * f64_lblocks(d.N) + lb) * M + j0) * F_LB * 4);
        for (int q = threadIdx.x; q < nj * F_LB; q += F_TH) (&sb[0][0])[q] = src[q];
        if (u == u0 || j0 == 0) {
            cd2 e = cis_neg64(half_phase(lb * F_LB, a));
#pragma unroll
            for (int q = 0; q < F_LB; ++q) {
                cx[q] = e.x;
                yx[q] = e.y;
                e = cmul64(e, sa);
            }
        }
        if (u == u0 || j0 % 64 == 0) ey = cis_neg64(half_phase(j0, b));
        __syncthreads();
        for (int j = 0; j < nj; ++j) {
            double t0 = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;
#pragma unroll
            for (int q = 0; q < F_LB; ++q) {
                const D4 v = sb[j][q];  // ss, sa, as, aa
                t0 = fma(cx[q], v.x, t0);
                t1 = fma(yx[q], v.y, t1);
                t2 = fma(cx[q], v.z, t2);
                t3 = fma(yx[q], v.w, t3);
            }
            w.x = fma(ey.x, t0, fma(-ey.y, t3, w.x));
            w.y = fma(ey.x, t1, fma(ey.y, t2, w.y));
            ey = cmul64(ey, sbv);
        }
    }
    if (gridDim.y > 1) {
        if (valid) wpart[(int64_t)blockIdx.y * z_total + k] = make_double2(w.x, w.y);
        return;
    }
    const double chi = valid ? finish64(d, k, w, mode, yout) : 0.0;
    chi_warp(chi, mode, chi_part + (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5));
}

// The shares' sums in order, then the mode.
__global__ void __launch_bounds__(F_TH) k_fwd_f64_finish(DevData d, const VisTile* __restrict__ tiles,
                                                         const double2* __restrict__ wpart, int shares,
                                                         int64_t z_total, int mode, double2* __restrict__ yout,
                                                         double* __restrict__ chi_part) {
    const VisTile t = tiles[blockIdx.x];
    double chi = 0.0;
    if ((int)threadIdx.x < t.count) {
        const int64_t k = t.start + threadIdx.x;
        cd2 w = {0.0, 0.0};
        for (int s = 0; s < shares; ++s) {
            const double2 q = wpart[(int64_t)s * z_total + k];
            w.x += q.x;
            w.y += q.y;
        }
        chi = finish64(d, k, w, mode, yout);
    }
    chi_warp(chi, mode, chi_part + (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5));
}

// ---------------------------------------------------------------------------
// Adjoint.  With y' = y exp(-i pi (a + b)), alpha = 2 pi (j + 1/2) b, beta =
// 2 pi (l + 1/2) a, the four pixels (rows +-, columns +-) of a quadruple are
//   G = cc - (+-)(+-) ss - (+-) sc - (+-) cs,
//   cc = sum Re y' cos a cos b,  ss = sum Re y' sin a sin b,
//   sc = sum Im y' sin a cos b,  cs = sum Im y' cos a sin b.
// A block owns 32 x 32 quadruples (2 x 2 per thread) over a share of the
// channel's visibilities; per 16 visibilities half of its threads write the row
// factors (times y') and column factors to shared memory, eight per thread from
// one sincospi and a complex recurrence.
// ---------------------------------------------------------------------------
constexpr int A_T = 32;   // quadruples per block side
constexpr int A_V = 16;   // visibilities per shared-memory batch
constexpr int A_TH = 256;

__global__ void __launch_bounds__(A_TH) k_adj_f64(DevData d, const double2* __restrict__ y,
                                                  double* __restrict__ gsum, int ks) {
    __shared__ D4 rowf[A_V][A_T];  // Re y' cos, Re y' sin, Im y' sin, Im y' cos
    __shared__ double2 colf[A_V][A_T];  // cos, sin
    const int N = d.N, M = N / 2, nt = (M + A_T - 1) / A_T;
    const int64_t NN = (int64_t)N * N;
    const int c = blockIdx.y;
    const int j0 = (blockIdx.x / nt) * A_T, l0 = (blockIdx.x % nt) * A_T;
    const int64_t v0 = d.off[c], len = d.off[c + 1] - v0;
    const int64_t k0 = v0 + len * blockIdx.z / ks, k1 = v0 + len * (blockIdx.z + 1) / ks;
    const int tj = threadIdx.x / 16, tl = threadIdx.x % 16;
    double acc[2][2][4];
#pragma unroll
    for (int q = 0; q < 16; ++q) acc[q >> 3][(q >> 2) & 1][q & 3] = 0.0;
    for (int64_t base = k0; base < k1; base += A_V) {
        const int cnt = (int)min((int64_t)A_V, k1 - base);
        __syncthreads();
        // thread -> (visibility, side, 8 factors)
        if (threadIdx.x < A_V * 8) {
            const int v = threadIdx.x >> 3, part = threadIdx.x & 7, f0 = (part & 3) * 8;
            if (v < cnt) {
                const uint64_t a = d.pa[base + v], b = d.pb[base + v];
                if (part < 4) {
                    const double2 yy = y[base + v];
                    const cd2 r = cis_neg64((uint64_t)((int64_t)a >> 1) + (uint64_t)((int64_t)b >> 1));
                    const double yr = fma(yy.x, r.x, -yy.y * r.y), yi = fma(yy.x, r.y, yy.y * r.x);
                    cd2 e = cis_neg64(half_phase(j0 + f0, b));
                    const cd2 st = cis_neg64(b);
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        rowf[v][f0 + q] = D4{yr * e.x, -yr * e.y, -yi * e.y, yi * e.x};
                        e = cmul64(e, st);
                    }
                } else {
                    cd2 e = cis_neg64(half_phase(l0 + f0, a));
                    const cd2 st = cis_neg64(a);
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        colf[v][f0 + q] = make_double2(e.x, -e.y);
                        e = cmul64(e, st);
                    }
                }
            }
        }
        __syncthreads();
        for (int v = 0; v < cnt; ++v) {
            const D4 r[2] = {rowf[v][tj], rowf[v][tj + 16]};
            const double2 q[2] = {colf[v][tl], colf[v][tl + 16]};
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    acc[i][h][0] = fma(r[i].x, q[h].x, acc[i][h][0]);
                    acc[i][h][1] = fma(r[i].y, q[h].y, acc[i][h][1]);
                    acc[i][h][2] = fma(r[i].z, q[h].x, acc[i][h][2]);
                    acc[i][h][3] = fma(r[i].w, q[h].y, acc[i][h][3]);
                }
        }
    }
    double* out = gsum + ((int64_t)blockIdx.z * d.C + c) * NN;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + tj + 16 * i, l = l0 + tl + 16 * h;
            if (j >= M || l >= M) continue;
            const double cc = acc[i][h][0], ss = acc[i][h][1], sc = acc[i][h][2], cs = acc[i][h][3];
            out[(int64_t)(M + j) * N + M + l] = (cc - ss) - (sc + cs);
            out[(int64_t)(M + j) * N + M - 1 - l] = (cc + ss) - (sc - cs);
            out[(int64_t)(M - 1 - j) * N + M + l] = (cc + ss) + (sc - cs);
            out[(int64_t)(M - 1 - j) * N + M - 1 - l] = (cc - ss) + (sc + cs);
        }
}

}  // namespace

int64_t f64_operand_doubles(int N) { return (int64_t)f64_lblocks(N) * F_LB * (N / 2) * 4; }
int f64_ent_blocks(int N) {
    const int t = f64_prep_threads(N);
    return (int)(((int64_t)(N / 2) * f64_lblocks(N) * F_LB + t - 1) / t);
}

// shares of a tile's work units: eight warps per SM, four per tile
int f64_shares(int N, int n_tiles, int num_sms) {
    const int units = f64_lblocks(N) * ((N / 2 + F_JC - 1) / F_JC);
    const int want = (2 * num_sms + std::max(n_tiles, 1) - 1) / std::max(n_tiles, 1);
    return std::max(1, std::min(want, units));
}

int f64_adj_splits(const DevData& d, int num_sms) {
    const int nt = (d.N / 2 + A_T - 1) / A_T;
    const int64_t blocks = (int64_t)nt * nt * d.C;
    return (int)std::max<int64_t>(1, std::min<int64_t>(152, (2 * num_sms + blocks - 1) / blocks));
}

void launch_prep_f64(const DevData& d, const ImgSrc& src, double* B, double* ent_part, cudaStream_t st) {
    const dim3 grid(f64_ent_blocks(d.N), d.C);
    if (f64_prep_threads(d.N) == 32) k_prep_f64<32><<<grid, 32, 0, st>>>(d, src, B, ent_part);
    else k_prep_f64<256><<<grid, 256, 0, st>>>(d, src, B, ent_part);
}

int launch_fwd_f64(const DevData& d, const VisTile* tiles, int n_tiles, const double* B, int mode, double2* yout,
                   double* chi_part, double2* wpart, int shares, int64_t z_total, cudaStream_t st) {
    if (n_tiles <= 0) return 0;
    k_fwd_f64<<<dim3(n_tiles, shares), F_TH, 0, st>>>(d, tiles, B, mode, yout, chi_part, wpart, z_total);
    if (shares == 1) return 1;
    k_fwd_f64_finish<<<n_tiles, F_TH, 0, st>>>(d, tiles, wpart, shares, z_total, mode, yout, chi_part);
    return 2;
}

void launch_adj_f64(const DevData& d, const double2* y, double* gsum, int ks, cudaStream_t st) {
    const int nt = (d.N / 2 + A_T - 1) / A_T;
    k_adj_f64<<<dim3(nt * nt, d.C, ks), A_TH, 0, st>>>(d, y, gsum, ks);
}

}  // namespace msk
