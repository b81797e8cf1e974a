// The paper's gridded forward (Section 2.4, the steps of the objective
// evaluation; Algorithm alg:chi2gpu): attenuation, zero padding to
// M = pad N, a 2-D FFT of every channel's image on the grid, the
// phase-centre modulation and bilinear interpolation at each sample's grid
// coordinates.  An approximation of Eq. (1): its error against the exact sum
// falls about as 1/pad^2 (bilinear interpolation of a band-limited grid).
//
// The 2-D real-to-complex transform is this file's own:
//   rows    : the N non-zero rows of the padded image, two real rows per
//             complex transform of length M (z = row_a + i row_b; the two
//             spectra follow from Hermitian symmetry), half spectrum
//             k = 0..M/2 written column-major, R[c][k][n];
//   columns : for each of the M/2 + 1 frequency columns, a complex
//             transform of length M over the padded rows (only the N window
//             rows are non-zero), giving F[c][l][k].
// Each transform runs in one CTA in shared memory: a Stockham (autosorting,
// ping-pong) mixed-radix FFT with radix-4 and radix-2 stages and, for the
// odd factor of pad (3, 5, 7), one stage of direct small DFTs; the twiddles are
// the M-th roots of unity, sincospif of exact fractions of a turn, tabulated once
// per CTA (a sincospif per factor and butterfly took rows 11.7 and columns 12.0 us
// at N = 256, M = 768; 4.6 and 5.1 us with the table, the same values).
// FP32 throughout; a sample's grid coordinates come from its fixed-point phases.
#include <cstdint>

#include "common.cuh"
#include "internal.h"

namespace msk {

namespace {

constexpr int FFT_THREADS = 256;

__device__ __forceinline__ float2 c_add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 c_sub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 c_mul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// exp(-2 pi i q / d) for integers 0 <= q < d
__device__ __forceinline__ float2 c_root(int q, int d) {
    float s, c;
    sincospif(2.0f * (float)q / (float)d, &s, &c);
    return make_float2(c, -s);
}

// Table of the M-th roots exp(-2 pi i q / M) in shared memory.
__device__ __forceinline__ void root_table(float2* w, int M) {
    for (int q = threadIdx.x; q < M; q += blockDim.x) w[q] = c_root(q, M);
}

// One Stockham stage of radix RADIX (0: any odd radix up to 7 in R), Ns (a power
// of two) the product of the radices before it: butterflies of a[] into b[].
template <int RADIX>
__device__ __forceinline__ void fft_stage(const float2* a, float2* b, const float2* w, int M, int Ns, int odd) {
    const int R = RADIX ? RADIX : odd;
    const int nb = M / R, tw = nb / Ns;  // tw: table step of the twiddle exp(-2 pi i / (Ns R))
    for (int j = threadIdx.x; j < nb; j += blockDim.x) {
        const int jm = j & (Ns - 1);
        const int base = (j - jm) * R + jm;
        float2 v[7];
#pragma unroll
        for (int r = 0; r < (RADIX ? RADIX : 7); ++r) {
            if (!RADIX && r >= R) break;
            const float2 x = a[j + r * nb];
            v[r] = r == 0 ? x : c_mul(x, w[r * jm * tw]);
        }
        if (RADIX == 4) {
            const float2 s02 = c_add(v[0], v[2]), d02 = c_sub(v[0], v[2]);
            const float2 s13 = c_add(v[1], v[3]), d13 = c_sub(v[1], v[3]);
            const float2 md13 = make_float2(d13.y, -d13.x);  // -i (v1 - v3)
            b[base] = c_add(s02, s13);
            b[base + Ns] = c_add(d02, md13);
            b[base + 2 * Ns] = c_sub(s02, s13);
            b[base + 3 * Ns] = c_sub(d02, md13);
        } else if (RADIX == 2) {
            b[base] = c_add(v[0], v[1]);
            b[base + Ns] = c_sub(v[0], v[1]);
        } else {
            for (int s = 0; s < R; ++s) {
                float2 acc = v[0];
                int q = 0;  // s t mod R
#pragma unroll
                for (int t = 1; t < 7; ++t) {
                    if (t >= R) break;
                    q += s;
                    if (q >= R) q -= R;
                    acc = c_add(acc, c_mul(v[t], w[q * nb]));
                }
                b[base + s * Ns] = acc;
            }
        }
    }
    __syncthreads();
}

// Forward DFT, X[k] = sum_t x[t] exp(-2 pi i k t / M), of the M values in
// a[] (shared memory; b[] is the ping-pong buffer, w[] the roots): the factors 4
// of M first, then one 2, then the odd one.  Returns the buffer that holds the
// result.  All threads of the block take part.
__device__ float2* fft_shared(float2* a, float2* b, const float2* w, int M) {
    const int pow2 = M & -M, odd = M / pow2;
    int Ns = 1;
    auto swap = [&](int R) {
        float2* t = a;
        a = b;
        b = t;
        Ns *= R;
    };
    while (pow2 / Ns >= 4) {
        fft_stage<4>(a, b, w, M, Ns, 1);
        swap(4);
    }
    if (pow2 / Ns == 2) {
        fft_stage<2>(a, b, w, M, Ns, 1);
        swap(2);
    }
    if (odd > 1) {
        fft_stage<0>(a, b, w, M, Ns, odd);
        swap(odd);
    }
    return a;
}

// Row pass: CTA (pair q, channel c) transforms rows 2q and 2q + 1 of the N x N
// window of A_c * I (centred in the M x M padded image) and writes their half
// spectra to R[c][k][n], k = 0..M/2.
__global__ void __launch_bounds__(FFT_THREADS) k_fft_rows(DevData d, const float* img, int M,
                                                          float2* __restrict__ R) {
    extern __shared__ float2 sh[];
    float2 *a = sh, *b = sh + M, *w = sh + 2 * M;
    root_table(w, M);
    chain_next();
    chain_wait();
    const int N = d.N, o = (M - N) / 2, H = M / 2 + 1;
    const int c = blockIdx.y, n0 = 2 * blockIdx.x;
    const int i = d.shared ? 0 : c;
    const int64_t NN = (int64_t)N * N;
    const float* A = d.beam + (int64_t)c * NN;
    const float* I = img + (int64_t)i * NN;
    for (int m = threadIdx.x; m < M; m += blockDim.x) {
        const int x = m - o;
        float2 z = make_float2(0.f, 0.f);
        if (x >= 0 && x < N) {
            const int64_t p0 = (int64_t)n0 * N + x, p1 = p0 + N;
            z = make_float2(A[p0] * I[p0], A[p1] * I[p1]);
        }
        a[m] = z;
    }
    __syncthreads();
    const float2* Zs = fft_shared(a, b, w, M);
    float2* Rc = R + (int64_t)c * H * N;
    for (int k = threadIdx.x; k < H; k += blockDim.x) {
        const float2 zk = Zs[k];
        const float2 zc = Zs[(M - k) % M];
        // X_a = (Z_k + conj Z_{M-k}) / 2,  X_b = (Z_k - conj Z_{M-k}) / (2i)
        const float2 xa = make_float2(0.5f * (zk.x + zc.x), 0.5f * (zk.y - zc.y));
        const float2 xb = make_float2(0.5f * (zk.y + zc.y), -0.5f * (zk.x - zc.x));
        Rc[(int64_t)k * N + n0] = xa;
        Rc[(int64_t)k * N + n0 + 1] = xb;
    }
}

// Column pass: CTA (column k, channel c) transforms R[c][k][.] placed at the
// window rows of a length-M column and writes F[c][l][k], modulated.
__global__ void __launch_bounds__(FFT_THREADS) k_fft_cols(int N, int M, const float2* R,
                                                          float2* __restrict__ F) {
    extern __shared__ float2 sh[];
    float2 *a = sh, *b = sh + M, *w = sh + 2 * M;
    root_table(w, M);
    chain_next();
    chain_wait();
    const int o = (M - N) / 2, H = M / 2 + 1;
    const int k = blockIdx.x, c = blockIdx.y;
    const float2* Rk = R + ((int64_t)c * H + k) * N;
    for (int l = threadIdx.x; l < M; l += blockDim.x) {
        const int n = l - o;
        a[l] = (n >= 0 && n < N) ? Rk[n] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const float2* Y = fft_shared(a, b, w, M);
    float2* Fc = F + (int64_t)c * M * H;
    // times (-1)^(k+l) for the phase centre at pixel N/2
    for (int l = threadIdx.x; l < M; l += blockDim.x) {
        const float2 y = Y[l];
        Fc[(int64_t)l * H + k] = (k + l) & 1 ? make_float2(-y.x, -y.y) : y;
    }
}

// Value of the modulated transform at grid frequency (k, l), 0 <= k, l < M, from
// the half spectrum (columns 0..M/2; the rest by Hermitian symmetry of a real
// image's transform; M is even, so the modulation survives the reduction mod M).
__device__ __forceinline__ float2 grid_value(const float2* F, int M, int k, int l) {
    const int H = M / 2 + 1;
    if (k < H) return F[(int64_t)l * H + k];
    const float2 f = F[(int64_t)(l ? M - l : 0) * H + (M - k)];
    return make_float2(f.x, -f.y);
}

// A sample's grid coordinates are M frac(u dx) and M frac(v dy): integer and
// fraction of the 64-bit fixed-point phases times M.  (In FP64, products, floors
// and 64-bit remainders took 44 us for 999,600 samples at M = 768, bound by the
// FP64 units; 10 us now, bound by the gathers.)
__global__ void __launch_bounds__(256) k_grid_interp(DevData d, int M, const float2* F,
                                                     int64_t z_total, float2* __restrict__ vis) {
    chain_next();
    chain_wait();
    const int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (j >= z_total) return;
    const uint64_t pa = d.pa[j], pb = d.pb[j];
    // channel of sample j (offsets ascending)
    int lo = 0, hi = d.C;
    while (hi - lo > 1) {
        const int mid = (lo + hi) / 2;
        if (d.off[mid] <= j) lo = mid;
        else hi = mid;
    }
    const float2* Fc = F + (int64_t)lo * M * (M / 2 + 1);
    const int k = (int)__umul64hi(pa, (uint64_t)M), l = (int)__umul64hi(pb, (uint64_t)M);
    // (all 64 bits of the fractions, rounded to FP32: small ones keep their digits)
    const float fx = __ull2float_rn(pa * (uint64_t)M) * 5.421010862427522e-20f;
    const float fy = __ull2float_rn(pb * (uint64_t)M) * 5.421010862427522e-20f;
    const int k1 = k + 1 == M ? 0 : k + 1, l1 = l + 1 == M ? 0 : l + 1;
    const float2 a = grid_value(Fc, M, k, l), b = grid_value(Fc, M, k1, l);
    const float2 e = grid_value(Fc, M, k, l1), f = grid_value(Fc, M, k1, l1);
    const float w00 = (1.f - fx) * (1.f - fy), w10 = fx * (1.f - fy), w01 = (1.f - fx) * fy, w11 = fx * fy;
    vis[j] = make_float2(w00 * a.x + w10 * b.x + w01 * e.x + w11 * f.x,
                         w00 * a.y + w10 * b.y + w01 * e.y + w11 * f.y);
}

}  // namespace

bool grid_fft_size_ok(int N, int M) {
    if (N < 2 || (N & 1) || M < N || M > GRID_FFT_MAX) return false;
    int odd = M;
    while (!(odd & 1)) odd >>= 1;
    return odd == 1 || odd == 3 || odd == 5 || odd == 7;
}

void launch_grid_fft(const DevData& d, const float* img, int M, float2* R, float2* F, cudaStream_t st) {
    const int H = M / 2 + 1;
    const int smem = 3 * M * (int)sizeof(float2);
    cudaFuncSetAttribute(k_fft_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaFuncSetAttribute(k_fft_cols, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    launch_chained(k_fft_rows, dim3(d.N / 2, d.C), FFT_THREADS, smem, st, d.chain, 1, d, img, M, R);
    launch_chained(k_fft_cols, dim3(H, d.C), FFT_THREADS, smem, st, d.chain, 1, d.N, M, (const float2*)R, F);
}

void launch_grid_interp(const DevData& d, int M, const float2* F, int64_t z_total, float2* vis, cudaStream_t st) {
    if (z_total <= 0) return;
    launch_chained(k_grid_interp, dim3((unsigned)((z_total + 255) / 256)), 256, 0, st, d.chain, 1, d, M, F, z_total, vis);
}

}  // namespace msk
