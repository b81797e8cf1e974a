// Internal interfaces of libmemsynth: device data views and kernel launchers.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

namespace msk {

// Device status word bits (the host maps them to mem_status).
enum : int { DEV_OK = 0, DEV_TIMEOUT = 1 };

// Consecutive visibilities of one channel (the forward kernels' unit: at most
// VIS_TILE, or TC_TILE).
struct VisTile {
    int32_t chan;
    int32_t count;
    int64_t start;
};

// Split-K unit of the tensor-core adjoint: one output block of one channel
// over a visibility range.
struct AdjUnit {
    int32_t chan;
    int32_t block;   // output block index (row-major over N/BLK x N/BLK; FP16X3: row blocks of mirror pairs)
    int64_t start;   // first visibility (global index)
    int64_t count;
};

// 1 / G for log_ratio; infinite, which takes the library's logarithm, where G times
// a number near 1 might leave the normal range.
inline double ratio_inverse(double G) { return G < 1e-300 || G > 1e300 ? HUGE_VAL : 1.0 / G; }

// Read-only problem data resident on the device.
struct DevData {
    int N;
    int C;
    int n_images;
    int shared;          // 1: one image for all channels
    double G, ginv;      // ginv = ratio_inverse(G)
    double lambda;
    const uint64_t* pa;  // frac(u dx) as 64-bit fixed-point turns
    const uint64_t* pb;  // frac(v dy)
    const double* u;     // wavelengths: launch_adj_tc_uv only (a context keeps their phases)
    const double* v;
    const double2* vo;   // observed visibilities
    const double* w;     // 1/sigma^2
    const float4* vo32;  // observed visibilities as FP32 pairs (Re hi, Im hi, Re lo, Im lo)
    const float* w32;    // 1/sigma^2 in FP32
    const float* beam;   // C*N*N
    const int64_t* off;  // C+1
    double dx, dy;       // pixel size (radians)
    // tensor-core tiling chosen by the autotuner (defaults: tc_bn(N), 4, 3)
    int fwd_bn;          // forward image column block (divides N, <= 256; N for the resident kernel)
    int fwd_stages;      // forward pipeline depth (streaming 3|4, resident 4..6)
    int adj_stages;      // adjoint pipeline depth (2 or 3)
    int chain;           // launch the evaluation's kernels as a chain (launch_chained)
};

// A launch whose grid may become resident while the kernel before it on the
// stream runs (programmatic dependent launch), if chain is set: the launch latency
// and the set-up of barriers and tensor memory overlap the kernel before.  A 64 x
// 64 evaluation 39 -> 32 us, 128 x 128 BF16X3 95 -> 90, the three maps at 256 x 256
// 235 -> 218.  Launches captured into a graph go without: a replay gains nothing
// (64 x 64: 30 us either way), and BF16X3's took 87 us instead of 83.  Its kernel calls
// chain_wait before it touches anything an earlier kernel writes, or writes
// anything an earlier kernel touches.  cluster: CTAs per cluster.
template <typename... P, typename... A>
void launch_chained(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, int chain,
                    int cluster, A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2] = {};
    unsigned n = 0;
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = cluster;
        at[n].val.clusterDim.y = at[n].val.clusterDim.z = 1;
        ++n;
    }
    if (chain) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = at;
    cfg.numAttrs = n;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Where pixel values come from: the caller's FP32 image, or the solver's FP64
// state, optionally moved along a direction and clipped: max(I + alpha_i d, G).
struct ImgSrc {
    const float* f32;
    const double* f64;
    const double* dir;
    const double* alpha;  // per image (device)
    double G;
    int diff;             // operand is max(I + alpha d, G) - I, entropy as a difference
    double* lg = nullptr; // log(I / G) per image and pixel (nullable): the entropy's pass writes
                          // it, the gradient's reads it instead of forming it again
};

// FWD_VIS: write V.  FWD_RESID: write y = w (V - V^o), chi^2 partials.
// FWD_CHI: chi^2 partials only.  FWD_CURV: 1/2 w |V|^2 partials.
// FWD_DCHI: chi^2 change for an operand that is an image difference delta,
//   Re(conj(y) F(A delta)) + 1/2 w |F(A delta)|^2, with y = w r of the base
//   image read from the y buffer.
enum FwdMode { FWD_VIS = 0, FWD_RESID = 1, FWD_CHI = 2, FWD_CURV = 3, FWD_DCHI = 4 };

// Visibilities per tile of the direct and the folded forward (VIS_TILE) and of
// the BF16X3 forward (TC_TILE), operand rows per tensor-core pipeline stage,
// and default column block.
constexpr int VIS_TILE = 128;
constexpr int TC_TILE = 64;
constexpr int TC_BK = 32;
__host__ __device__ inline int tc_bn(int N) { return N < 256 ? N : 256; }
constexpr int MEAN_L = 16;  // folded columns l that share the operand's means and scale
// First column (P) of folded column l within a part: groups of eight P columns
// followed by the eight Q columns of the same l (Q = P + 8).
__host__ __device__ inline int fold_col(int l) { return 16 * (l / 8) + l % 8; }
// Adjoint tensor-core tiling: output block side, and the multiple of
// visibilities at which units are cut.
constexpr int TCA_BK = 16;
inline int tca_blk(int N) { return N < 256 ? N : 256; }

// Message returned by mem_last_error(NULL) (thread-local).
void set_global_error(const char* msg);

// ---- launchers (all asynchronous on `st`) ----
void launch_phase_prep(int64_t Z, const double* u, const double* v, double dx, double dy,
                       uint64_t* pa, uint64_t* pb, cudaStream_t st);

// FP32 direct form: B_c = A_c * img(c) for every channel; entropy partials S_i
// per (image, block of 256 pixels) when ent_part != nullptr.
void launch_prep(const DevData& d, const ImgSrc& src, float* bout, double* ent_part, cudaStream_t st);
// BF16X3: means of every column of B_c into cmean[C][N].  psum holds
// colmean_tmp_count(N, C) entries; count holds C completion counters, zero
// between calls (each call leaves them zero).  ent_part (nullable):
// tc_ent_blocks(N) entropy partials per image.
void launch_colmean(const DevData& d, const ImgSrc& src, float* cmean, double* psum, unsigned* count,
                    double* ent_part, cudaStream_t st);
int colmean_tmp_count(int N, int C);
constexpr int COL_RB = 16;  // row blocks of the column sums
__host__ __device__ inline int tc_ent_blocks(int N) { return (N + 31) / 32 * COL_RB; }
// BF16X3: the centred operand split into 16-bit hi and lo planes in the
// forward kernel's chunk layout.
void launch_planes(const DevData& d, const ImgSrc& src, void* planes, const float* cmean, cudaStream_t st);
// FP16X3: the folded operand, centred and scaled per strip of MEAN_L columns l,
// split into planes; cmean[C][2 parts][N/2/MEAN_L] holds (P mean, Q mean, 1 /
// scale).  ymax_clear (nullable) is set to zero.  ent_part (nullable):
// fold_ent_blocks(N) entropy partials per image.
void launch_prep_fold(const DevData& d, const ImgSrc& src, void* planes, float4* cmean, float* ymax_clear,
                      double* ent_part, cudaStream_t st);
// pixels per entropy partial of launch_prep_fold, partials per image
__host__ __device__ inline int fold_ent_pixels(int N) { return N <= 256 ? 256 : 1024; }
__host__ __device__ inline int fold_ent_blocks(int N) { return (N * N + fold_ent_pixels(N) - 1) / fold_ent_pixels(N); }
// max |component| of Z visibilities into ymax[0]; the FP16X3 adjoint scales y by
// pow2_scale_for(ymax[0]).  The forward writes the same maximum of the y it
// produces (RESID mode) when given ymax (zeroed before), and so does
// launch_dirty_y.  count: two words, zero between launches.
void launch_absmax(int64_t Z, const float2* y, int num_sms, unsigned* count, float* ymax, cudaStream_t st);
__host__ __device__ inline int prep_blocks(int N) { return (int)(((int64_t)N * N + 255) / 256); }

void launch_fwd_direct(const DevData& d, const VisTile* tiles, int n_tiles, const float* B, int mode, float2* yout,
                       double* chi_part, cudaStream_t st);
// gsum: [ks][C][N*N] doubles, per-channel sums without the beam factor.
void launch_adj_direct(const DevData& d, const float2* y, double* gsum, int ks, cudaStream_t st);
int adj_direct_splits(const DevData& d, int num_sms);

// FP64 form, folded (kernels_f64.cu).  Operand: f64_operand_doubles(N) per
// channel; f64_ent_blocks(N) entropy partials per image.  The forward cuts a
// tile's work into f64_shares(...) shares, whose sums (wpart[share][Z], needed
// for more than one) a second kernel adds; returns the launches.
int64_t f64_operand_doubles(int N);
int f64_ent_blocks(int N);
int f64_shares(int N, int n_tiles, int num_sms);
int f64_adj_splits(const DevData& d, int num_sms);
void launch_prep_f64(const DevData& d, const ImgSrc& src, double* B, double* ent_part, cudaStream_t st);
int launch_fwd_f64(const DevData& d, const VisTile* tiles, int n_tiles, const double* B, int mode, double2* yout,
                   double* chi_part, double2* wpart, int shares, int64_t z_total, cudaStream_t st);
void launch_adj_f64(const DevData& d, const double2* y, double* gsum, int ks, cudaStream_t st);

// Tensor-core forms.
// FP16X3 forward on the folded image: operand streamed (any N) or resident (N <=
// 256).  For fold_combines(N) the resident form splits every tile over two
// CTAs, whose partial sums (vpart, two float4 per visibility) a second kernel
// adds.  planes and cmean from launch_prep_fold.  ymax (nullable, RESID mode): max
// |component| of the weighted residual written to yout is combined into ymax[0]
// (which the caller zeroes).  Returns the number of kernels launched.
int fold_smem_bytes(int N, int BN, int stages, int resident);
bool fold_combines(int N);
int launch_fwd_fold(const DevData& d, int resident, const VisTile* tiles, int n_tiles, const void* planes,
                    const float4* cmean, int mode, float2* yout, double* chi_part, float* ymax,
                    float4* vpart, int64_t z_total, int num_sms, uint64_t spin, int* status, cudaStream_t st);
// BF16X3 forward, streamed operand (TC_TILE tiles).
int fwd_tc_smem_bytes(int N, int BN, int stages);
void launch_fwd_tc(const DevData& d, const VisTile* tiles, int n_tiles, const void* planes, const float* cmean,
                   int mode, float2* yout, double* chi_part, int grid, uint64_t spin, int* status, cudaStream_t st);
// BF16X3 forward, resident operand (N <= 256): the image rows are cut into
// slices of fwd_rs_ks(N); each CTA keeps one slice of the operand planes in
// shared memory; the partials of several slices (FP64, [slice][visibility]) are
// combined by a second kernel, which then applies the forward mode.  Returns the
// launches.
__host__ __device__ inline int fwd_rs_ks(int N) { return N < 128 ? N : 128; }
int fwd_rs_smem_bytes(int N, int stages);
int launch_fwd_rs(const DevData& d, const VisTile* tiles, int n_tiles, const void* planes, const float* cmean,
                   int mode, float2* yout, double* chi_part, double2* vpart, int64_t z_total, int num_sms,
                   uint64_t spin, int* status, cudaStream_t st);
// The paper's gridded forward: the 2-D real-to-complex transform of every
// channel's A_c * I zero-padded to M x M (image centred), as this library's
// own FFT kernels (rows into R[C][M/2+1][N], columns into F[C][M][M/2+1]),
// then the modulated bilinear interpolation of the half spectra.
constexpr int GRID_FFT_MAX = 8192;  // M <= 8192: two M-point buffers and the roots per CTA in shared memory (196 KB)
bool grid_fft_size_ok(int N, int M);  // N even, M = 2^a q with q in {1, 3, 5, 7}, M <= GRID_FFT_MAX
void launch_grid_fft(const DevData& d, const float* img, int M, float2* R, float2* F, cudaStream_t st);
// Dirty image / PSF / residual map: weighted adjoint inputs (what: 0 data,
// 1 PSF, 2 residuals against the model in y32 / y64), and the per-channel
// image from the adjoint's FP64 sums (no primary-beam factor).
void launch_dirty_y(const DevData& d, const double* wsum, int what, int64_t z_total, float2* y32, double2* y64,
                    int num_sms, unsigned* count, float* ymax, cudaStream_t st);
void launch_dirty_out(const DevData& d, const double* gsum, int ks, float* out, cudaStream_t st);
void launch_grid_interp(const DevData& d, int M, const float2* F, int64_t z_total, float2* vis, cudaStream_t st);
// Adjoint: units sorted by CTA: CTA b runs units [cta_unit_off[b],
// cta_unit_off[b+1]) into partials of BLK x BLK floats each, which the reductions
// below sum in unit order per (channel, block).
//
// FP16X3, folded: y scaled by pow2_scale_for(ymax[0]) (the partials carry the
// scale); a unit's output block is its two D blocks.
int adj_fold_smem_bytes(int N, int stages);
void launch_adj_fold(const DevData& d, const AdjUnit* units, const int* cta_unit_off, int n_ctas, const float2* y,
                     const float* ymax, float* partial, uint64_t spin, int* status, cudaStream_t st);
// into gsum[C][N*N], without the beam factor
void launch_adj_fold_reduce(const DevData& d, const int* cb_unit_off, const float* partial, const float* ymax,
                            double* gsum, float* out32, cudaStream_t st);
// BF16X3.
int adj_tc_smem_bytes(int N, int stages);
void launch_adj_tc(const DevData& d, const AdjUnit* units, const int* cta_unit_off, int n_ctas, const float2* y,
                   float* partial, uint64_t spin, int* status, cudaStream_t st);
void launch_adj_tc_reduce(const DevData& d, const int* cb_unit_off, const float* partial, double* gsum,
                          float* out32, cudaStream_t st);
// Variant reading u, v (FP64, wavelengths) instead of the prepared phase
// increments: the caller passes d.u, d.v, d.dx, d.dy; d.pa / d.pb are unused.
void launch_adj_tc_uv(const DevData& d, const AdjUnit* units, const int* cta_unit_off, int n_ctas,
                      const float2* y, float* partial, uint64_t spin, int* status, cudaStream_t st);
// out[p] = A[p] * sum of unit partials (single channel, unit order,
// compensated FP32 two-sum).
void launch_adj_tc_reduce_out(int N, const int* cb_unit_off, const float* partial, const float* beam,
                              float* out, cudaStream_t st);
// Inputs of the objective's scalar reduction, in a launch of its own or inside
// another one (there scal == nullptr: not run).
struct ScalarArgs {
    const int* tile_off = nullptr;
    const double* chi_part = nullptr;
    const double* ent_part = nullptr;
    int with_entropy = 0;
    int n_ent = 0;   // entropy partials per image
    int splits = 1;  // blocks per image: scalar_splits
    double* scal = nullptr;
    double* img_tmp = nullptr;
    // pinned host memory (nullable): receives the status word's slot, then scal,
    // so that the caller only waits for the stream (with a copy after the kernels a
    // 64 x 64 evaluation took 58 us, without 52)
    double* host = nullptr;
    const int* status = nullptr;
};
// One block sums up to 4,096 partials of an image; beyond that SCAL_SPLIT do.
// (256 threads read 4,096 partials in four rounds of four loads; the hand-over
// between blocks costs as much as eight such rounds.)
constexpr int SCAL_SPLIT = 32;
inline int scalar_splits(int64_t partials) { return partials <= 4096 ? 1 : SCAL_SPLIT; }
// Unit-partial sum plus gradient assembly in one launch, for images of one
// channel each (not the shared-image mode); with sc.scal set, the same launch
// also forms the objective scalars (as launch_scalars).
void launch_adj_fold_reduce_grad(const DevData& d, const ImgSrc& src, const int* cb_unit_off, const float* partial,
                                 const float* ymax, int projected, float* out32, double* full64, double* proj64,
                                 const ScalarArgs& sc, cudaStream_t st);
void launch_adj_tc_reduce_grad(const DevData& d, const ImgSrc& src, const int* cb_unit_off, const float* partial,
                               int projected, float* out32, double* full64, double* proj64, const ScalarArgs& sc,
                               int n_units, cudaStream_t st);

// grad_i = sum_{c in image i} A_c * sum_k gsum[k][c] + lambda (1 + log(I/G)); optional projection.
// fast_log: log_ratio instead of the library's logarithm (tensor-core forms).
void launch_finalize(const DevData& d, const ImgSrc& src, int fast_log, const double* gsum, int ks, int projected,
                     float* out32, double* full64, double* proj64, cudaStream_t st);

// chi_part holds 4 partials per visibility tile (one per 32 visibilities),
// ent_part n_ent entropy partials per image.
// Per-image chi^2 / S / Phi into scal[3 + 3 i ...] and totals into scal[0..2].
void launch_scalars(const DevData& d, const ScalarArgs& sc, cudaStream_t st);
int scalars_tmp_doubles(int n_images);

// Solver vector kernel (FP64, per image).
// I = max(I + alpha d, G) where alpha > 0; g_prev = g everywhere.
void launch_cg_step(const DevData& d, double* I, const double* dir, const double* alpha, const double* g,
                    double* g_prev, cudaStream_t st);
void launch_clip_f32_to_f64(const DevData& d, const float* in, double* out, cudaStream_t st);
void launch_f64_to_f32(int64_t n, const double* in, float* out, cudaStream_t st);

}  // namespace msk
