// Tensor-core forward operator of the FP16X3 form (Eq. 1 on the pixel grid) with
// the fused per-visibility reduction, residual, weight and chi^2 partials.
//
// Folded image.  About the point half a pixel below pixel N/2 the grid is
// symmetric: row n = N/2 + j sits at j + 1/2 and row N/2 - 1 - j at -(j + 1/2),
// j = 0 .. N/2 - 1, and likewise for the columns.  With
//   c_j + i y_j = exp(-2 pi i (j + 1/2) b),  b = frac(v dy)   (x side: a, l)
// and the four mirror sums of a pixel quadruple (first sign: rows, second:
// columns)  Bss = B++ + B+- + B-+ + B--,  Bsa = B++ - B+- + B-+ - B--,
//           Bas = B++ + B+- - B-+ - B--,  Baa = B++ - B+- - B-+ + B--,
//   V = exp(i pi (a + b)) sum_l [ c_l Tss_l - y_l Taa_l + i (y_l Tsa_l + c_l Tas_l) ],
//   Tss, Tsa = sum_j c_j (Bss, Bsa)     the cosine part,
//   Tas, Taa = sum_j y_j (Bas, Baa)     the sine part.
// Each part is a real contraction over N/2 rows with N columns, so a
// visibility takes N^2 multiply-adds and N table entries where the unfolded
// sum takes 2 N^2 and 2 N: half the tensor-core work and half the table
// generation, with exactly the same sum.
//
// Columns of a part: groups of 16, eight P columns (multiplied by c_l: Tss or
// Tas) and the eight Q columns (multiplied by y_l: Tsa or Taa) of the same l.
//
// The operand is centred, B' = B - cm, with one mean cm per column type over
// all rows j and MEAN_L neighbouring l (a strip, which also has a scale), and T = sum_j t_j B'_j + cm S with the
// closed forms
//   sum_j c_j = sin(pi N b) / (2 sin(pi b)),  sum_j y_j = -sin^2(pi N b / 2) / sin(pi b).
// For low spatial frequencies the uncentred partial sums grow monotonically
// and the tensor core's FP32 accumulation (which rounds towards zero) then
// shrinks T systematically; the centred sums wander around zero instead.
// (A mean per column measured no better than one per MEAN_L columns, and costs
// the epilogue a fifth of its instructions; no mean at all is up to four times
// worse on smooth images.)
//
// A tile is 128 visibilities, one row of the M = 128 MMA each (TMEM lane =
// visibility).  The two parts of a column block alternate between the two
// TMEM accumulators (2 x BN columns) and between two groups of four epilogue
// warps, so that one part drains while the other accumulates.  A stage is 32
// rows j (two K steps, hi x lo, lo x hi, hi x hi): 768 clocks of MMA work at
// BN = 256.  One accumulation covers at most F2_KSEG rows j (256 image rows):
// every MMA rounds its addition into the FP32 accumulator towards zero, a
// shrink of up to one ulp each; larger images run several accumulations per
// column block and the epilogue folds each into the same compensated sums.
// (Accumulations twice as long halve the drains, 1.60 -> 1.50 ms at 1024 x 1024
// with 499,968 visibilities, but raise the rms error of V from 0.6e-6 to 1.0e-6,
// and above the unfolded kernel's in some images.)
//
// Operand residency (template RES):
//   RES_STREAM  the operand chunk of a stage streams from L2 next to the tables
//               (any N);
//   RES_BOTH    (N <= 128) both parts of the channel's operand stay in shared
//               memory; the correction products of a whole accumulation are
//               issued before its main ones, while the accumulator is small;
//   RES_PART    (N = 256) a CTA keeps one part (128 KB) and writes partial
//               sums; k_fold_combine adds the parts and applies the mode.
//
// Roles (five warpgroups): warps 0-3 and 4-7 epilogue groups; warp 8 MMA issue
// (converged, one elected lane) + TMEM owner + resident copies, warp 9 copies
// of the streamed operand, warps 10 and 11 (RES_BOTH: 9 too) finish the tiles (both
// parts' sums -> V -> mode); warps 12-19 table producers.  Every SM sub-partition holds two
// epilogue warps, two producers and one of the others; the register split
// gives the epilogue 128 registers.  Every mbarrier wait is bounded.
//
// What bounds it: at 256 x 256 with 999,600 visibilities 0.22 ms, against 0.51 ms
// for the unfolded kernel it replaces (CUDA events around the launch); a
// 128 x 256 x 16 MMA takes 128 clocks, so the MMAs alone need 0.16 ms.  With the
// table and the epilogue arithmetic taken out it takes 0.20 ms: the rest is the
// issue path.  Four producer warps instead of eight, or an epilogue without the
// register split and the finishing warps, took 0.27 to 0.30 ms: each warp issues
// an instruction every six or seven clocks, and a part's drain (256 columns,
// about 700 instructions) has to end within the other part's 3,072 clocks of
// MMA work.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace msk {

namespace {

enum Residency { RES_STREAM = 0, RES_BOTH = 1, RES_PART = 2 };

constexpr int F2_MAX_STAGES = 6;
constexpr int FW_PRODUCERS = 8;  // producer warps: two groups of four, alternate stages
constexpr int FW_THREADS = 32 * (12 + FW_PRODUCERS);
// registers per thread: at launch, epilogue, producers, the other warpgroup
constexpr int FW_REGS = 96, FW_REGS_EPI = 128, FW_REGS_PROD = 72, FW_REGS_MISC = 80;
static_assert(8 * FW_REGS_EPI + FW_PRODUCERS * FW_REGS_PROD + 4 * FW_REGS_MISC <= (12 + FW_PRODUCERS) * FW_REGS,
              "the shares add up to the registers at launch");
constexpr int F2_APLANE = 128 * TC_BK * 2;            // bytes of one A plane (hi or lo), 8 KB
constexpr int F2_ABYTES = 2 * F2_APLANE;
constexpr int F2_KSEG = 128;                          // rows j per accumulation (at most)
// Epilogue phase factors advance by complex recurrence: PHASE_REFRESH chunks by
// one step, the next such group by another (a step's own rounding accumulates
// linearly).
constexpr int PHASE_REFRESH = 4;

__host__ __device__ inline int f2_chunk_bytes(int BN) { return 2 * BN * TC_BK * 2; }  // hi + lo
__host__ __device__ inline uint32_t f2_tmem_cols(int BN) {
    uint32_t c = 32;
    while ((int)c < 2 * BN) c <<= 1;
    return c;
}

struct F2Shared {
    uint64_t full[F2_MAX_STAGES];   // four producer warps (+ the copy warp once the stage's streamed chunk landed)
    uint64_t bfull[F2_MAX_STAGES];  // streamed chunk (transaction bytes; watched by the copy warp)
    uint64_t empty[F2_MAX_STAGES];  // MMA completion (tcgen05.commit)
    uint64_t tfull[2];
    uint64_t tempty[2];   // 4 epilogue warps
    uint64_t xfull[2];    // both parts' sums of a tile (8 epilogue warps)
    uint64_t xempty[2];   // both halves of a tile read by finishing warps
    uint64_t bres;        // resident operand copy (transaction bytes)
    uint64_t bfree;       // MMAs reading the resident operand done
    uint64_t drain;
    uint32_t tmem_base;
    int abort;
};

// Dynamic shared memory: [resident operand][ring][sums: 2 slots x 2 parts x 128 float4].
__host__ __device__ inline int f2_resident_bytes(int N, int res) {
    const int part = N / 2 * N * 4;  // N/2 rows x N columns, hi + lo
    return res == RES_STREAM ? 0 : res == RES_BOTH ? 2 * part : part;
}
__host__ __device__ inline int f2_stage_bytes(int BN, int res) {
    return F2_ABYTES + (res == RES_STREAM ? f2_chunk_bytes(BN) : 0);
}
__host__ inline int f2_smem_bytes(int N, int BN, int stages, int res) {
    return f2_resident_bytes(N, res) + stages * f2_stage_bytes(BN, res) +
           (res == RES_PART ? 0 : 2 * 2 * 128 * 16) + 1024;
}

// A visibility's last steps: from both parts' sums, compensated pairs
//   c = (sum c_l Tss, sum y_l Tsa),  s = (sum c_l Tas, sum y_l Taa),
// V = exp(i pi (a + b)) W, then the forward mode.  finish_vis returns the
// visibility's chi^2 term (twice that, but for FWD_DCHI); ym receives max
// |component| of the weighted residual.  Finish holds what they read besides the
// sums, loaded ahead of them.
//
// RES_STREAM: FP32 pairs.  The residual V - V° is an exact pair difference, and
// chi^2 per visibility needs only FP32 relative accuracy (the partials are summed
// in FP64).  The resident forms take residual, weight and chi^2 in FP64: any weight
// and residual that FP64 holds (sigma below 5e-20 overflows an FP32 weight).  A
// thread then waits out a chain of a dozen FP64 operations and five more per sum,
// so RES_BOTH has three finishing warps instead of two, and loads a job ahead: with
// two and without, 128 x 128 with 400,000 visibilities took 71 us, now 60.6, with
// FP32 pairs 57.4 (64 x 64 with 10,260: 10.9, 10.4, 9.9; CUDA events).
template <typename T>
struct Finish;

template <>
struct Finish<float> {
    uint64_t a, b;
    float4 o;  // V° as FP32 pairs (Re hi, Im hi, Re lo, Im lo)
    float2 y;  // FWD_DCHI: the base image's weighted residual
    float w;
};
template <>
struct Finish<double> {
    uint64_t a, b;
    double2 o;
    double w;
    float2 y;
};
template <typename T>
__device__ __forceinline__ Finish<T> finish_load(const DevData& d, int64_t j, int mode, const float2* yout) {
    Finish<T> f{};
    f.a = d.pa[j];
    f.b = d.pb[j];
    if (mode == FWD_DCHI) f.y = yout[j];
    if constexpr (sizeof(T) == 8) {
        if (mode != FWD_VIS) f.w = d.w[j];
        if (mode == FWD_RESID || mode == FWD_CHI) f.o = d.vo[j];
    } else {
        if (mode != FWD_VIS) f.w = d.w32[j];
        if (mode == FWD_RESID || mode == FWD_CHI) f.o = d.vo32[j];
    }
    return f;
}

// W turned to V = exp(i pi (a + b)) W, as pairs.
__device__ __forceinline__ void turn_sums(uint64_t a_, uint64_t b_, float4 c, float4 s, float2& vre, float2& vim) {
    const uint64_t half = (uint64_t)((int64_t)a_ >> 1) + (uint64_t)((int64_t)b_ >> 1);
    const cf2 e = cis_neg_accurate((uint32_t)((0 - half) >> 32));
    const float2 wre = df_add(c.x, c.y, -s.z, -s.w);  // c Tss - y Taa
    const float2 wim = df_add(c.z, c.w, s.x, s.y);    // y Tsa + c Tas
    auto prod = [](float c, float2 w) {  // c * (w.x + w.y) as a pair
        const float p = c * w.x;
        return make_float2(p, fmaf(c, w.y, fmaf(c, w.x, -p)));
    };
    const float2 a = prod(e.x, wre), b = prod(-e.y, wim), g = prod(e.x, wim), h = prod(e.y, wre);
    vre = df_add(a.x, a.y, b.x, b.y);
    vim = df_add(g.x, g.y, h.x, h.y);
}

// Only a valid visibility writes and counts; the arithmetic has no branch on it,
// so that two of a thread's visibilities share the FP64 units' latency.
__device__ __forceinline__ double finish_vis(const Finish<double>& f, int64_t j, bool valid, float4 c, float4 s,
                                             int mode, float2* yout, float& ym) {
    float2 vre, vim;
    turn_sums(f.a, f.b, c, s, vre, vim);
    if (mode == FWD_VIS) {
        if (valid) yout[j] = make_float2(vre.x + vre.y, vim.x + vim.y);
        return 0.0;
    }
    // V° is zero here in FWD_CURV and FWD_DCHI
    const double rr = ((double)vre.x - f.o.x) + (double)vre.y, ri = ((double)vim.x - f.o.y) + (double)vim.y;
    double chi;
    if (mode == FWD_DCHI) {
        const double h = 0.5 * f.w;
        chi = fma(fma(h, rr, (double)f.y.x), rr, fma(h, ri, (double)f.y.y) * ri);
    } else {
        const double yr = f.w * rr, yi = f.w * ri;
        chi = fma(yr, rr, yi * ri);
        if (mode == FWD_RESID && valid) {
            const float2 yv = make_float2((float)yr, (float)yi);
            yout[j] = yv;
            ym = fmaxf(fabsf(yv.x), fabsf(yv.y));
        }
    }
    return valid ? chi : 0.0;
}

__device__ __forceinline__ float finish_vis(const Finish<float>& f, int64_t j, bool valid, float4 c, float4 s,
                                            int mode, float2* yout, float& ym) {
    if (!valid) return 0.f;
    float2 vre, vim;
    turn_sums(f.a, f.b, c, s, vre, vim);
    if (mode == FWD_VIS) {
        yout[j] = make_float2(vre.x + vre.y, vim.x + vim.y);
        return 0.f;
    }
    if (mode == FWD_DCHI) {
        const float vr = vre.x + vre.y, vi = vim.x + vim.y;
        return f.y.x * vr + f.y.y * vi + 0.5f * f.w * (vr * vr + vi * vi);
    }
    // V° is zero here in FWD_CURV
    const float2 r0 = df_add(vre.x, vre.y, -f.o.x, -f.o.z);
    const float2 r1 = df_add(vim.x, vim.y, -f.o.y, -f.o.w);
    const float rr = r0.x + r0.y, ri = r1.x + r1.y;
    if (mode == FWD_RESID) {
        const float2 yv = make_float2(f.w * rr, f.w * ri);
        yout[j] = yv;
        ym = fmaxf(fabsf(yv.x), fabsf(yv.y));
    }
    return f.w * (rr * rr + ri * ri);
}

// Order-independent maximum (non-negative floats order as their bits).
__device__ __forceinline__ void finish_max(float ym, int mode, unsigned* ymax_bits, int lane) {
    if (mode != FWD_RESID || !ymax_bits) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ym = fmaxf(ym, __shfl_down_sync(0xffffffffu, ym, o));
    if (lane == 0) atomicMax(ymax_bits, __float_as_uint(ym));
}

// The tile partials of two groups of 32 visibilities, one of each per lane, summed
// later in a fixed order.  After the first step the warp's halves hold one group
// each, so that both take five additions together.  finish_vis leaves the factor
// 1/2 of FWD_RESID, FWD_CHI and FWD_CURV to the sum.
template <typename T>
__device__ __forceinline__ void finish_chi(T chi0, T chi1, int mode, double* chi_slots, int lane) {
    if (mode == FWD_VIS) return;
    const bool up = lane >= 16;
    const T other = __shfl_xor_sync(0xffffffffu, up ? chi0 : chi1, 16);
    T x = (up ? chi1 : chi0) + other;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o, 16);
    if ((lane & 15) == 0) chi_slots[lane >> 4] = mode == FWD_DCHI ? (double)x : 0.5 * (double)x;
}

// The operand's strips of MEAN_L columns l are scaled by powers of two, undone in
// the epilogue.
// STAGES: depth of the shared-memory pipeline (autotuned).
template <int STAGES, int RES>
__global__ void __launch_bounds__(FW_THREADS, 1)
    k_fwd_fold(DevData d, const VisTile* __restrict__ tiles, int n_tiles, const uint16_t* planes,
             const float4* cmean, int mode, float2* yout, double* __restrict__ chi_part, unsigned* __restrict__ ymax_bits,
             float4* __restrict__ vpart, int64_t z_total, uint64_t spin, int* status) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ F2Shared S;
    const int N = d.N;
    const int BN = RES == RES_STREAM ? d.fwd_bn : N;
    const int n_mb = N / BN, nk = N / (2 * TC_BK);
    // stages per accumulation and accumulations per (column block, part)
    const int kseg = nk < F2_KSEG / TC_BK ? nk : F2_KSEG / TC_BK;
    const int n_seg = nk / kseg;
    const int chunk_bytes = f2_chunk_bytes(BN);
    const int stage_bytes = f2_stage_bytes(BN, RES);
    unsigned char* ring = smem + f2_resident_bytes(N, RES);
    const uint32_t tcols = f2_tmem_cols(BN);
    const int64_t NN = (int64_t)N * N;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort = &S.abort;
    // Tiles of this CTA and the accumulations of a tile: (column block, K
    // segment, part), the part fastest; RES_PART: one part only.
    const int my_part = blockIdx.x & 1;  // RES_PART
    int t_begin, t_end, t_step;
    if (RES == RES_STREAM) {
        t_begin = blockIdx.x;
        t_end = n_tiles;
        t_step = gridDim.x;
    } else {
        // contiguous run of tiles per CTA: few channel changes, so few reloads
        const int g = RES == RES_PART ? blockIdx.x >> 1 : blockIdx.x;
        const int ng = RES == RES_PART ? gridDim.x >> 1 : gridDim.x;
        t_begin = (int)((int64_t)n_tiles * g / ng);
        t_end = (int)((int64_t)n_tiles * (g + 1) / ng);
        t_step = 1;
    }
    constexpr int n_part = RES == RES_PART ? 1 : 2;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&S.full[s], FW_PRODUCERS / 2 + (RES == RES_STREAM ? 1 : 0));
            mbar_init(&S.bfull[s], 1);
            mbar_init(&S.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&S.tfull[b], 1);
            mbar_init(&S.tempty[b], 4);
            mbar_init(&S.xfull[b], 8);
            mbar_init(&S.xempty[b], 2);
        }
        mbar_init(&S.bres, 1);
        mbar_init(&S.bfree, 1);
        mbar_init(&S.drain, 1);
        S.abort = 0;
        mbar_fence_init();
    }
    if (warp == 8) {
        tmem_alloc(&S.tmem_base, tcols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;
    chain_next();
    chain_wait();

    if (warp >= 8 && warp < 12) regs_dec<FW_REGS_MISC>();
    if (warp == 8) {
        // ---------------------------------------------------------------- MMA
        // The whole warp runs the issue loop, converged (every wait's outcome
        // is made warp-uniform), and one elected lane issues the MMAs and
        // commits.
        const uint32_t idesc = idesc_f16kind(128, BN, 0, 0, 0);
        const uint32_t abase = smem_u32(ring);
        const uint32_t bbase = RES == RES_STREAM ? abase + F2_ABYTES : smem_u32(smem);
        const uint32_t lboB = (uint32_t)(BN / 8) * 128;
        // Operand descriptors of slot 0; another slot, chunk or K step only
        // moves the start address, whose field (address >> 4, low 14 bits of
        // the low word) takes the offset by plain 32-bit addition (shared
        // memory < 256 KB, no carry).  A second K step is 2 core-matrix
        // columns on: 2 x 2048 bytes in A, 2 x lboB in B.
        const uint64_t d_ah = smem_desc(abase, 2048, 128);
        const uint64_t d_al = smem_desc(abase + F2_APLANE, 2048, 128);
        const uint64_t d_bh = smem_desc(bbase, lboB, 128);
        const uint64_t d_bl = smem_desc(bbase + BN * TC_BK * 2, lboB, 128);
        const uint32_t lo_ah = (uint32_t)d_ah, lo_al = (uint32_t)d_al;
        const uint32_t lo_bh = (uint32_t)d_bh, lo_bl = (uint32_t)d_bl;
        const uint32_t hi_a = (uint32_t)(d_ah >> 32), hi_b = (uint32_t)(d_bh >> 32);
        const uint32_t ka16 = (2u * 2048u) >> 4, kb16 = (2u * lboB) >> 4;
        static_assert(TC_BK == 32, "one stage is two K steps of 16");
        uint32_t sc = 0, it = 0, nres = 0;
        int cur_chan = -1;
        bool ok = true;
        for (int t = t_begin; t < t_end && ok; t += t_step) {
            if (RES != RES_STREAM) {
                const int chan = tiles[t].chan;
                if (chan != cur_chan) {
                    if (nres > 0) {
                        // every MMA that read the previous channel's operand has completed
                        umma_commit_elect(&S.bfree);
                        ok = __all_sync(~0u, mbar_wait(&S.bfree, (nres - 1) & 1, spin, abort, status));
                        if (!ok) break;
                    }
                    if (lane == 0) {
                        const int n_chunks = RES == RES_BOTH ? 2 * nk : nk;
                        const unsigned char* src = (const unsigned char*)(planes + (int64_t)chan * 2 * NN) +
                                                   (RES == RES_PART ? (int64_t)my_part * nk * chunk_bytes : 0);
                        mbar_arrive_expect_tx(&S.bres, (uint32_t)(n_chunks * chunk_bytes));
                        for (int q = 0; q < n_chunks; ++q)
                            bulk_g2s(smem + (size_t)q * chunk_bytes, src + (size_t)q * chunk_bytes,
                                     (uint32_t)chunk_bytes, &S.bres);
                    }
                    __syncwarp();
                    ok = __all_sync(~0u, mbar_poll(&S.bres, nres & 1, spin, abort, status));
                    ++nres;
                    if (!ok) break;
                    cur_chan = chan;
                }
            }
            for (int mb = 0, ks0 = 0, part = 0; mb < n_mb && ok; ++it) {
                const int b = it & 1;
                ok = __all_sync(~0u, mbar_wait(&S.tempty[b], ((it >> 1) & 1) ^ 1, spin, abort, status));
                if (!ok) break;
                tc_fence_after();
                const uint32_t dt = tmem + (uint32_t)(b * BN);
                for (int ks = ks0; ks < ks0 + kseg; ++ks, ++sc) {
                    const int s = sc % STAGES;
                    // one wait: the producers' tables and the streamed chunk
                    ok = __all_sync(~0u, mbar_wait(&S.full[s], (sc / STAGES) & 1, spin, abort, status));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t so = (uint32_t)(s * stage_bytes) >> 4;
                    const uint32_t bo = RES == RES_STREAM ? so : (uint32_t)((part * nk + ks) * chunk_bytes) >> 4;
                    if (RES == RES_BOTH) {
                        umma_corrections_elect(dt, lo_ah + so, lo_al + so, lo_bh + bo, lo_bl + bo, hi_a, hi_b, ka16,
                                               kb16, idesc, ks > ks0 ? 1u : 0u);
                    } else {
                        umma6_fold_elect(dt, lo_ah + so, lo_al + so, lo_bh + bo, lo_bl + bo, hi_a, hi_b, ka16, kb16,
                                          idesc, ks > ks0 ? 1u : 0u);
                        umma_commit_elect(&S.empty[s]);
                    }
                }
                if (!ok) break;
                if (RES == RES_BOTH) {
                    // the main products, over the accumulation's (at most two) stages
                    for (int ks = ks0; ks < ks0 + kseg; ++ks) {
                        const uint32_t q = sc - (uint32_t)(ks0 + kseg - ks);
                        const uint32_t so = (uint32_t)((q % STAGES) * stage_bytes) >> 4;
                        const uint32_t bo = (uint32_t)((part * nk + ks) * chunk_bytes) >> 4;
                        umma_main_elect(dt, lo_ah + so, lo_bh + bo, hi_a, hi_b, ka16, kb16, idesc);
                        umma_commit_elect(&S.empty[q % STAGES]);
                    }
                }
                umma_commit_elect(&S.tfull[b]);
                if (++part == n_part) {
                    part = 0;
                    ks0 += kseg;
                    if (ks0 == nk) {
                        ks0 = 0;
                        ++mb;
                    }
                }
            }
        }
        // every issued MMA completes before TMEM is released, and every
        // resident-operand copy lands before shared memory is released
        umma_commit_elect(&S.drain);
        int dummy = 0;
        mbar_wait(&S.drain, 0, drain_limit(spin), (volatile int*)&dummy, status);
        if (!ok && nres > 0) mbar_wait(&S.bres, (nres - 1) & 1, drain_limit(spin), (volatile int*)&dummy, status);
        __syncwarp();
    } else if (warp == 9 && RES != RES_BOTH) {
        // --------------------------------------------- streamed operand copies
        if (RES == RES_STREAM && lane == 0) {
            uint32_t sc = 0;
            bool ok = true;
            // once stage q's chunk has landed (bfull), the copy warp is the
            // last arrival on full[q]; it does so one stage behind the copy it
            // issues, so that a copy is always in flight
            auto land = [&](uint32_t q) -> bool {
                if (!mbar_wait(&S.bfull[q % STAGES], (q / STAGES) & 1, spin, abort, status)) return false;
                mbar_arrive(&S.full[q % STAGES]);
                return true;
            };
            for (int t = t_begin; t < t_end && ok; t += t_step) {
                const int chan = tiles[t].chan;
                const unsigned char* cbase = (const unsigned char*)(planes + (int64_t)chan * 2 * NN);
                for (int mb = 0, ks0 = 0, part = 0; mb < n_mb && ok;) {
                    const unsigned char* src = cbase + (int64_t)((2 * mb + part) * nk + ks0) * chunk_bytes;
                    for (int k = 0; k < kseg; ++k, ++sc, src += chunk_bytes) {
                        const int s = sc % STAGES;
                        ok = mbar_wait(&S.empty[s], ((sc / STAGES) & 1) ^ 1, spin, abort, status);
                        if (!ok) break;
                        mbar_arrive_expect_tx(&S.bfull[s], (uint32_t)chunk_bytes);
                        bulk_g2s(ring + s * stage_bytes + F2_ABYTES, src, (uint32_t)chunk_bytes, &S.bfull[s]);
                        if (sc > 0) {
                            ok = land(sc - 1);
                            if (!ok) {
                                ++sc;  // the copy just issued is in flight too
                                break;
                            }
                        }
                    }
                    if (++part == 2) {
                        part = 0;
                        ks0 += kseg;
                        if (ks0 == nk) {
                            ks0 = 0;
                            ++mb;
                        }
                    }
                }
            }
            if (ok && sc > 0) ok = land(sc - 1);
            if (!ok) {
                // copies already issued land on their own; wait for them before
                // the CTA's shared memory is released
                int dummy = 0;
                for (uint32_t q = (sc > STAGES ? sc - STAGES : 0); q < sc; ++q)
                    mbar_wait(&S.bfull[q % STAGES], (q / STAGES) & 1, drain_limit(spin), (volatile int*)&dummy,
                              status);
            }
        }
        __syncwarp();
    } else if (warp < 12 && warp >= 9) {
        // ------------------------------------------------- finishing warps
        // A job is half a tile, two visibilities per thread; the finishing warps
        // (10 and 11, with RES_BOTH 9 too) take them in turn.
        if (RES != RES_PART) {
            using T = std::conditional_t<RES == RES_STREAM, float, double>;
            constexpr int N_FIN = RES == RES_BOTH ? 3 : 2;
            constexpr bool AHEAD = RES == RES_BOTH;
            const float4* xsum = (const float4*)(ring + STAGES * stage_bytes);
            const int jobs = t_begin < t_end ? 2 * ((t_end - t_begin + t_step - 1) / t_step) : 0;
            auto tile_of = [&](int job) { return tiles[t_begin + (job >> 1) * t_step]; };
            auto load = [&](const VisTile& tl, int job, Finish<T>(&f)[2]) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int jv = 64 * (job & 1) + 32 * h + lane;
                    f[h] = finish_load<T>(d, tl.start + (jv < tl.count ? jv : 0), mode, yout);
                }
            };
            // AHEAD: a job's inputs arrive while the one before it is finished, its
            // tile's descriptor another job ahead
            const int job0 = warp - (12 - N_FIN);
            VisTile tl_next = {}, tl_after = {};
            Finish<T> next[2];
            if (AHEAD && job0 < jobs) {
                tl_next = tile_of(job0);
                if (job0 + N_FIN < jobs) tl_after = tile_of(job0 + N_FIN);
                load(tl_next, job0, next);
            }
            bool ok = true;
            for (int job = job0; job < jobs && ok; job += N_FIN) {
                const uint32_t ti = (uint32_t)job >> 1;
                VisTile tl;
                Finish<T> in[2];
                if (AHEAD) {
                    tl = tl_next;
                    in[0] = next[0];
                    in[1] = next[1];
                    if (job + N_FIN < jobs) {
                        tl_next = tl_after;
                        if (job + 2 * N_FIN < jobs) tl_after = tile_of(job + 2 * N_FIN);
                        load(tl_next, job + N_FIN, next);
                    }
                } else {
                    tl = tile_of(job);
                    load(tl, job, in);
                }
                ok = __all_sync(0xffffffffu, mbar_wait(&S.xfull[ti & 1], (ti >> 1) & 1, spin, abort, status, 250));
                if (!ok) break;
                const float4* slot = xsum + (ti & 1) * 256;
                T chi[2];
                float ym[2] = {0.f, 0.f};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int jv = 64 * (job & 1) + 32 * h + lane;
                    chi[h] = finish_vis(in[h], tl.start + jv, jv < tl.count, slot[jv], slot[128 + jv], mode, yout,
                                        ym[h]);
                }
                finish_max(fmaxf(ym[0], ym[1]), mode, ymax_bits, lane);
                finish_chi(chi[0], chi[1], mode, chi_part + ((int64_t)(t_begin + (int)ti * t_step) * 2 + (job & 1)) * 2,
                           lane);
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.xempty[ti & 1]);
            }
        }
    } else if (warp >= 12) {
        // ------------------------------------------------- table producers
        // Two groups of four warps build alternate stages: a stage's latencies
        // (slot wait, stores, proxy fence) then overlap the other group's.
        // thread -> visibility jv = A row: 32 entries c_j (cosine part) or y_j
        // (sine part), as four groups of 8 rows.  A warp's 16-byte stores fill
        // whole 128-byte core matrices, four wavefronts each.
        regs_dec<FW_REGS_PROD>();
        const int ptid = threadIdx.x - 384;
        const int jv = ptid & 127;
        const uint32_t grp = ptid >> 7;
        const int off = (jv >> 3) * 128 + (jv & 7) * 16;
        uint32_t sc = 0;
        bool ok = true;
        // the next tile's descriptor and phases arrive while this one is built
        uint64_t pb_next = 0;
        auto load_tile = [&](int t) {
            const VisTile tl = tiles[t];
            // rows beyond the tile's count repeat its first visibility; the
            // epilogue does not read them
            pb_next = d.pb[tl.start + (jv < tl.count ? jv : 0)];
        };
        if (t_begin < t_end) load_tile(t_begin);
        for (int t = t_begin; t < t_end && ok; t += t_step) {
            const uint64_t pb = pb_next;
            if (t + t_step < t_end) load_tile(t + t_step);
            const HalfSteps hs = half_steps(pb);
            const HalfPairs w = half_pairs(hs);
            const cf2 step8 = hs.s8;
            const cf2 step64 = cis_neg_accurate((uint32_t)((2 * TC_BK * pb) >> 32));  // over two stages
            for (int mb = 0, ks0 = 0, part = RES == RES_PART ? my_part : 0; mb < n_mb && ok;) {
                // Phase factor x + i y at the centre of the first 8 rows of this
                // group's first stage of the accumulation (row j0 + 3.5, so
                // (j + 1/2) b = (j0 + 4) b there), held as (x, q) with q = y in the sine part and
                // -y in the cosine part (products of conjugates), so that
                //   Re(base w) = x Re w + q Im w,  Im(base w) = q Re w + x Im w.
                const int k0 = (int)((sc ^ grp) & 1);
                cf2 base0 = cis_neg_accurate(phase_hi((ks0 + k0) * TC_BK + 4, pb));
                const float sgn = part ? 1.f : -1.f;
                base0.y *= sgn;
                const cf2 s64 = {step64.x, step64.y * sgn};
                const float2 s8x = make_float2(step8.x, step8.x), s8q = make_float2(step8.y * sgn, step8.y * sgn);
                const float2 s8n = make_float2(-s8q.x, -s8q.x);
                for (int k = k0; k < kseg; k += 2) {
                    const uint32_t q = sc + k;
                    const int s = q % STAGES;
                    ok = __all_sync(0xffffffffu,
                                    mbar_wait(&S.empty[s], ((q / STAGES) & 1) ^ 1, spin, abort, status, 32));
                    if (!ok) break;
                    unsigned char* A = ring + s * stage_bytes + off;
                    float2 x = make_float2(base0.x, base0.x), y = make_float2(base0.y, base0.y);
                    auto build = [&](bool sine) {
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            uint4 h, l;
                            table8_real(sine ? y : x, sine ? x : y, w, h, l);
                            *(uint4*)(A + g * 2048) = h;
                            *(uint4*)(A + F2_APLANE + g * 2048) = l;
                            if (g < 3) {  // the next 8 rows' factor
                                const float2 x1 = __ffma2_rn(x, s8x, __fmul2_rn(y, s8n));
                                y = __ffma2_rn(x, s8q, __fmul2_rn(y, s8x));
                                x = x1;
                            }
                        }
                    };
                    if (part) build(true);
                    else build(false);
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&S.full[s]);
                    base0 = cmul(base0, s64);
                }
                sc += kseg;
                if (RES != RES_PART && part == 0) {
                    part = 1;
                } else {
                    if (RES != RES_PART) part = 0;
                    ks0 += kseg;
                    if (ks0 == nk) {
                        ks0 = 0;
                        ++mb;
                    }
                }
            }
        }
    } else if (warp < 8) {
        // ------------------------ epilogue (two groups of four warps)
        // TMEM lane = visibility: warp q of a group holds visibilities
        // 32q .. 32q+31.  Group 0 drains accumulator 0 (the cosine part),
        // group 1 accumulator 1 (the sine part); with RES_PART both hold the
        // CTA's part and the groups alternate tiles.  Each lane forms
        //   s0 = sum_l c_l P_l,  s1 = sum_l y_l Q_l.
        regs_inc<FW_REGS_EPI>();
        const int grp = warp >> 2, quad = warp & 3;
        const int jv = 32 * quad + lane;
        const int part = RES == RES_PART ? my_part : grp;
        float4* xsum = (float4*)(ring + STAGES * stage_bytes);
        uint32_t it = 0;  // accumulations of this group
        bool ok = true;
        const int e_begin = RES == RES_PART ? t_begin + grp : t_begin, e_step = RES == RES_PART ? 2 : t_step;
        uint32_t ti = 0;  // tiles of this group
        // the next tile's descriptor and phases arrive while this tile's
        // accumulators drain
        VisTile tl_next = {};
        uint64_t pa_next = 0, pb_next = 0;
        auto load_tile = [&](int t) {
            tl_next = tiles[t];
            const int64_t jn = tl_next.start + (jv < tl_next.count ? jv : 0);
            pa_next = d.pa[jn];
            pb_next = d.pb[jn];
        };
        if (e_begin < t_end) load_tile(e_begin);
        for (int t = e_begin; t < t_end && ok; t += e_step, ++ti) {
            const VisTile tl = tl_next;
            const uint64_t pb = pb_next;
            const uint64_t pa = pa_next, ha = (uint64_t)((int64_t)pa >> 1);
            if (t + e_step < t_end) load_tile(t + e_step);
            cf2 step8;  // chunk to chunk (recurrence below)
            const Rot8 wx8 = rot8_steps(pa, step8);
            const cf2 step32 = cis_neg_accurate((uint32_t)((32 * pa) >> 32));  // over PHASE_REFRESH chunks
            // the part's table sum over all rows (accurate sinpi of the exact
            // half-turn and N/2-multiple phases, which keep small angles'
            // relative accuracy)
            float scomp;
            {
                const float th = (float)((int64_t)pb >> 1) * 5.421010862427522e-20f;             // b/2, turns
                const float tn = (float)(int64_t)phase_mul(N / 2, pb) * 5.421010862427522e-20f;  // N b/2
                const float sh = sinpif(2.0f * th);             // sin(pi b)
                const float sn = sinpif(part ? tn : 2.0f * tn);  // sin(pi N b / 2) up to its sign, or sin(pi N b)
                if (part == 0) scomp = (sh != 0.f) ? 0.5f * sn / sh : 0.5f * (float)N;
                else scomp = (sh != 0.f) ? -sn * sn / sh : 0.f;
            }
            // (P mean, Q mean, 1 / scale) per strip of MEAN_L folded columns, and
            // the sum of the step factors over them times S
            const float4* cm_part = cmean + ((int64_t)tl.chan * 2 + part) * (N / 2 / MEAN_L);
            cf2 wsum;
            {
                const float2 x = __fadd2_rn(__fadd2_rn(wx8.x[0], wx8.x[1]), __fadd2_rn(wx8.x[2], wx8.x[3]));
                const float2 y = __fadd2_rn(__fadd2_rn(wx8.y[0], wx8.y[1]), __fadd2_rn(wx8.y[2], wx8.y[3]));
                const cf2 w8 = {x.x + x.y, y.x + y.y}, w16 = cmul(w8, step8);
                wsum = {(w8.x + w16.x) * scomp, (w8.y + w16.y) * scomp};
                static_assert(MEAN_L == 16, "two chunks share their means");
            }
            float s0 = 0.f, s1 = 0.f, c0s = 0.f, c1s = 0.f;  // compensated sums
            const int b = grp;
            const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * BN);
            for (int mb = 0; mb < n_mb && ok; ++mb) {
                // the phase factor exp(-2 pi i (l0 + 1/2) a) of the block's first l
                const cf2 base_mb = cis_neg_accurate(phase_hi(mb * BN + 1, ha));
                for (int seg = 0; seg < n_seg; ++seg, ++it) {
                    // Lane i holds the i-th strip's means and inverse scale; the
                    // mean's term cm S enters once per column: with the block's
                    // first segment only.
                    float4 cm = {0.f, 0.f, 0.f, 0.f};
                    if (lane < BN / (2 * MEAN_L)) cm = cm_part[mb * (BN / (2 * MEAN_L)) + lane];
                    if (seg != 0) cm.x = cm.y = 0.f;
                    ok = __all_sync(0xffffffffu, mbar_wait(&S.tfull[b], it & 1, spin, abort, status, 32));
                    if (!ok) break;
                    tc_fence_after();
                    // software pipeline over 16-column chunks: the TMEM load of
                    // chunk q+1 is in flight while chunk q is reduced
                    const int nq = BN / 16;
                    uint32_t tv[2][16];
                    auto load_chunk = [&](int q, int slot) { tmem_ld16(lane_base + q * 16, tv[slot]); };
                    // adds the chunk's sum_l c_l P_l and sum_l y_l Q_l to x0 and x1:
                    // c_l + i y_l = base * step_k; packed over even and odd k
                    auto reduce_chunk = [&](const cf2 base, int slot, float& x0, float& x1) {
                        float2 uc, us, wc, ws;
#pragma unroll
                        for (int p = 0; p < 4; ++p) {
                            const float2 tp = make_float2(__uint_as_float(tv[slot][2 * p]),
                                                          __uint_as_float(tv[slot][2 * p + 1]));
                            const float2 tq = make_float2(__uint_as_float(tv[slot][2 * p + 8]),
                                                          __uint_as_float(tv[slot][2 * p + 9]));
                            uc = p ? __ffma2_rn(wx8.x[p], tp, uc) : __fmul2_rn(wx8.x[0], tp);
                            us = p ? __ffma2_rn(wx8.y[p], tp, us) : __fmul2_rn(wx8.y[0], tp);
                            wc = p ? __ffma2_rn(wx8.x[p], tq, wc) : __fmul2_rn(wx8.x[0], tq);
                            ws = p ? __ffma2_rn(wx8.y[p], tq, ws) : __fmul2_rn(wx8.y[0], tq);
                        }
                        const float vuc = uc.x + uc.y, vus = us.x + us.y, vwc = wc.x + wc.y, vws = ws.x + ws.y;
                        x0 = fmaf(base.x, vuc, fmaf(-base.y, vus, x0));
                        x1 = fmaf(base.x, vws, fmaf(base.y, vwc, x1));
                    };
                    // two chunks (32 columns) from q on: slot 0 is loaded, slot 1
                    // and the next slot 0 load on the way
                    float x0 = 0.f, x1 = 0.f;
                    auto pair = [&](int q, cf2& base) {
                        load_chunk(q + 1, 1);
                        // the two chunks' means: sum_l (c_l + i y_l) S = base * wsum
                        const cf2 bw = cmul(base, wsum);
                        x0 = fmaf(__shfl_sync(0xffffffffu, cm.x, q / 2), bw.x, x0);
                        x1 = fmaf(__shfl_sync(0xffffffffu, cm.y, q / 2), bw.y, x1);
                        // (a power of two: exact)
                        const float inv = __shfl_sync(0xffffffffu, cm.z, q / 2);
                        cf2 bs = {base.x * inv, base.y * inv};
                        reduce_chunk(bs, 0, x0, x1);
                        tmem_ld_wait(tv[1]);
                        load_chunk(q + 2 < nq ? q + 2 : 0, 0);  // (the last one is not used)
                        base = cmul(base, step8);
                        bs = {base.x * inv, base.y * inv};
                        reduce_chunk(bs, 1, x0, x1);
                        tmem_ld_wait(tv[0]);
                    };
                    // chunk phase factors: step8 from chunk to chunk, step32 over
                    // PHASE_REFRESH chunks, so that few roundings add up
                    cf2 base4 = base_mb;
                    load_chunk(0, 0);
                    tmem_ld_wait(tv[0]);
                    for (int q = 0; q < nq; q += PHASE_REFRESH) {  // 64 columns
                        cf2 base = base4;
                        pair(q, base);
                        if (q + 2 < nq) {
                            base = cmul(base, step8);
                            pair(q + 2, base);
                        }
                        base4 = cmul(base4, step32);
                        two_sum_acc(s0, c0s, x0);
                        two_sum_acc(s1, c1s, x1);
                        x0 = x1 = 0.f;
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&S.tempty[b]);
                }
            }
            if (!ok) break;
            const float4 sums = make_float4(s0, c0s, s1, c1s);
            if (RES == RES_PART) {
                if (jv < tl.count) vpart[(int64_t)part * z_total + tl.start + jv] = sums;
                continue;
            }
            // hand the part's sums to the finishing warps
            ok = __all_sync(0xffffffffu,
                            mbar_wait(&S.xempty[ti & 1], ((ti >> 1) & 1) ^ 1, spin, abort, status, 32));
            if (!ok) break;
            xsum[(ti & 1) * 256 + part * 128 + jv] = sums;
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.xfull[ti & 1]);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 8) {
        tc_fence_after();
        tmem_dealloc(tmem, tcols);
    }
}

// RES_PART: one block of 64 threads per tile adds the two parts' sums and
// applies the mode.
__global__ void __launch_bounds__(64) k_fold_combine(DevData d, const VisTile* __restrict__ tiles,
                                                     const float4* vpart, int64_t z_total, int mode,
                                                     float2* yout, double* chi_part, unsigned* ymax_bits) {
    chain_next();
    chain_wait();
    const VisTile tl = tiles[blockIdx.x];
    // two visibilities per thread, one of each half of the tile's groups
    double chi[2];
    float ym[2] = {0.f, 0.f};
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int jv = 32 * (2 * warp + h) + lane;
        const int64_t j = tl.start + (jv < tl.count ? jv : 0);
        chi[h] = finish_vis(finish_load<double>(d, j, mode, yout), j, jv < tl.count, vpart[j], vpart[z_total + j], mode,
                            yout, ym[h]);
    }
    finish_max(fmaxf(ym[0], ym[1]), mode, ymax_bits, lane);
    finish_chi(chi[0], chi[1], mode, chi_part + (int64_t)blockIdx.x * 4 + 2 * warp, lane);
}

struct FwdArgs {
    DevData d;
    const VisTile* tiles;
    int n_tiles;
    const uint16_t* planes;
    const float4* cmean;
    int mode;
    float2* yout;
    double* chi_part;
    unsigned* ymax_bits;
    float4* vpart;
    int64_t z_total;
    uint64_t spin;
    int* status;
    cudaStream_t st;
};

template <int STAGES, int RES>
void launch_variant(const FwdArgs& a, int grid) {
    const int smem = f2_smem_bytes(a.d.N, a.d.fwd_bn, STAGES, RES);
    // the register split waits for registers that only a launch with FW_REGS holds
    static const bool regs_ok = [] {
        cudaFuncAttributes at;
        return cudaFuncGetAttributes(&at, k_fwd_fold<STAGES, RES>) == cudaSuccess && at.numRegs == FW_REGS;
    }();
    if (!regs_ok) {  // a launch with no threads leaves an error for the caller's check
        k_fwd_fold<STAGES, RES><<<grid, 0, 0, a.st>>>(a.d, a.tiles, a.n_tiles, a.planes, a.cmean, a.mode,
                                                        a.yout, a.chi_part, a.ymax_bits, a.vpart, a.z_total, a.spin,
                                                        a.status);
        return;
    }
    cudaFuncSetAttribute(k_fwd_fold<STAGES, RES>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    launch_chained(k_fwd_fold<STAGES, RES>, dim3(grid), FW_THREADS, smem, a.st, a.d.chain, 1, a.d, a.tiles, a.n_tiles,
                   a.planes, a.cmean, a.mode, a.yout, a.chi_part, a.ymax_bits, a.vpart, a.z_total, a.spin, a.status);
}

void launch_stages(const FwdArgs& a, int res, int grid) {
    const int st = a.d.fwd_stages;
    if (res == RES_STREAM) {
        if (st == 3) launch_variant<3, RES_STREAM>(a, grid);
        else launch_variant<4, RES_STREAM>(a, grid);
    } else if (res == RES_BOTH) {
        if (st <= 4) launch_variant<4, RES_BOTH>(a, grid);
        else if (st == 5) launch_variant<5, RES_BOTH>(a, grid);
        else launch_variant<6, RES_BOTH>(a, grid);
    } else {
        if (st <= 4) launch_variant<4, RES_PART>(a, grid);
        else if (st == 5) launch_variant<5, RES_PART>(a, grid);
        else launch_variant<6, RES_PART>(a, grid);
    }
}

int resident_kind(int N) { return N <= 128 ? RES_BOTH : RES_PART; }

}  // namespace

int fold_smem_bytes(int N, int BN, int stages, int resident) {
    return f2_smem_bytes(N, BN, stages, resident ? resident_kind(N) : RES_STREAM);
}

bool fold_combines(int N) { return resident_kind(N) == RES_PART; }

int launch_fwd_fold(const DevData& d, int resident, const VisTile* tiles, int n_tiles, const void* planes,
                    const float4* cmean, int mode, float2* yout, double* chi_part, float* ymax,
                  float4* vpart, int64_t z_total, int num_sms, uint64_t spin, int* status, cudaStream_t st) {
    if (n_tiles <= 0) return 0;
    const FwdArgs a{d,      tiles,   n_tiles,         (const uint16_t*)planes, cmean, mode, yout,
                    chi_part, (unsigned*)ymax, vpart, z_total, spin, status, st};
    const int res = resident ? resident_kind(d.N) : RES_STREAM;
    // one CTA per SM, at most one per tile (RES_PART: a pair of CTAs per tile)
    const int grid = res == RES_PART ? 2 * std::max(1, std::min(num_sms / 2, n_tiles)) : std::min(num_sms, n_tiles);
    launch_stages(a, res, grid);
    if (res != RES_PART) return 1;
    launch_chained(k_fold_combine, dim3(n_tiles), 64, 0, st, d.chain, 1, d, tiles, (const float4*)vpart, z_total, mode, yout,
                   chi_part, (unsigned*)ymax);
    return 2;
}

}  // namespace msk
