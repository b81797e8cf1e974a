// Tensor-core forward operator of the BF16X3 form (Eq. 1 on the pixel grid) for
// images of side N <= 256, with the image operand resident in shared memory.
//
//   T_s = Ey[:, rows of slice s] B'[rows of slice s, :]^T   (tcgen05.mma kind::f16)
//   V_k = sum_s sum_m Ex[k,m] T_s[k,m]  (+ c_m S_k from slice 0)
//
// The image rows (the contraction index n) are cut into slices of at most
// 128 rows.  A persistent CTA owns one slice: it copies that slice of the
// split operand planes (hi and lo, N columns, 128 KB at N = 256) into shared
// memory once per channel and keeps it, so only the phase-table operand Ey
// streams through the pipeline.  Re-streaming the whole image operand for
// every 64-visibility tile is what bounds the streaming kernel (about 5 TB/s
// of L2 traffic at N = 256).  Each of several slices writes a partial
// visibility per sample (FP64); k_fwd_combine adds the slices in a fixed order and
// applies the residual, weight and chi^2 partials.  The one slice of N <= 128
// hands its sums to two finishing warps instead.
//
// Accumulation order.  The tensor core adds each MMA's exact product sum to
// the FP32 accumulator rounding towards zero, so every MMA of an output can
// shrink it by up to one ulp.  The correction products (hi*lo, lo*hi, about
// 2^-11 of the result for the FP16 split, 2^-8 for BF16) are issued first
// over the whole slice, while the accumulator is still small; the hi*hi
// products follow.  Of the 3 KS/16 MMAs per output only the KS/16 hi*hi ones
// then act on an accumulator of full magnitude.  A slice is at most four stages,
// which stay in the ring for both (tables built a second time for the hi*hi
// products were a third of the kernel's time).
//
// Tile: 64 visibilities, A rows 32 (j >> 4) + (j & 15) (Re Ey) and 16 below
// (Im Ey), as in the streaming kernel.  Roles (seven warpgroups): warps 0-3 and 4-7
// epilogue (TMEM lane = A row; a group per accumulator, so alternate tiles), warp
// 8 MMA issuer, TMEM owner and resident-operand loader, warps 12-27 Ey producers.
// Every wait is bounded.
//
// What bounds it: the SIMT instructions of the table and of the drain, not the
// MMAs (128 x 128: 1,536 clocks a tile).  Sixteen producer warps and the register
// split instead of eight without: 125 -> 121 us at 128 x 128 with 400,000
// visibilities; the finishing warps instead of k_fwd_combine: 121 -> 107 us.
// Altogether 63 -> 35 us with 100,003 visibilities (one epilogue group, the tables
// built twice before; CUDA events around the launches), the same bits.
#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "internal.h"

namespace msk {

namespace {

constexpr int RS_PRODUCERS = 16;  // producer warps: two groups of eight, alternate stages
constexpr int RS_THREADS = 32 * (12 + RS_PRODUCERS);
// registers per thread: at launch, epilogue, producers, the MMA warp's warpgroup
constexpr int RS_REGS = 72, RS_REGS_EPI = 104, RS_REGS_PROD = 64, RS_REGS_MISC = 40;
static_assert(8 * RS_REGS_EPI + RS_PRODUCERS * RS_REGS_PROD + 4 * RS_REGS_MISC <= (12 + RS_PRODUCERS) * RS_REGS,
              "the shares add up to the registers at launch");
constexpr int RS_MAX_STAGES = 6;
constexpr int RS_APLANE = 128 * TC_BK * 2;  // one A plane of a stage (hi or lo), 8 KB
constexpr int RS_ABYTES = 2 * RS_APLANE;


__host__ __device__ inline uint32_t rs_tmem_cols(int N) {
    uint32_t c = 32;
    while ((int)c < 2 * N) c <<= 1;
    return c;
}

struct RsShared {
    uint64_t full[RS_MAX_STAGES];   // the 8 producer warps of a group
    uint64_t empty[RS_MAX_STAGES];  // MMA completion (tcgen05.commit)
    uint64_t bres;                  // resident operand copy (transaction bytes)
    uint64_t bfree;                 // MMAs reading the resident operand done
    uint64_t tfull[2];
    uint64_t tempty[2];  // 4 epilogue warps
    uint64_t xfull[2];   // V of a tile (4 epilogue warps)
    uint64_t xempty[2];  // read by the two finishing warps
    uint64_t drain;
    uint32_t tmem_base;
    int abort;
};

// What a visibility's last steps read besides V, loaded ahead of it.
struct RsFinishIn {
    double2 vo;
    double w;
    float2 y;  // FWD_DCHI: the base image's weighted residual
};
__device__ __forceinline__ RsFinishIn rs_finish_load(const DevData& d, int64_t j, int mode, const float2* yout) {
    RsFinishIn f;
    f.vo = make_double2(0.0, 0.0);
    f.w = 0.0;
    f.y = make_float2(0.f, 0.f);
    if (mode != FWD_VIS) f.w = d.w[j];
    if (mode == FWD_DCHI) f.y = yout[j];
    if (mode == FWD_RESID || mode == FWD_CHI) f.vo = d.vo[j];
    return f;
}

// The forward mode applied to one visibility (model visibilities, weighted
// residual, chi^2, curvature or line-search difference); its chi^2 term.
__device__ __forceinline__ double rs_finish_vis(const RsFinishIn& f, int64_t j, double Vre, double Vim, int mode,
                                                float2* yout) {
    if (mode == FWD_VIS) {
        yout[j] = make_float2((float)Vre, (float)Vim);
        return 0.0;
    }
    if (mode == FWD_DCHI)
        return (double)f.y.x * Vre + (double)f.y.y * Vim + 0.5 * f.w * (Vre * Vre + Vim * Vim);
    // V° is zero here in FWD_CURV
    const double rr = Vre - f.vo.x, ri = Vim - f.vo.y;
    if (mode == FWD_RESID) yout[j] = make_float2((float)(f.w * rr), (float)(f.w * ri));
    return 0.5 * f.w * (rr * rr + ri * ri);
}

// One chi^2 partial per 16 visibilities, the layout the scalar reduction reads
// (4 per tile).
__device__ __forceinline__ void rs_finish_chi(double chi, int mode, int jv, double* chi_tile) {
    if (mode == FWD_VIS) return;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) chi += __shfl_down_sync(0xffffffffu, chi, o, 16);
    if ((jv & 15) == 0) chi_tile[jv >> 4] = chi;
}

template <int STAGES>
__global__ void __launch_bounds__(RS_THREADS, 1)
    k_fwd_rs(DevData d, const VisTile* __restrict__ tiles, int n_tiles, const uint16_t* planes,
             const float* cmean, double2* __restrict__ vpart,
             int64_t z_total, int mode, float2* yout, double* __restrict__ chi_part, uint64_t spin,
             int* status) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ RsShared S;
    const int N = d.N, c0 = N / 2;
    const int KS = fwd_rs_ks(N), n_slices = N / KS, nks = KS / TC_BK;
    const int slice = blockIdx.x % n_slices;
    const int group = blockIdx.x / n_slices, n_groups = gridDim.x / n_slices;
    // contiguous run of tiles per CTA: few channel changes, so few reloads
    const int t_begin = (int)((int64_t)n_tiles * group / n_groups);
    const int t_end = (int)((int64_t)n_tiles * (group + 1) / n_groups);
    const uint32_t chunk_bytes = 2u * N * TC_BK * 2;  // one 32-row chunk, hi + lo planes
    unsigned char* sB = smem;                         // resident slice: nks chunks
    unsigned char* sA = smem + (size_t)nks * chunk_bytes;
    double2* xsum = (double2*)(sA + STAGES * RS_ABYTES);  // one slice: V of two tiles, 64 each
    const uint32_t tcols = rs_tmem_cols(N);
    const int64_t NN = (int64_t)N * N;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort = &S.abort;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&S.full[s], RS_PRODUCERS / 2);
            mbar_init(&S.empty[s], 1);
        }
        mbar_init(&S.bres, 1);
        mbar_init(&S.bfree, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&S.tfull[b], 1);
            mbar_init(&S.tempty[b], 4);
            mbar_init(&S.xfull[b], 4);
            mbar_init(&S.xempty[b], 2);
        }
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

    if (warp >= 8 && warp < 12) regs_dec<RS_REGS_MISC>();
    if (warp == 8) {
        // ------------------------------------------ MMA + resident operand
        // (the whole warp runs the loop, converged; an elected lane issues)
        {
            const uint32_t idesc = idesc_f16kind(128, N, 0, 0, 1);
            const uint32_t abase = smem_u32(sA), bbase = smem_u32(sB);
            const uint32_t lboB = (uint32_t)(N / 8) * 128;
            // operand descriptors of slot 0 / chunk 0: another one, or a second K
            // step, only moves the start address (see k_fwd_tc)
            const uint64_t d_ah = smem_desc(abase, 2048, 128);
            const uint64_t d_al = smem_desc(abase + RS_APLANE, 2048, 128);
            const uint64_t d_bh = smem_desc(bbase, lboB, 128);
            const uint64_t d_bl = smem_desc(bbase + (uint32_t)N * TC_BK * 2, lboB, 128);
            const uint32_t lo_ah = (uint32_t)d_ah, lo_al = (uint32_t)d_al;
            const uint32_t lo_bh = (uint32_t)d_bh, lo_bl = (uint32_t)d_bl;
            const uint32_t hi_a = (uint32_t)(d_ah >> 32), hi_b = (uint32_t)(d_bh >> 32);
            const uint32_t ka16 = (2u * 2048u) >> 4, kb16 = (2u * lboB) >> 4;
            static_assert(TC_BK == 32, "one stage is two K steps of 16");
            uint32_t sc = 0, it = 0, nres = 0;
            int cur_chan = -1;
            bool ok = true;
            for (int t = t_begin; t < t_end && ok; ++t, ++it) {
                const int chan = tiles[t].chan;
                if (chan != cur_chan) {
                    if (nres > 0) {
                        // every MMA that read the previous channel's slice has completed
                        umma_commit_elect(&S.bfree);
                        ok = __all_sync(~0u, mbar_wait(&S.bfree, (nres - 1) & 1, spin, abort, status));
                        if (!ok) break;
                    }
                    if (lane == 0) {
                        const unsigned char* src = (const unsigned char*)(planes + (int64_t)chan * 2 * NN) +
                                                   (int64_t)slice * nks * chunk_bytes;
                        mbar_arrive_expect_tx(&S.bres, (uint32_t)nks * chunk_bytes);
                        for (int q = 0; q < nks; ++q)
                            bulk_g2s(sB + (size_t)q * chunk_bytes, src + (size_t)q * chunk_bytes, chunk_bytes,
                                     &S.bres);
                    }
                    __syncwarp();
                    ok = __all_sync(~0u, mbar_wait(&S.bres, nres & 1, spin, abort, status));
                    ++nres;
                    if (!ok) break;
                    cur_chan = chan;
                }
                const int b = it & 1;
                ok = __all_sync(~0u, mbar_wait(&S.tempty[b], ((it >> 1) & 1) ^ 1, spin, abort, status));
                if (!ok) break;
                tc_fence_after();
                const uint32_t dt = tmem + (uint32_t)(b * N);
                // hi*lo and lo*hi over the slice, then hi*hi over the same stages
                for (int ks = 0; ks < nks; ++ks) {
                    const uint32_t q = sc + ks;
                    ok = __all_sync(~0u, mbar_wait(&S.full[q % STAGES], (q / STAGES) & 1, spin, abort, status));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t so = (uint32_t)((q % STAGES) * RS_ABYTES) >> 4;
                    const uint32_t bo = (uint32_t)ks * chunk_bytes >> 4;
                    umma_cross_elect(dt, lo_ah + so, lo_al + so, lo_bh + bo, lo_bl + bo, hi_a, hi_b, ka16, kb16,
                                     idesc, ks > 0 ? 1u : 0u);
                }
                if (!ok) break;
                for (int ks = 0; ks < nks; ++ks, ++sc) {
                    const uint32_t so = (uint32_t)((sc % STAGES) * RS_ABYTES) >> 4;
                    const uint32_t bo = (uint32_t)ks * chunk_bytes >> 4;
                    umma_main_elect(dt, lo_ah + so, lo_bh + bo, hi_a, hi_b, ka16, kb16, idesc);
                    umma_commit_elect(&S.empty[sc % STAGES]);
                }
                umma_commit_elect(&S.tfull[b]);
            }
            // every issued MMA completes before TMEM is released, and every
            // resident-operand copy lands before shared memory is released
            umma_commit_elect(&S.drain);
            int dummy = 0;
            mbar_wait(&S.drain, 0, drain_limit(spin), (volatile int*)&dummy, status);
            if (!ok && nres > 0) mbar_wait(&S.bres, (nres - 1) & 1, drain_limit(spin), (volatile int*)&dummy, status);
        }
        __syncwarp();
    } else if (warp >= 10 && warp < 12) {
        // ------------------------------------------------- finishing warps
        // One slice: its sums are V.  Warp 10 takes visibilities 0 .. 31 of a
        // tile, warp 11 the others.
        if (n_slices == 1) {
            const int jv = 32 * (warp - 10) + lane;
            bool ok = true;
            uint32_t ti = 0;
            for (int t = t_begin; t < t_end && ok; ++t, ++ti) {
                const VisTile tl = tiles[t];
                const int64_t j = tl.start + (jv < tl.count ? jv : 0);
                const RsFinishIn in = rs_finish_load(d, j, mode, yout);
                ok = __all_sync(0xffffffffu, mbar_wait(&S.xfull[ti & 1], (ti >> 1) & 1, spin, abort, status, 250));
                if (!ok) break;
                const double2 v = xsum[(ti & 1) * 64 + jv];
                double chi = 0.0;
                if (jv < tl.count) chi = rs_finish_vis(in, j, v.x, v.y, mode, yout);
                rs_finish_chi(chi, mode, jv, chi_part + (int64_t)t * 4);
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.xempty[ti & 1]);
            }
        }
    } else if (warp >= 12) {
        // --------------------------------------- Ey producers (two groups of 256 threads)
        // The groups build alternate stages: a stage's latencies (slot wait,
        // stores, proxy fence) then overlap the other group's.
        // thread -> (visibility j = ptid & 63, row group g = ptid >> 6): 8 image
        // rows of one visibility per stage, written as A rows row(j, Re), row(j, Im)
        regs_dec<RS_REGS_PROD>();
        const int pgrp = (threadIdx.x - 384) >> 8, ptid = (threadIdx.x - 384) & 255;
        const int jv = ptid & 63, g = ptid >> 6;
        // row(j, c) = 32 (j >> 4) + 16 c + (j & 15): the 32 lanes of a store
        // instruction fill four whole 128-byte core matrices (no bank conflicts)
        const int r0 = 32 * (jv >> 4) + (jv & 15);
        const int off = (g * 16 + (r0 >> 3)) * 128 + (r0 & 7) * 16;  // Re row; Im row at +256
        uint32_t sc = 0;
        bool ok = true;
        // the next tile's descriptor and phases arrive while this one is built
        bool valid_next = false;
        uint64_t pb_next = 0;
        auto load_tile = [&](int t) {
            const VisTile tl = tiles[t];
            valid_next = jv < tl.count;
            pb_next = valid_next ? d.pb[tl.start + jv] : 0;
        };
        if (t_begin < t_end) load_tile(t_begin);
        for (int t = t_begin; t < t_end && ok; ++t) {
            const bool valid = valid_next;
            const uint64_t pb = pb_next;
            if (t + 1 < t_end) load_tile(t + 1);
            cf2 step[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) step[q] = cis_neg(phase_mul(q, pb));
            const Rot8 w = rot8_of(step);
            for (int ks = 0; ks < nks; ++ks, ++sc) {
                if ((int)(sc & 1) != pgrp) continue;
                const int s = sc % STAGES;
                // the table values need no ring slot: compute them, then wait
                uint4 rh = {0, 0, 0, 0}, rl = {0, 0, 0, 0}, ih = {0, 0, 0, 0}, il = {0, 0, 0, 0};
                if (valid) {
                    const int n0 = slice * KS + ks * TC_BK + g * 8;
                    table8_split(cis_neg(phase_mul(n0 - c0, pb)), w, rh, rl, ih, il);
                }
                ok = __all_sync(0xffffffffu,
                                mbar_wait(&S.empty[s], ((sc / STAGES) & 1) ^ 1, spin, abort, status, 64));
                if (!ok) break;
                unsigned char* A = sA + s * RS_ABYTES;
                *(uint4*)(A + off) = rh;
                *(uint4*)(A + off + 256) = ih;
                *(uint4*)(A + RS_APLANE + off) = rl;
                *(uint4*)(A + RS_APLANE + off + 256) = il;
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.full[s]);
            }
        }
    } else if (warp < 8) {
        // ----------------------- epilogue (two groups of four warps)
        regs_inc<RS_REGS_EPI>();
        // TMEM lane = A row: warp q of a group holds visibilities 16q .. 16q+15,
        // lane L component L >> 4 (0: Re T, 1: Im T) of visibility 16q + (L & 15)
        const int grp = warp >> 2, quad = warp & 3;
        const int jv = 16 * quad + (lane & 15), comp = lane >> 4;
        uint32_t it = 0;  // tiles of this group
        bool ok = true;
        VisTile tl_next = {};
        uint64_t pa_next = 0, pb_next = 0;
        auto load_tile = [&](int t) {
            tl_next = tiles[t];
            const int64_t jn = tl_next.start + (jv < tl_next.count ? jv : 0);
            pa_next = d.pa[jn];
            pb_next = d.pb[jn];
        };
        if (t_begin + grp < t_end) load_tile(t_begin + grp);
        for (int t = t_begin + grp; t < t_end && ok; t += 2, ++it) {
            const VisTile tl = tl_next;
            const uint64_t pa = pa_next, pb = pb_next;
            if (t + 2 < t_end) load_tile(t + 2);
            const bool valid = jv < tl.count;
            const int64_t j = tl.start + (valid ? jv : 0);
            cf2 step[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) step[q] = cis_neg(phase_mul(q, pa));
            const cf2 step8 = cis_neg(phase_mul(8, pa));
            // slice 0 adds the column-mean part c_m S_k, S_k = sum_n Ey[k,n] in
            // closed form (accurate sincospi of the exact half-turn phases)
            float scomp = 0.f;
            if (slice == 0) {
                const float th = (float)(int64_t)((int64_t)pb >> 1) * 5.421010862427522e-20f;       // b/2, turns
                const float tn = (float)(int64_t)phase_mul(N / 2, pb) * 5.421010862427522e-20f;  // N b/2
                float sh, ch;
                sincospif(2.0f * th, &sh, &ch);      // sin(pi b), cos(pi b)
                const float snb = sinpif(2.0f * tn);  // sin(pi N b)
                const float D = (sh != 0.f) ? snb / sh : (float)N;
                scomp = comp ? sh * D : ch * D;
            }
            const float* cm = cmean + (int64_t)tl.chan * N;
            float s0 = 0.f, s1 = 0.f, c0s = 0.f, c1s = 0.f;  // compensated sums
            const int b = grp;
            ok = __all_sync(0xffffffffu, mbar_wait(&S.tfull[b], it & 1, spin, abort, status, 64));
            if (!ok) break;
            tc_fence_after();
            const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * N);
            // software pipeline over 16-column chunks: the TMEM load of chunk
            // q+1 is in flight while chunk q is reduced
            const int nq = N / 16;
            uint32_t tv[2][16];
            auto load_chunk = [&](int q, int slot) { tmem_ld16(lane_base + q * 16, tv[slot]); };
            // sum_k Ex[m0+k] t_k = base * sum_{k<8} step_k t_k + base8 * sum_{k<8} step_k t_{k+8}
            auto reduce_chunk = [&](int q, int slot) {
                const int m0 = q * 16;
                float4 cq4[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) cq4[k] = ((const float4*)(cm + m0))[k];
                const cf2 base = cis_neg(phase_mul(m0 - c0, pa));
                const cf2 base8 = cmul(base, step8);
                const float* cq = (const float*)cq4;
                float ux = 0.f, uy = 0.f, wx = 0.f, wy = 0.f;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float tk = fmaf(cq[k], scomp, __uint_as_float(tv[slot][k]));
                    const float tw = fmaf(cq[k + 8], scomp, __uint_as_float(tv[slot][k + 8]));
                    ux = fmaf(step[k].x, tk, ux);
                    uy = fmaf(step[k].y, tk, uy);
                    wx = fmaf(step[k].x, tw, wx);
                    wy = fmaf(step[k].y, tw, wy);
                }
                const float a0 = fmaf(base.x, ux, fmaf(-base.y, uy, fmaf(base8.x, wx, -base8.y * wy)));
                const float a1 = fmaf(base.x, uy, fmaf(base.y, ux, fmaf(base8.x, wy, base8.y * wx)));
                two_sum_acc(s0, c0s, a0);
                two_sum_acc(s1, c1s, a1);
            };
            load_chunk(0, 0);
            tmem_ld_wait(tv[0]);
            for (int q = 0; q < nq; q += 2) {
                load_chunk(q + 1, 1);  // nq is even
                reduce_chunk(q, 0);
                tmem_ld_wait(tv[1]);
                if (q + 2 < nq) load_chunk(q + 2, 0);
                reduce_chunk(q + 1, 1);
                if (q + 2 < nq) tmem_ld_wait(tv[0]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.tempty[b]);
            // lane < 16: (sum ReEx ReT, sum ImEx ReT); lane >= 16: (sum ReEx ImT, sum ImEx ImT)
            const double p0 = (double)s0 + (double)c0s, p1 = (double)s1 + (double)c1s;
            const double q0 = __shfl_xor_sync(0xffffffffu, p0, 16);
            const double q1 = __shfl_xor_sync(0xffffffffu, p1, 16);
            const double2 v = make_double2(p0 - q1, q0 + p1);
            if (n_slices > 1) {
                if (valid && comp == 0) vpart[(int64_t)slice * z_total + j] = v;
                continue;
            }
            // hand V to the finishing warps
            ok = __all_sync(0xffffffffu, mbar_wait(&S.xempty[grp], (it & 1) ^ 1, spin, abort, status, 32));
            if (!ok) break;
            if (comp == 0) xsum[grp * 64 + jv] = v;
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.xfull[grp]);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 8) {
        tc_fence_after();
        tmem_dealloc(tmem, tcols);
    }
}

// One block of 64 threads per tile: V = sum of the slice partials (fixed
// order), then the forward mode.
__global__ void __launch_bounds__(64) k_fwd_combine(DevData d, const VisTile* __restrict__ tiles,
                                                    const double2* vpart, int n_slices,
                                                    int64_t z_total, int mode, float2* yout, double* chi_part) {
    chain_next();
    chain_wait();
    const int t = blockIdx.x;
    const VisTile tl = tiles[t];
    const int jv = threadIdx.x;
    double chi = 0.0;
    if (jv < tl.count) {
        const int64_t j = tl.start + jv;
        double Vre = 0.0, Vim = 0.0;
        for (int s = 0; s < n_slices; ++s) {
            const double2 p = vpart[(int64_t)s * z_total + j];
            Vre += p.x;
            Vim += p.y;
        }
        chi = rs_finish_vis(rs_finish_load(d, j, mode, yout), j, Vre, Vim, mode, yout);
    }
    rs_finish_chi(chi, mode, jv, chi_part + (int64_t)t * 4);
}

template <int STAGES>
void launch_rs_variant(const DevData& d, const VisTile* tiles, int n_tiles, const void* planes, const float* cmean,
                       double2* vpart, int64_t z_total, int mode, float2* yout, double* chi_part, int grid, uint64_t spin,
                       int* status, cudaStream_t st) {
    const int smem = fwd_rs_smem_bytes(d.N, STAGES);
    // the register split waits for registers that only a launch with RS_REGS holds
    static const bool regs_ok = [] {
        cudaFuncAttributes at;
        return cudaFuncGetAttributes(&at, k_fwd_rs<STAGES>) == cudaSuccess && at.numRegs == RS_REGS;
    }();
    if (!regs_ok) grid = 0;  // a launch with no blocks leaves an error for the caller's check
    cudaFuncSetAttribute(k_fwd_rs<STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    launch_chained(k_fwd_rs<STAGES>, dim3(grid), RS_THREADS, smem, st, d.chain, 1, d, tiles, n_tiles,
                   (const uint16_t*)planes, cmean, vpart, z_total, mode, yout, chi_part, spin, status);
}

}  // namespace

int fwd_rs_smem_bytes(int N, int stages) {
    return fwd_rs_ks(N) * N * 4 + stages * RS_ABYTES + (fwd_rs_ks(N) == N ? 2 * 64 * 16 : 0) + 1024;
}

int launch_fwd_rs(const DevData& d, const VisTile* tiles, int n_tiles, const void* planes, const float* cmean,
                  int mode, float2* yout, double* chi_part, double2* vpart, int64_t z_total, int num_sms,
                  uint64_t spin, int* status, cudaStream_t st) {
    if (n_tiles <= 0) return 0;
    const int n_slices = d.N / fwd_rs_ks(d.N);
    // CTAs per slice: one per SM, at most one per tile
    const int per = std::max(1, std::min(num_sms / n_slices, n_tiles));
    const int grid = per * n_slices;
    const int stages = d.fwd_stages;
    auto launch = stages <= 4 ? launch_rs_variant<4> : stages == 5 ? launch_rs_variant<5> : launch_rs_variant<6>;
    launch(d, tiles, n_tiles, planes, cmean, vpart, z_total, mode, yout, chi_part, grid, spin, status, st);
    if (n_slices == 1) return 1;
    launch_chained(k_fwd_combine, dim3(n_tiles), 64, 0, st, d.chain, 1, d, tiles, (const double2*)vpart, n_slices, z_total,
                   mode, yout, chi_part);
    return 2;
}

}  // namespace msk
