// Tensor-core (tcgen05) adjoint of the BF16X3 form (its forward is in
// kernels_fwd.cu and kernels_fwd_rs.cu).  Both take the same table entries, so
// that the computed pair stays adjoint to itself: with the folded adjoint of
// FP16X3 (kernels_adj_fold.cu) beside the unfolded forward, a converged 64 x 64
// solve stops at Phi* + 3.6e-6 instead of Phi* + 2.8e-6.
//
// On the regular pixel grid the phase of Eq. (1) separates,
//   exp(-2 pi i (u x_m + v y_n)) = Ex[k,m] Ey[k,n],
//   Ex[k,m] = exp(-2 pi i u_k x_m),  Ey[k,n] = exp(-2 pi i v_k y_n),
// so the forward sum is   V_k = sum_m Ex[k,m] T[k,m],  T = Ey B^T  (B = A*I),
// and the chi^2 gradient (Eq. chi2gradient, Appendix C) is
//   G[n,m] = sum_k Re(Ey)[k,n] Re(P)[k,m] + Im(Ey)[k,n] Im(P)[k,m],
//   P[k,m] = y_k conj(Ex[k,m]),  y = w r.
// Both contractions run on the 5th-generation tensor cores (tcgen05.mma,
// kind::f16, accumulators in TMEM) in a 3-term BF16 split: x = hi + lo,
// a b ~= a_hi b_hi + a_hi b_lo + a_lo b_hi, FP32 accumulation.  The phase
// tables are never stored: producer warps generate each tile in shared
// memory from the exact fixed-point phases (one SFU sincos per 8 entries,
// the rest by complex rotation), already split and laid out as UMMA operands.
//
// Every mbarrier wait is bounded; a wait that runs out sets the device status
// word and the whole CTA unwinds, releasing its TMEM.
#include <cstdint>

#include "common.cuh"
#include "internal.h"
#include "reduce.cuh"

namespace msk {

// ===========================================================================
// Adjoint: split-K over visibilities.  A CTA owns a contiguous run of
// (channel, output block, visibility range) units, accumulates each unit's
// BLK x BLK block of G in TMEM over stages of 16 or 32 visibilities and drains it to an
// FP32 partial buffer; partials are summed in unit order afterwards (compensated
// FP32 two-sum).
// Operands are MN-major (8 consecutive pixels of one visibility per 16-byte
// core-matrix row), the layout the per-visibility phase recurrences produce.
// Roles: warps 0-3 (TMEM lane quadrants 0-3) drain the accumulator to the split-K
// partials every ADJ_DRAIN stages and at the end of each unit; warp 4 MMA + TMEM
// owner; warps 8-23 produce operand stages, two groups of eight on alternate
// stages, so that a stage's latencies (inputs, slot wait, stores, proxy fence)
// overlap the other group's.
//
// What bounds it: the MMAs (N >= 256: 1,536 clocks a stage) and the issue slots of
// the producers, which need nearly as many.  With all producer warps on the same
// stage its chain of latencies, about 2,100 clocks whatever N, was the bound.
// 1024 x 1024 with 100,000 visibilities: 743 -> 598 us (the MMAs alone 0.52 ms),
// 256 x 256 with 300,000: 148 -> 121 us, 128 x 128 with 100,003: 51 -> 31 us, and
// 28 with stages of 32 (CUDA events around the launch, about 5 us of which are
// theirs); the same bits.
// ===========================================================================
constexpr int ADJ_MAX_STAGES = 3;
// Stages of 16 visibilities (half as many of 32) accumulated in TMEM before the
// accumulator is added into the unit's FP32 partial.  The tensor core rounds each
// MMA's addition into its FP32 accumulator toward zero, so an accumulation of K
// MMAs (6 per 16 visibilities, K = 1,536) shrinks by up to K ulp, 1e-4 to 2e-4 at
// worst; sums of one sign, which shrink most, measured 4.3e-6 low however many
// visibilities a unit spans.  The drains add with round-to-nearest FP32 reductions,
// which have no such bias.
constexpr int ADJ_DRAIN = 256;
constexpr int ADJ_PRODUCERS = 16;  // producer warps: two groups of eight, alternate stages
constexpr int ADJ_THREADS = 32 * (8 + ADJ_PRODUCERS);

__host__ __device__ inline int adj_rows(int BLK) { return BLK < 128 ? 128 : BLK; }
// Visibilities per stage: 32 where three stages of them fit, one per lane of a
// producer warp, so that no two lanes form the same step table (128 x 128 with
// 100,003 visibilities 31 -> 28 us, 400,000 94 -> 80); else 16, and a warp's
// halves take different pixels.
__host__ __device__ inline int adj_vb(int BLK) { return BLK <= 128 ? 32 : 16; }
__host__ __device__ inline int adj_stage_bytes(int BLK) {
    return 4 * adj_rows(BLK) * adj_vb(BLK) * 2 + 4 * BLK * adj_vb(BLK) * 2;
}
int adj_tc_smem_bytes(int N, int stages) { return stages * adj_stage_bytes(tca_blk(N)) + 1024; }
__host__ __device__ inline uint32_t adj_tmem_cols(int BLK) {
    int c = (adj_rows(BLK) / 128) * BLK;
    uint32_t p = 32;
    while ((int)p < c) p <<= 1;
    return p;
}

// Layout of a unit's partial block (BLK x BLK floats): the element of block
// row n and column m lives at ((mt * BLK/16 + q) * 16 + k) * RB + r, with
// n = mt * 128 + r (r < RB = min(BLK, 128)) and m = 16 q + k.  For a fixed
// column, the rows a warp drains from its TMEM lanes are adjacent, so each
// drain load and store is one coalesced 128-byte access.
__host__ __device__ inline int64_t adj_partial_index(int n, int m, int BLK) {
    const int RB = BLK < 128 ? BLK : 128;
    return ((int64_t)((n / 128) * (BLK / 16) + m / 16) * 16 + (m % 16)) * RB + (n % 128);
}

// Inverse of adj_partial_index: block row and column of partial element i.
__host__ __device__ inline void adj_partial_rc(int64_t i, int BLK, int& n, int& m) {
    const int RB = BLK < 128 ? BLK : 128;
    const int r = (int)(i % RB);
    int64_t t = i / RB;
    const int k = (int)(t % 16);
    t /= 16;
    const int q = (int)(t % (BLK / 16)), mt = (int)(t / (BLK / 16));
    n = mt * 128 + r;
    m = q * 16 + k;
}

// Drain of the TMEM accumulator by warps 0-3 (TMEM lane quadrant = warp):
// partial (one unit's block, layout above) = [partial +] accumulator.
__device__ void adj_drain(uint32_t tmem, float* out, int BLK, int n_mt, int warp, int lane,
                                       bool first) {
    const int RB = BLK < 128 ? BLK : 128;
    for (int mt = 0; mt < n_mt; ++mt) {
        const int nrow = mt * 128 + warp * 32 + lane;
        const bool row_ok = nrow < BLK;
        const uint32_t lb = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(mt * BLK);
        // column m of this lane's row: base[m * RB], coalesced over the warp
        float* base = out + (row_ok ? adj_partial_index(nrow, 0, BLK) : 0);
        // one TMEM wait per 16-column chunk; the unit's first drain stores,
        // later ones add in place with reductions that return nothing, so the
        // drain never waits for a load of the partial (each element is added
        // to by one thread, in program order: the sum keeps its fixed order;
        // the reduction flushes subnormal values, far below any gradient
        // scale, to zero)
        for (int q = 0; q < BLK / 16; ++q) {
            uint32_t r[16];
            tmem_ld16(lb + q * 16, r);
            tmem_ld_wait(r);
            if (row_ok) {
                if (first) {
#pragma unroll
                    for (int k = 0; k < 16; ++k) base[(int64_t)(q * 16 + k) * RB] = __uint_as_float(r[k]);
                } else {
#pragma unroll
                    for (int k = 0; k < 16; ++k) atomicAdd(base + (int64_t)(q * 16 + k) * RB, __uint_as_float(r[k]));
                }
            }
        }
    }
}

struct AdjShared {
    uint64_t full[ADJ_MAX_STAGES];
    uint64_t empty[ADJ_MAX_STAGES];
    uint64_t tfull;
    uint64_t tempty;
    uint64_t drain;
    uint32_t tmem_base;
    int abort;
};

// FROM_UV: phase increments reduced from u, v inside the producers instead of
// read from the prepared arrays.
// ADJ_STAGES: depth of the shared-memory pipeline (autotuned).
template <bool FROM_UV, int ADJ_STAGES, int VB>
__global__ void __launch_bounds__(ADJ_THREADS, 1)
    k_adj_tc(DevData d, const AdjUnit* __restrict__ units, const int* __restrict__ cta_unit_off,
             const float2* y, float* __restrict__ partial, uint64_t spin, int* status) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ AdjShared S;
    constexpr int DRAIN = ADJ_DRAIN * 16 / VB;  // stages per accumulation
    const int N = d.N, c0 = N / 2;
    const int BLK = N < 256 ? N : 256;
    const int R = adj_rows(BLK);           // A rows (image rows n, padded to 128)
    const int n_mt = R / 128;
    const int nbx = N / BLK;
    const int a_plane = R * VB * 2, b_plane = BLK * VB * 2;
    const int stage_bytes = 4 * a_plane + 4 * b_plane;
    const uint32_t tcols = adj_tmem_cols(BLK);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u0 = cta_unit_off[blockIdx.x], u1 = cta_unit_off[blockIdx.x + 1];
    volatile int* abort = &S.abort;

    if (threadIdx.x == 0) {
        for (int s = 0; s < ADJ_STAGES; ++s) {
            mbar_init(&S.full[s], ADJ_PRODUCERS / 2);
            mbar_init(&S.empty[s], 1);
        }
        mbar_init(&S.tfull, 1);
        mbar_init(&S.tempty, 4);
        mbar_init(&S.drain, 1);
        S.abort = 0;
        mbar_fence_init();
    }
    if (warp == 4) {
        tmem_alloc(&S.tmem_base, tcols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;
    chain_next();
    chain_wait();

    if (warp == 4) {
        // The whole warp runs the issue loop, converged (every wait's outcome is
        // made warp-uniform), and one elected lane issues the MMAs and commits.
        {
            const uint32_t idesc = idesc_f16kind(128, BLK, 1, 1, 1);
            const uint32_t sbase = smem_u32(smem);
            const uint32_t lboA = (uint32_t)(R / 8) * 128, lboB = (uint32_t)(BLK / 8) * 128;
            // Operand descriptors of slot 0; another slot or row block only
            // moves the start address, whose field (address >> 4, low 14 bits)
            // takes the offset by plain addition (shared memory < 256 KB).
            // (the four planes of an operand share their strides: plane i is
            // plane 0 moved by i planes)
            const uint64_t d_a = smem_desc(sbase, lboA, 128);
            const uint64_t d_b = smem_desc(sbase + 4 * a_plane, lboB, 128);
            const uint64_t pa16 = (uint64_t)(a_plane >> 4), pb16 = (uint64_t)(b_plane >> 4);
            uint32_t sc = 0;
            bool ok = true;
            uint32_t it = 0;  // accumulation segments so far (tfull / tempty phases)
            for (int u = u0; u < u1 && ok; ++u) {
              const int nst = (int)((units[u].count + VB - 1) / VB);
              for (int seg0 = 0; seg0 < nst && ok; seg0 += DRAIN, ++it) {
                ok = __all_sync(~0u, mbar_wait(&S.tempty, (it & 1) ^ 1, spin, abort, status));
                if (!ok) break;
                tc_fence_after();
                const int seg1 = min(nst, seg0 + DRAIN);
                for (int ks = seg0; ks < seg1; ++ks, ++sc) {
                    const int s = sc % ADJ_STAGES;
                    ok = __all_sync(~0u, mbar_wait(&S.full[s], (sc / ADJ_STAGES) & 1, spin, abort, status));
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t so = (uint64_t)((uint32_t)(s * stage_bytes) >> 4);
                    const uint64_t bre_h = d_b + so, bre_l = bre_h + pb16;
                    const uint64_t bim_h = bre_h + 2 * pb16, bim_l = bre_h + 3 * pb16;
#pragma unroll
                    for (int kk = 0; kk < VB / 16; ++kk) {
                        for (int mt = 0; mt < n_mt; ++mt) {
                            const uint64_t ka = (uint64_t)(kk * 2 * lboA >> 4), kb = (uint64_t)(kk * 2 * lboB >> 4);
                            const uint64_t are_h = d_a + so + ka + (uint64_t)(mt * 2048 >> 4);  // 16 groups of 8 rows
                            const uint64_t are_l = are_h + pa16, aim_h = are_h + 2 * pa16, aim_l = are_h + 3 * pa16;
                            const uint32_t dt = tmem + (uint32_t)(mt * BLK);
                            const uint32_t acc = ks > seg0 || kk > 0 ? 1u : 0u;
                            // products sharing an A tile read it once (collector buffer)
                            umma_f16_elect<MMA_FILL>(dt, are_h, bre_h + kb, idesc, acc);
                            umma_f16_elect<MMA_LASTUSE>(dt, are_h, bre_l + kb, idesc, 1u);
                            umma_f16_elect<MMA_PLAIN>(dt, are_l, bre_h + kb, idesc, 1u);
                            umma_f16_elect<MMA_FILL>(dt, aim_h, bim_h + kb, idesc, 1u);
                            umma_f16_elect<MMA_LASTUSE>(dt, aim_h, bim_l + kb, idesc, 1u);
                            umma_f16_elect<MMA_PLAIN>(dt, aim_l, bim_h + kb, idesc, 1u);
                        }
                    }
                    umma_commit_elect(&S.empty[s]);
                }
                if (ok) umma_commit_elect(&S.tfull);
              }
            }
            umma_commit_elect(&S.drain);
            int dummy = 0;
            mbar_wait(&S.drain, 0, drain_limit(spin), (volatile int*)&dummy, status);
        }
        __syncwarp();
    } else if (warp < 4) {
        // -------------------------------------------------------------- drain
        // after the last stage of each accumulation segment into the unit's
        // partial
        uint32_t dr = 0;
        bool ok = true;
        for (int u = u0; u < u1 && ok; ++u) {
            const int nst = (int)((units[u].count + VB - 1) / VB);
            for (int seg0 = 0; seg0 < nst; seg0 += DRAIN, ++dr) {
                ok = __all_sync(0xffffffffu, mbar_wait(&S.tfull, dr & 1, spin, abort, status, 1024));
                if (!ok) break;
                tc_fence_after();
                adj_drain(tmem, partial + (int64_t)u * BLK * BLK, BLK, n_mt, warp, lane,
                          seg0 == 0 /* the unit's first segment stores */);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.tempty);
            }
        }
    } else if (warp >= 8) {
        // ---------------------------------------- producers (two groups of 8)
        // A warp-iteration builds an item (8 pixels of 32 visibilities), or two of
        // 16 visibilities, one per half-warp.  Whole warps take one side, Ey items (A operand)
        // or P items (B operand), so each thread builds one step table per
        // stage and the halves of a warp never diverge.  Every SM sub-partition
        // (warp % 4) has one warp of each side and group.
        const uint32_t grp = (warp - 8) >> 3;
        const bool ey_side = ((warp >> 2) & 1) == 0;
        constexpr int IPW = 32 / VB;          // items per warp-iteration
        const int half = VB == 16 ? lane >> 4 : 0;
        const int jj = lane & (VB - 1);       // visibility within the stage
        const int ngA = R / 8, ngB = BLK / 8;
        const int wi_end = (ey_side ? ngA : ngB) / IPW;
        const int ng = ey_side ? ngA : ngB, plane = ey_side ? a_plane : b_plane;
        const int side = ey_side ? 0 : 4 * a_plane;  // offset within a stage
        uint32_t sc = 0;  // stages so far, both groups'
        bool ok = true;
        for (int u = u0; u < u1 && ok; ++u) {
            const AdjUnit un = units[u];
            const int p0 = (ey_side ? un.block / nbx : un.block % nbx) * BLK - c0;  // first pixel
            const int nst = (int)((un.count + VB - 1) / VB);
            // this group's inputs of its next stage are loaded one stage ahead
            // (the phase of the side, and y on the P side)
            uint64_t np = 0;
            float2 ny = make_float2(0.f, 0.f);
            auto fetch = [&](int ks) {
                const int64_t kv = (int64_t)ks * VB + jj;
                np = 0;
                ny = make_float2(0.f, 0.f);
                if (ks < nst && kv < un.count) {
                    if (FROM_UV) np = ey_side ? to_fixed_turns(d.v[un.start + kv] * d.dy)
                                              : to_fixed_turns(d.u[un.start + kv] * d.dx);
                    else np = (ey_side ? d.pb : d.pa)[un.start + kv];
                    if (!ey_side) ny = y[un.start + kv];
                }
            };
            const int k0 = (int)((sc ^ grp) & 1);
            fetch(k0);
            for (int ks = k0; ks < nst; ks += 2) {
                const uint32_t q = sc + ks;
                const int s = q % ADJ_STAGES;
                const uint64_t ph = np;
                const cf2 yv = {ny.x, ny.y};
                const bool valid = (int64_t)ks * VB + jj < un.count;
                fetch(ks + 2);
                // rotation steps exp(-i 2 pi q c), q = 0..7, by powers of one SFU
                // value: c = b for the Ey side, a for the P side (computed before
                // the wait for the ring slot, which they do not need)
                cf2 st[8];
                st[0] = {1.f, 0.f};
                st[1] = cis_neg(ph);
                st[2] = cmul(st[1], st[1]);
                st[4] = cmul(st[2], st[2]);
                st[3] = cmul(st[2], st[1]);
                st[5] = cmul(st[4], st[1]);
                st[6] = cmul(st[4], st[2]);
                st[7] = cmul(st[4], st[3]);
                if (!ey_side) {
                    // P = y conj(Ex): conj(base) times conj(steps)
#pragma unroll
                    for (int k = 0; k < 8; ++k) st[k].y = -st[k].y;
                }
                const Rot8 w = rot8_of(st);
                ok = __all_sync(0xffffffffu, mbar_wait(&S.empty[s], ((q / ADJ_STAGES) & 1) ^ 1, spin,
                                                       abort, status, 64));
                if (!ok) break;
                unsigned char* dst0 = smem + s * stage_bytes + side + (jj >> 3) * ng * 128 + (jj & 7) * 16;
#pragma unroll 2
                for (int wi = warp & 3; wi < wi_end; wi += 4) {
                    const int g = IPW * wi + half;
                    uint4 rh = {0, 0, 0, 0}, rl = {0, 0, 0, 0}, ih = {0, 0, 0, 0}, il = {0, 0, 0, 0};
                    if (valid && g * 8 < BLK) {
                        const cf2 e = cis_neg(phase_mul(p0 + g * 8, ph));
                        table8_split(ey_side ? e : cmul(yv, cf2{e.x, -e.y}), w, rh, rl, ih, il);
                    }
                    unsigned char* dst = dst0 + g * 128;
                    *(uint4*)(dst + 0 * plane) = rh;
                    *(uint4*)(dst + 1 * plane) = rl;
                    *(uint4*)(dst + 2 * plane) = ih;
                    *(uint4*)(dst + 3 * plane) = il;
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.full[s]);
            }
            sc += nst;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 4) {
        tc_fence_after();
        tmem_dealloc(tmem, tcols);
    }
}

template <bool FROM_UV, int STAGES>
static void launch_adj_variant(const DevData& d, const AdjUnit* units, const int* cta_unit_off, int n_ctas,
                               const float2* y, float* partial, uint64_t spin, int* status, cudaStream_t st) {
    const int smem = adj_tc_smem_bytes(d.N, STAGES);
    auto kernel = adj_vb(tca_blk(d.N)) == 32 ? k_adj_tc<FROM_UV, STAGES, 32> : k_adj_tc<FROM_UV, STAGES, 16>;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    launch_chained(kernel, dim3(n_ctas), ADJ_THREADS, smem, st, d.chain, 1, d, units, cta_unit_off, y, partial, spin,
                   status);
}

void launch_adj_tc(const DevData& d, const AdjUnit* units, const int* cta_unit_off, int n_ctas, const float2* y,
                   float* partial, uint64_t spin, int* status, cudaStream_t st) {
    if (n_ctas <= 0) return;
    if (d.adj_stages == 2) launch_adj_variant<false, 2>(d, units, cta_unit_off, n_ctas, y, partial, spin, status, st);
    else launch_adj_variant<false, 3>(d, units, cta_unit_off, n_ctas, y, partial, spin, status, st);
}

void launch_adj_tc_uv(const DevData& d, const AdjUnit* units, const int* cta_unit_off, int n_ctas,
                      const float2* y, float* partial, uint64_t spin, int* status, cudaStream_t st) {
    if (n_ctas <= 0) return;
    launch_adj_variant<true, ADJ_MAX_STAGES>(d, units, cta_unit_off, n_ctas, y, partial, spin, status, st);
}

// Single channel: out[p] = A[p] * (unit partials summed in unit order,
// compensated FP32 (two-sum)).
__global__ void __launch_bounds__(256) k_adj_tc_reduce_out(int N, const int* __restrict__ cb_unit_off,
                                                           const float* __restrict__ partial,
                                                           const float* __restrict__ beam,
                                                           float* __restrict__ out) {
    const int64_t NN = (int64_t)N * N;
    const int BLK = N < 256 ? N : 256;
    const int nbx = N / BLK;
    // threads run over the partials' layout (coalesced reads); p is the pixel
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= NN) return;
    const int blk = (int)(i / ((int64_t)BLK * BLK));
    const int64_t loc = i % ((int64_t)BLK * BLK);
    int nl, ml;
    adj_partial_rc(loc, BLK, nl, ml);
    const int64_t p = (int64_t)((blk / nbx) * BLK + nl) * N + (blk % nbx) * BLK + ml;
    float s = 0.f, comp = 0.f;
    for (int u = cb_unit_off[blk]; u < cb_unit_off[blk + 1]; ++u)
        two_sum_acc(s, comp, partial[(int64_t)u * BLK * BLK + loc]);
    out[p] = beam[p] * (s + comp);
}

void launch_adj_tc_reduce_out(int N, const int* cb_unit_off, const float* partial, const float* beam,
                              float* out, cudaStream_t st) {
    k_adj_tc_reduce_out<<<prep_blocks(N), 256, 0, st>>>(N, cb_unit_off, partial, beam, out);
}

// Sum the unit partials of each (channel, block) in unit order (compensated
// FP32, stored as FP64) into gsum[c][N*N] (without the beam factor).
// Sum of the unit partials [u0, u1) at one element, compensated FP32 (Neumaier).
// A block of 256 threads handles 64 elements with 4 threads each: thread
// group g sums the g-th quarter of the units, and the four quarters are then
// combined in group order, so the sum has a fixed order (independent of the
// launch) and four times the loads in flight of one thread per element.
constexpr int RED_ELEMS = 64;
template <int SPLIT>
__device__ __forceinline__ void unit_sum_share(const float* src, int64_t stride, int u0, int u1, int g,
                                               float& s, float& comp) {
    const int ua = u0 + (u1 - u0) * g / SPLIT, ub = u0 + (u1 - u0) * (g + 1) / SPLIT;
    s = 0.f;
    comp = 0.f;
    int u = ua;
    for (; u + 8 <= ub; u += 8) {
        float q[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) q[k] = src[(int64_t)(u + k) * stride];
#pragma unroll
        for (int k = 0; k < 8; ++k) two_sum_acc(s, comp, q[k]);
    }
    for (; u < ub; ++u) two_sum_acc(s, comp, src[(int64_t)u * stride]);
}

// Combine the four groups' (sum, compensation) pairs through shared memory;
// returns the total in group 0's threads.
__device__ __forceinline__ float unit_sum_combine(float s, float comp, int el, int g, float (*sh)[RED_ELEMS][2]) {
    sh[g][el][0] = s;
    sh[g][el][1] = comp;
    __syncthreads();
    float t = sh[0][el][0], c = sh[0][el][1];
    for (int k = 1; k < 4; ++k) {
        two_sum_acc(t, c, sh[k][el][0]);
        c += sh[k][el][1];
    }
    return t + c;
}

__global__ void __launch_bounds__(256) k_adj_tc_reduce(DevData d, const int* __restrict__ cb_unit_off,
                                                       const float* partial,
                                                       double* __restrict__ gsum, float* __restrict__ out32) {
    __shared__ float sh[4][RED_ELEMS][2];
    chain_next();
    chain_wait();
    const int N = d.N;
    const int64_t NN = (int64_t)N * N;
    const int BLK = N < 256 ? N : 256;
    const int nbx = N / BLK;
    const int c = blockIdx.y;
    const int el = threadIdx.x % RED_ELEMS, g = threadIdx.x / RED_ELEMS;
    // threads run over the partials' layout (coalesced reads); p is the pixel
    const int64_t i = (int64_t)blockIdx.x * RED_ELEMS + el;
    const bool in = i < NN;
    const int blk = in ? (int)(i / ((int64_t)BLK * BLK)) : 0;
    const int64_t loc = in ? i % ((int64_t)BLK * BLK) : 0;
    const int cb = c * nbx * nbx + blk;
    const int u0 = in ? cb_unit_off[cb] : 0, u1 = in ? cb_unit_off[cb + 1] : 0;
    float s, comp;
    unit_sum_share<4>(partial + loc, (int64_t)BLK * BLK, u0, u1, g, s, comp);
    const float tot = unit_sum_combine(s, comp, el, g, sh);
    if (g != 0 || !in) return;
    int nl, ml;
    adj_partial_rc(loc, BLK, nl, ml);
    const int64_t p = (int64_t)((blk / nbx) * BLK + nl) * N + (blk % nbx) * BLK + ml;
    if (out32) out32[(int64_t)c * NN + p] = tot;
    else gsum[(int64_t)c * NN + p] = (double)tot;
}

void launch_adj_tc_reduce(const DevData& d, const int* cb_unit_off, const float* partial, double* gsum, float* out32,
                          cudaStream_t st) {
    const int64_t NN = (int64_t)d.N * d.N;
    dim3 grid((unsigned)((NN + RED_ELEMS - 1) / RED_ELEMS), d.C);
    launch_chained(k_adj_tc_reduce, grid, 256, 0, st, d.chain, 1, d, cb_unit_off, partial, gsum, out32);
}

// The unit-partial sum of k_adj_tc_reduce followed directly by the gradient
// assembly (Eq. chi2gradient with the beam factor, Eq. Sgradient, the positive
// projection at I = G), for images of one channel each (one image, or a cube):
// the same arithmetic as the separate reduction and assembly, one launch.
// log(I/G) stays FP64: with an FP32 log the 50-iteration solve of the
// 64x64 problem ended 1.4e-3 (relative L2) from the oracle's image in the
// BF16X3 form, against 4.6e-4.
// With sc.scal set, sc.splits further blocks per image (the first ones in
// x, so that they start with the first wave) run the objective's scalar
// reduction (scalars_block): it needs only the forward's chi^2 partials and
// the prep's entropy partials, so it shares this launch instead of taking one
// of its own.
// SPLIT groups per element as above, or one where an output block has few units and
// the images fill the SMs with a thread per pixel: every thread then has a pixel's
// FP64 operations, which a quarter of the threads would have to wait out.  One against
// four groups, us by CUDA events: 1024 x 1024 (10 units a block) 31 and 58, 512 x 512
// (38) 18 and 21, 256 x 256 with 64 channels (3) 99 and 214, 6 (26) 22 and 33, 3 (51) 19
// and 22, 2 (76) 22 and 19, 1 (152) 31 and 16; 128 x 128 with 4 channels (38) 14 and
// 14; 64 x 64 with 4 (38, 64 blocks of a thread per pixel) 14 and 12.
template <int SPLIT>
__global__ void __launch_bounds__(256) k_adj_tc_reduce_grad(DevData d, ImgSrc src,
                                                            const int* __restrict__ cb_unit_off,
                                                            const float* partial, int projected,
                                                            float* out32, double* full64, double* proj64,
                                                            ScalarArgs sc) {
    constexpr int ELEMS = 256 / SPLIT;
    __shared__ float sh[4][RED_ELEMS][2];
    chain_next();
    chain_wait();
    const int N = d.N;
    const int64_t NN = (int64_t)N * N;
    const int n_scal = sc.scal ? sc.splits : 0;
    if ((int)blockIdx.x < n_scal) {
        scalars_block<256>(d, sc, blockIdx.y, blockIdx.x);
        return;
    }
    const int BLK = N < 256 ? N : 256;
    const int nbx = N / BLK;
    const int c = blockIdx.y;  // channel = image
    const int el = threadIdx.x % ELEMS, g = threadIdx.x / ELEMS;
    const int64_t i = (int64_t)(blockIdx.x - n_scal) * ELEMS + el;
    const bool in = i < NN;
    const int blk = in ? (int)(i / ((int64_t)BLK * BLK)) : 0;
    const int64_t loc = in ? i % ((int64_t)BLK * BLK) : 0;
    const int cb = c * nbx * nbx + blk;
    const int u0 = in ? cb_unit_off[cb] : 0, u1 = in ? cb_unit_off[cb + 1] : 0;
    float s, comp;
    unit_sum_share<SPLIT>(partial + loc, (int64_t)BLK * BLK, u0, u1, g, s, comp);
    float tot = s + comp;
    if constexpr (SPLIT == 4) tot = unit_sum_combine(s, comp, el, g, sh);
    if (g != 0 || !in) return;
    int nl, ml;
    adj_partial_rc(loc, BLK, nl, ml);
    const int64_t p = (int64_t)((blk / nbx) * BLK + nl) * N + (blk % nbx) * BLK + ml;
    const double x = img_value(src, c, p, NN);
    // (a converged solve of this form stops within 7 % of its test's bound: not one
    // rounding moves)
    double gr = (double)d.beam[(int64_t)c * NN + p] * (double)tot;
    if (d.lambda != 0.0)
        gr += d.lambda * (1.0 + (src.lg ? src.lg[(int64_t)c * NN + p] : log_ratio(x, d.G, d.ginv)));
    const double gp = project_pixel(d, x, gr);
    if (full64) full64[(int64_t)c * NN + p] = gr;
    if (proj64) proj64[(int64_t)c * NN + p] = gp;
    if (out32) out32[(int64_t)c * NN + p] = (float)(projected ? gp : gr);
}

void launch_adj_tc_reduce_grad(const DevData& d, const ImgSrc& src, const int* cb_unit_off, const float* partial,
                               int projected, float* out32, double* full64, double* proj64,
                               const ScalarArgs& sc, int n_units, cudaStream_t st) {
    const int64_t NN = (int64_t)d.N * d.N;
    const int nbx = d.N / tca_blk(d.N);
    const bool one = n_units <= 40ll * d.C * nbx * nbx && d.C * NN >= 256 * 256;
    const int elems = one ? 256 : RED_ELEMS;
    const dim3 grid((unsigned)((NN + elems - 1) / elems) + (sc.scal ? sc.splits : 0), d.C);
    auto kernel = one ? k_adj_tc_reduce_grad<1> : k_adj_tc_reduce_grad<4>;
    launch_chained(kernel, grid, 256, 0, st, d.chain, 1, d, src, cb_unit_off, partial, projected, out32, full64, proj64, sc);
}

}  // namespace msk
