// Tensor-core (tcgen05) adjoint of the FP16X3 form (its forward is in
// kernels_fold.cu, the BF16X3 pair in kernels_fwd*.cu and kernels_tc.cu).
//
// On the regular pixel grid the phase of Eq. (1) separates, and about the point
// half a pixel below pixel N/2 the rows are symmetric: row n = N/2 + j sits at
// j + 1/2, row N/2 - 1 - j at -(j + 1/2).  With
//   c_j + i y_j = exp(-2 pi i (j + 1/2) b),  b = frac(v dy),  a = frac(u dx),
//   P[k,m] = y_k exp(2 pi i ((m - N/2) a_k - b_k / 2)),   y = w r,
// the chi^2 gradient (Eq. chi2gradient, Appendix C) of the two rows is
//   G[N/2 + j, m] = D0 + D1,  G[N/2 - 1 - j, m] = D0 - D1,
//   D0[j,m] = sum_k c_j[k] Re P[k,m],  D1[j,m] = sum_k y_j[k] Im P[k,m]:
// a visibility takes N^2 multiply-adds where the unfolded sum takes 2 N^2, and
// 3 N table entries instead of 4 N, with exactly the same sums.
//
// Both contractions run on the 5th-generation tensor cores (tcgen05.mma,
// kind::f16, accumulators in TMEM) in a 3-term FP16 split: x = hi + lo,
// a b ~= a_hi b_hi + a_hi b_lo + a_lo b_hi, FP32 accumulation.  The phase
// tables are never stored: producer warps generate each stage in shared memory
// from the exact fixed-point phases (one evaluated phase factor per thread and
// stage, the rest by complex rotation), already split and laid out as UMMA
// operands.
//
// Every mbarrier wait is bounded; a wait that runs out sets the device status
// word and the whole CTA unwinds, releasing its TMEM.
#include <cstdint>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "reduce.cuh"

namespace msk {

// ===========================================================================
// Adjoint: split-K over visibilities.  A CTA owns a contiguous run of
// (channel, output block, visibility range) units, accumulates each unit's
// D0 and D1 blocks in TMEM over stages of VB visibilities and drains them to an
// FP32 partial buffer; partials are summed in unit order afterwards
// (compensated FP32 two-sum).
//
// Shapes (the M side of an MMA has 128 rows):
//   N >= 256  rows j (128 per block), columns m (256 per block): D0 and D1 fill
//             the 512 TMEM columns;
//   N = 128   rows m, columns j (64): full MMAs that rows j would half fill;
//   N = 64    rows [Re P; Im P] of the 64 m, columns [c_j, y_j] (32 + 32): one
//             product whose two diagonal quarters are D0 and D1.
// Operands are MN-major (8 consecutive pixels of one visibility per 16-byte
// core-matrix row), the layout the per-visibility phase recurrences produce.
//
// Roles: warps 0-11 produce the stages (4 of them the row factors, 8 the P
// entries: 4, 2 or 1 groups of 8 pixels each, so every warp and every SM
// sub-partition carries the same work) and drain the accumulators; warp 12
// issues the MMAs and owns TMEM.
//
// What bounds it: at 256 x 256 with 999,600 visibilities 0.22 ms, against 0.45 ms
// for the unfolded kernel it replaces (CUDA events); a stage of 32 visibilities
// holds 1,536 clocks of MMA work (0.16 ms) and takes about 2,000.  The producers
// set that: issue slots are 66 % active, about 440 instructions per producer warp and
// stage, and a warp can only fill a slot while the ring's other one is in the MMAs.
// Stages of 16 visibilities repeat the step factors twice as often
// (0.28 ms); rotating every entry instead of sharing products about a group's
// centre, and converting hi back to FP32, took 0.245 ms; packed FP32 pairs 0.258.
// ===========================================================================
constexpr int ADJ_MAX_STAGES = 3;
// Visibilities accumulated in TMEM before the accumulators are added into the
// unit's FP32 partials.  The tensor core rounds each MMA's addition into its
// FP32 accumulator toward zero, so an accumulation of K MMAs (3 per 16
// visibilities, K = 1,536) shrinks by up to K ulp, 1e-4 to 2e-4 at worst; sums of
// one sign, which shrink most, measured 8.6e-6 low however many visibilities a unit
// spans.  The drains add with round-to-nearest FP32 reductions, which have no such
// bias.
constexpr int ADJ_DRAIN = 8192;
constexpr int ADJ_PRODUCER_WARPS = 12;
constexpr int ADJ_THREADS = 32 * (ADJ_PRODUCER_WARPS + 1);

enum AdjShape { ADJ_WIDE = 0, ADJ_128 = 1, ADJ_64 = 2 };
template <int SHAPE>
struct AdjGeo {
    static constexpr int NSET = SHAPE == ADJ_64 ? 1 : 2;           // products D0, D1 (ADJ_64: one for both)
    static constexpr int NB = SHAPE == ADJ_WIDE ? 256 : 64;        // MMA columns
    static constexpr int GPW = SHAPE == ADJ_WIDE ? 4 : SHAPE == ADJ_128 ? 2 : 1;  // 8-pixel groups per producer warp
    static constexpr int ROWS = SHAPE == ADJ_64 ? 64 : 128;        // rows and columns of a D block
    static constexpr int COLS = SHAPE == ADJ_WIDE ? 256 : SHAPE == ADJ_128 ? 64 : 32;
    static constexpr int a_plane(int vb) { return 128 * vb * 2; }
    static constexpr int b_plane(int vb) { return NB * vb * 2; }
    static constexpr int stage_bytes(int vb) { return 2 * NSET * (a_plane(vb) + b_plane(vb)); }
};

// Visibilities per stage: 32 (one per lane of a producer warp, so a thread's
// step factors serve all of its groups); 16 where three stages would not fit.
__host__ __device__ inline int adj_vb(int N, int stages) { return N >= 256 && stages > 2 ? 16 : 32; }
int adj_fold_smem_bytes(int N, int stages) {
    const int vb = adj_vb(N, stages);
    const int st = N >= 256 ? AdjGeo<ADJ_WIDE>::stage_bytes(vb)
                 : N > 64   ? AdjGeo<ADJ_128>::stage_bytes(vb)
                            : AdjGeo<ADJ_64>::stage_bytes(vb);
    return stages * st + 1024;
}

// A unit's partials (BLK x BLK floats): the D0 block, then the D1 block, each
// [column][row].  For a fixed column, the rows a warp drains from its TMEM
// lanes are adjacent, so each drain access is one coalesced 128-byte line.
//
// Drain of the accumulators by the twelve producer warps: warp w reads TMEM
// lane quadrant w % 4, the columns are dealt to the three warps of a quadrant.
// The unit's first drain stores, later ones add in place with reductions that
// return nothing, so the drain never waits for a load of the partial (each
// element is added to by one thread, in program order: the sum keeps its fixed
// order; the reduction flushes subnormal values, far below any gradient scale,
// to zero).  Kept out of line so that its registers do not add to the
// producers' loop.
template <int SHAPE>
__device__ __noinline__ void adj_drain(uint32_t tmem, float* out, int warp, int lane, bool first) {
    using Geo = AdjGeo<SHAPE>;
    const int quad = warp & 3;
    const uint32_t lb = tmem + ((uint32_t)(quad * 32) << 16);
    constexpr int TC = Geo::NSET * Geo::NB;  // TMEM columns
    // ADJ_64: lanes 0-63 hold Re P (its c columns: D0), lanes 64-127 Im P (its
    // y columns: D1)
    const int row = SHAPE == ADJ_64 ? (quad & 1) * 32 + lane : quad * 32 + lane;
    for (int q = warp >> 2; q < TC / 16; q += 3) {
        if (SHAPE == ADJ_64 && (q * 16 >= 32) != (quad >= 2)) continue;
        uint32_t r[16];
        tmem_ld16(lb + q * 16, r);
        tmem_ld_wait(r);
        float* base = out + (int64_t)q * 16 * Geo::ROWS + row;
        if (first) {
#pragma unroll
            for (int k = 0; k < 16; ++k) base[k * Geo::ROWS] = __uint_as_float(r[k]);
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) atomicAdd(base + k * Geo::ROWS, __uint_as_float(r[k]));
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

// y is scaled by pow2_scale_for(ymax[0]) (a power of two, undone when the
// partials are summed).
// STAGES: depth of the shared-memory pipeline (autotuned).
template <int SHAPE, int VB, int STAGES>
__global__ void __launch_bounds__(ADJ_THREADS, 1)
    k_adj_fold(DevData d, const AdjUnit* __restrict__ units, const int* __restrict__ cta_unit_off,
             const float2* y, const float* ymax, float* __restrict__ partial,
             uint64_t spin, int* status) {
    using Geo = AdjGeo<SHAPE>;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ AdjShared S;
    const int N = d.N, c0 = N / 2;
    constexpr int A_PLANE = Geo::a_plane(VB), B_PLANE = Geo::b_plane(VB);
    constexpr int STAGE = Geo::stage_bytes(VB);
    constexpr int B_OFF = 2 * Geo::NSET * A_PLANE;  // B planes after the A planes: [set][hi, lo]
    constexpr uint32_t TCOLS = Geo::NSET * Geo::NB;
    constexpr int64_t UNIT = 2ll * Geo::ROWS * Geo::COLS;  // floats of a unit's partials
    const int nbx = SHAPE == ADJ_WIDE ? N / 256 : 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u0 = cta_unit_off[blockIdx.x], u1 = cta_unit_off[blockIdx.x + 1];
    volatile int* abort = &S.abort;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&S.full[s], ADJ_PRODUCER_WARPS);
            mbar_init(&S.empty[s], 1);
        }
        mbar_init(&S.tfull, 1);
        mbar_init(&S.tempty, ADJ_PRODUCER_WARPS);
        mbar_init(&S.drain, 1);
        S.abort = 0;
        mbar_fence_init();
    }
    if (warp == ADJ_PRODUCER_WARPS) {
        tmem_alloc(&S.tmem_base, TCOLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;
    chain_next();
    chain_wait();

    if (warp == ADJ_PRODUCER_WARPS) {
        // The whole warp runs the issue loop, converged (every wait's outcome is
        // made warp-uniform), and one elected lane issues the MMAs and commits.
        const uint32_t idesc = idesc_f16kind(128, Geo::NB, 1, 1, 0);
        const uint32_t sbase = smem_u32(smem);
        constexpr uint32_t LBO_A = 128 / 8 * 128, LBO_B = Geo::NB / 8 * 128;
        // Operand descriptors of slot 0; another slot, plane or K step (two
        // 8-visibility groups) only moves the start address, whose field
        // (address >> 4, low 14 bits) takes the offset by plain addition
        // (shared memory < 256 KB).
        const uint64_t d_a = smem_desc(sbase, LBO_A, 128);
        const uint64_t d_b = smem_desc(sbase + B_OFF, LBO_B, 128);
        uint32_t sc = 0;
        bool ok = true;
        uint32_t it = 0;  // accumulation segments so far (tfull / tempty phases)
        for (int u = u0; u < u1 && ok; ++u) {
            const int nst = (int)((units[u].count + VB - 1) / VB);
            for (int seg0 = 0; seg0 < nst && ok; seg0 += ADJ_DRAIN / VB, ++it) {
                ok = __all_sync(~0u, mbar_wait(&S.tempty, (it & 1) ^ 1, spin, abort, status));
                if (!ok) break;
                tc_fence_after();
                const int seg1 = min(nst, seg0 + ADJ_DRAIN / VB);
                for (int ks = seg0; ks < seg1; ++ks, ++sc) {
                    const int s = sc % STAGES;
                    ok = __all_sync(~0u, mbar_wait(&S.full[s], (sc / STAGES) & 1, spin, abort, status));
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t so = (uint64_t)((uint32_t)(s * STAGE) >> 4);
#pragma unroll
                    for (int kk = 0; kk < VB / 16; ++kk) {
#pragma unroll
                        for (int p = 0; p < Geo::NSET; ++p) {
                            const uint64_t ah = d_a + so + ((2 * p * A_PLANE + kk * 2 * LBO_A) >> 4);
                            const uint64_t bh = d_b + so + ((2 * p * B_PLANE + kk * 2 * LBO_B) >> 4);
                            const uint64_t al = ah + (A_PLANE >> 4), bl = bh + (B_PLANE >> 4);
                            const uint32_t dt = tmem + (uint32_t)(p * Geo::NB);
                            // products sharing an A tile read it once (collector buffer)
                            umma_f16_elect<MMA_FILL>(dt, ah, bh, idesc, (ks > seg0 || kk > 0) ? 1u : 0u);
                            umma_f16_elect<MMA_LASTUSE>(dt, ah, bl, idesc, 1u);
                            umma_f16_elect<MMA_PLAIN>(dt, al, bh, idesc, 1u);
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
        __syncwarp();
    } else {
        // ---------------------------------------------------- producers
        // Warps 0-3: row factors (c_j, y_j); warps 4-11: P.  Warp w of a side
        // builds GPW consecutive groups of 8 pixels; lane = visibility (VB = 16:
        // the half-warps take different groups).
        const float ysc = pow2_scale_for(ymax[0]);
        auto produce = [&](auto side) {
            constexpr bool ROW = decltype(side)::value;
            constexpr int GPT = VB == 32 ? Geo::GPW : (Geo::GPW + 1) / 2;  // groups per thread
            const int kv = lane & (VB - 1);
            const int g0 = (ROW ? warp : warp - 4) * Geo::GPW + (VB == 32 ? 0 : (lane >> 4) * GPT);
            // A side: 128 rows; B side: NB columns.  SECOND (y_j or Im P) is the
            // other product's plane pair, or for ADJ_64 the other half of the
            // rows or columns.
            constexpr bool A_SIDE = ROW == (SHAPE == ADJ_WIDE);
            constexpr int NG = (A_SIDE ? 128 : Geo::NB) / 8;
            constexpr int PLANE = A_SIDE ? A_PLANE : B_PLANE;
            constexpr int SECOND = Geo::NSET == 2 ? 2 * PLANE : NG / 2 * 128;
            unsigned char* dst0 = smem + (A_SIDE ? 0 : B_OFF) + ((kv >> 3) * NG + g0) * 128 + (kv & 7) * 16;
            uint32_t sc = 0, dr = 0;  // stages produced; accumulator drains
            bool ok = true;
            for (int u = u0; u < u1 && ok; ++u) {
                const AdjUnit un = units[u];
                const int count = (int)un.count, nst = (count + VB - 1) / VB;
                // centre of this thread's first 8 pixels within the image: j + 1/2,
                // or m - N/2 in half units
                const int pix = ROW ? (un.block / nbx) * 128 + g0 * 8 + 4
                                    : 2 * ((un.block % nbx) * 256 + g0 * 8 - c0) + 7;
                const uint32_t neg = pix < 0 ? ~0u : 0u;
                // per-visibility inputs of the next stage are loaded one stage
                // ahead; beyond the unit y is zero (and with it P)
                uint64_t na = 0, nb = 0;
                float2 ny = {0.f, 0.f};
                auto fetch = [&](int ks) {
                    const int k = ks * VB + kv;
                    if (!ROW) ny = make_float2(0.f, 0.f);
                    if (k < count) {
                        const int64_t i = un.start + k;
                        nb = d.pb[i];
                        if (!ROW) {
                            na = d.pa[i];
                            ny = y[i];
                        }
                    }
                };
                fetch(0);
                for (int seg0 = 0; seg0 < nst && ok; seg0 += ADJ_DRAIN / VB) {
                    const int seg1 = min(nst, seg0 + ADJ_DRAIN / VB);
                    for (int ks = seg0; ks < seg1; ++ks, ++sc) {
                        const int s = sc % STAGES;
                        // steps and the first group's factor, before the wait for
                        // the ring slot, which they do not need; P rotates the
                        // other way
                        HalfSteps st = half_steps(ROW ? nb : na);
                        cf2 e;
                        if (ROW) {
                            e = cis_neg_accurate(phase_hi((uint32_t)pix, nb));
                        } else {
                            // high word of pix (a / 2) - b / 2
                            const uint64_t ha = (uint64_t)((int64_t)na >> 1);
                            const uint32_t ph = phase_hi((uint32_t)pix, ha) - ((uint32_t)ha & neg) -
                                                (uint32_t)((int32_t)(uint32_t)(nb >> 32) >> 1);
                            const cf2 f = cis_neg_accurate(ph);
                            e = cmul(cf2{ny.x * ysc, ny.y * ysc}, cf2{f.x, -f.y});
#pragma unroll
                            for (int k = 0; k < 4; ++k) st.s[k].y = -st.s[k].y;
                            st.s8.y = -st.s8.y;
                        }
                        fetch(ks + 1);
                        ok = __all_sync(0xffffffffu, mbar_wait(&S.empty[s], ((sc / STAGES) & 1) ^ 1, spin, abort,
                                                               status, 32));
                        if (!ok) break;
                        unsigned char* dst = dst0 + s * STAGE;
#pragma unroll
                        for (int r = 0; r < GPT; ++r) {
                            uint4 rh, rl, ih, il;
                            table8_complex(e, st, rh, rl, ih, il);
                            *(uint4*)(dst + r * 128) = rh;
                            *(uint4*)(dst + r * 128 + PLANE) = rl;
                            *(uint4*)(dst + r * 128 + SECOND) = ih;
                            *(uint4*)(dst + r * 128 + SECOND + PLANE) = il;
                            if (r + 1 < GPT) e = cmul(e, st.s8);
                        }
                        fence_async_smem();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&S.full[s]);
                    }
                    // drain after the last stage of each accumulation segment
                    if (!ok) break;
                    ok = __all_sync(0xffffffffu, mbar_wait(&S.tfull, dr & 1, spin, abort, status, 100));
                    if (!ok) break;
                    tc_fence_after();
                    adj_drain<SHAPE>(tmem, partial + u * UNIT, warp, lane,
                                     seg0 == 0 /* the unit's first segment stores */);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&S.tempty);
                    ++dr;
                }
            }
        };
        if (warp < 4) produce(std::true_type{});
        else produce(std::false_type{});
    }

    tc_fence_before();
    __syncthreads();
    if (warp == ADJ_PRODUCER_WARPS) {
        tc_fence_after();
        tmem_dealloc(tmem, TCOLS);
    }
}

struct AdjArgs {
    DevData d;
    const AdjUnit* units;
    const int* cta_unit_off;
    int n_ctas;
    const float2* y;
    const float* ymax;
    float* partial;
    uint64_t spin;
    int* status;
    cudaStream_t st;
};

template <int SHAPE, int VB, int STAGES>
static void launch_adj_variant(const AdjArgs& a) {
    const int smem = STAGES * AdjGeo<SHAPE>::stage_bytes(VB) + 1024;
    cudaFuncSetAttribute(k_adj_fold<SHAPE, VB, STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    launch_chained(k_adj_fold<SHAPE, VB, STAGES>, dim3(a.n_ctas), ADJ_THREADS, smem, a.st, a.d.chain, 1, a.d, a.units,
                   a.cta_unit_off, a.y, a.ymax, a.partial, a.spin, a.status);
}

void launch_adj_fold(const DevData& d, const AdjUnit* units, const int* cta_unit_off, int n_ctas, const float2* y,
                     const float* ymax, float* partial, uint64_t spin, int* status, cudaStream_t st) {
    if (n_ctas <= 0) return;
    const AdjArgs a{d, units, cta_unit_off, n_ctas, y, ymax, partial, spin, status, st};
    if (d.N >= 256) {
        if (d.adj_stages <= 2) launch_adj_variant<ADJ_WIDE, 32, 2>(a);
        else launch_adj_variant<ADJ_WIDE, 16, 3>(a);
    } else if (d.N > 64) {
        if (d.adj_stages <= 2) launch_adj_variant<ADJ_128, 32, 2>(a);
        else launch_adj_variant<ADJ_128, 32, 3>(a);
    } else {
        if (d.adj_stages <= 2) launch_adj_variant<ADJ_64, 32, 2>(a);
        else launch_adj_variant<ADJ_64, 32, 3>(a);
    }
}

// ===========================================================================
// Sum of the unit partials per (channel, block), then the two mirror rows of
// every element.  A block takes 32 rows x COLS columns of both D blocks, with
// SPLIT threads per element: group g sums the g-th share of the units in order
// (compensated FP32, Neumaier) and the shares are combined in order, so the sum
// has a fixed order (independent of the launch) and SPLIT times the loads in
// flight of one thread per element.  The loads are coalesced along the rows of
// the partials' layout.  N >= 256: four columns (whose pixels are neighbours in
// an image row); smaller images take one, so that 64 x 64 still fills 64 blocks.
// ===========================================================================
constexpr int RED_ROWS = 32;
constexpr int RED_AHEAD = 8;  // units whose partials are loaded together
template <bool WIDE>
struct RedGeo {
    static constexpr int COLS = WIDE ? 4 : 1, ELEMS = RED_ROWS * COLS;
    static constexpr int SPLIT = WIDE ? 4 : 8, THREADS = ELEMS * SPLIT;
};
enum RedOut { RED_GSUM = 0, RED_GRAD = 1 };

struct RedArgs {
    const int* cb_unit_off;
    const float* partial;
    const float* ymax;   // partials are divided by pow2_scale_for(ymax[0])
    double* gsum;        // RED_GSUM: [C][N*N], without the beam factor (or as FP32 in out32)
    int projected;       // RED_GRAD
    float* out32;        // (each output nullable)
    double *full64, *proj64;
    ScalarArgs sc;       // RED_GRAD: objective scalars, see below
};

// RED_GRAD is the unit-partial sum followed directly by the gradient assembly
// (Eq. chi2gradient with the beam factor, Eq. Sgradient, the positive projection
// at I = G), for images of one channel each (one image, or a cube): the same
// arithmetic as RED_GSUM and k_finalize, one launch.
// log(I/G) stays FP64: with an FP32 log the 50-iteration solve of the
// 64x64 problem ended 1.4e-3 (relative L2) from the oracle's image in the
// BF16X3 form, against 4.6e-4.
// With sc.scal set, sc.splits further blocks per image (the first ones in
// x, so that they start with the first wave) run the objective's scalar
// reduction (scalars_block): it needs only the forward's chi^2 partials and
// the prep's entropy partials, so it shares this launch instead of taking one
// of its own.
template <int OUT, bool WIDE>
__global__ void __launch_bounds__(RedGeo<WIDE>::THREADS) k_adj_fold_reduce(DevData d, ImgSrc src, RedArgs a) {
    constexpr int COLS = RedGeo<WIDE>::COLS, ELEMS = RedGeo<WIDE>::ELEMS, SPLIT = RedGeo<WIDE>::SPLIT;
    constexpr int THREADS = RedGeo<WIDE>::THREADS;
    __shared__ float sh[2][SPLIT][ELEMS][2];
    const int N = d.N;
    const int64_t NN = (int64_t)N * N;
    chain_next();
    chain_wait();
    const int n_scal = OUT == RED_GRAD && a.sc.scal ? a.sc.splits : 0;
    if (OUT == RED_GRAD && (int)blockIdx.x < n_scal) {
        scalars_block<THREADS>(d, a.sc, blockIdx.y, blockIdx.x);
        return;
    }
    const int BLK = N < 256 ? N : 256, nbx = N / BLK;
    const int rows = BLK < 128 ? BLK : 128, half = BLK * BLK / 2;
    const int c = blockIdx.y;  // channel
    // element of this thread: block, row r and column q of the D blocks
    const int el = threadIdx.x % ELEMS, g = threadIdx.x / ELEMS;
    const int tiles_blk = half / ELEMS, row_tiles = rows / RED_ROWS;
    const int tile = blockIdx.x - n_scal, blk = tile / tiles_blk, t = tile % tiles_blk;
    const int r = (t % row_tiles) * RED_ROWS + el % RED_ROWS;
    const int q = (t / row_tiles) * COLS + el / RED_ROWS;
    const int cb = c * nbx * nbx + blk;
    const int u0 = a.cb_unit_off[cb], u1 = a.cb_unit_off[cb + 1];
    const int ua = u0 + (u1 - u0) * g / SPLIT, ub = u0 + (u1 - u0) * (g + 1) / SPLIT;
    const int64_t stride = 2ll * half;
    const float* p = a.partial + (int64_t)ua * stride + (int64_t)q * rows + r;
    float s0 = 0.f, e0 = 0.f, s1 = 0.f, e1 = 0.f;
    int u = ua;
    for (; u + RED_AHEAD <= ub; u += RED_AHEAD) {
        float x[RED_AHEAD], z[RED_AHEAD];
#pragma unroll
        for (int k = 0; k < RED_AHEAD; ++k) {
            x[k] = p[k * stride];
            z[k] = p[k * stride + half];
        }
#pragma unroll
        for (int k = 0; k < RED_AHEAD; ++k) {
            two_sum_acc(s0, e0, x[k]);
            two_sum_acc(s1, e1, z[k]);
        }
        p += RED_AHEAD * stride;
    }
    for (; u < ub; ++u, p += stride) {
        two_sum_acc(s0, e0, p[0]);
        two_sum_acc(s1, e1, p[half]);
    }
    sh[0][g][el][0] = s0;
    sh[0][g][el][1] = e0;
    sh[1][g][el][0] = s1;
    sh[1][g][el][1] = e1;
    __syncthreads();
    // one thread per pixel, two per element; consecutive threads along the image
    // row (N >= 256: the element's column; else its row)
    for (int o = threadIdx.x; o < 2 * ELEMS; o += THREADS) {
        const int sign = o / ELEMS, i = o % ELEMS;
        const int er = WIDE ? i / COLS : i % RED_ROWS, eq = WIDE ? i % COLS : i / RED_ROWS;
        const int e = eq * RED_ROWS + er;
        float tot[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float s = sh[h][0][e][0], cc = sh[h][0][e][1];
            for (int k = 1; k < SPLIT; ++k) {
                two_sum_acc(s, cc, sh[h][k][e][0]);
                cc += sh[h][k][e][1];
            }
            tot[h] = s + cc;
        }
        const int rr = (t % row_tiles) * RED_ROWS + er, qq = (t / row_tiles) * COLS + eq;
        const int j = WIDE ? (blk / nbx) * 128 + rr : qq, m = WIDE ? (blk % nbx) * 256 + qq : rr;
        const int n = sign ? N / 2 - 1 - j : N / 2 + j;
        const double inv = pow2_inverse(pow2_scale_for(a.ymax[0]));
        const float other = sign ? -tot[1] : tot[1];
        const int64_t pix = (int64_t)c * NN + (int64_t)n * N + m;
        if (OUT == RED_GSUM) {
            const double g = ((double)tot[0] + (double)other) * inv;
            if (a.out32) a.out32[pix] = (float)g;
            else a.gsum[pix] = g;
        } else {
            const double x = img_value(src, c, (int64_t)n * N + m, NN);
            // (an image per channel: pix is the image's pixel too)
            const double gr = pixel_gradient(d, d.beam[pix], tot[0], other, inv, x, src.lg ? src.lg + pix : nullptr);
            const double gp = project_pixel(d, x, gr);
            if (a.full64) a.full64[pix] = gr;
            if (a.proj64) a.proj64[pix] = gp;
            if (a.out32) a.out32[pix] = (float)(a.projected ? gp : gr);
        }
    }
}

template <int OUT>
static void launch_red(const DevData& d, const ImgSrc& src, const RedArgs& a, int extra, cudaStream_t st) {
    const int64_t half = (int64_t)d.N * d.N / 2;
    if (d.N >= 256)
        launch_chained(k_adj_fold_reduce<OUT, true>, dim3((unsigned)(half / RedGeo<true>::ELEMS) + extra, d.C),
                       RedGeo<true>::THREADS, 0, st, d.chain, 1, d, src, a);
    else
        launch_chained(k_adj_fold_reduce<OUT, false>, dim3((unsigned)(half / RedGeo<false>::ELEMS) + extra, d.C),
                       RedGeo<false>::THREADS, 0, st, d.chain, 1, d, src, a);
}

void launch_adj_fold_reduce(const DevData& d, const int* cb_unit_off, const float* partial, const float* ymax,
                            double* gsum, float* out32, cudaStream_t st) {
    RedArgs a{};
    a.out32 = out32;
    a.cb_unit_off = cb_unit_off;
    a.partial = partial;
    a.ymax = ymax;
    a.gsum = gsum;
    launch_red<RED_GSUM>(d, ImgSrc{}, a, 0, st);
}

void launch_adj_fold_reduce_grad(const DevData& d, const ImgSrc& src, const int* cb_unit_off, const float* partial,
                               const float* ymax, int projected, float* out32, double* full64, double* proj64,
                               const ScalarArgs& sc, cudaStream_t st) {
    const RedArgs a{cb_unit_off, partial, ymax, nullptr, projected, out32, full64, proj64, sc};
    launch_red<RED_GRAD>(d, src, a, sc.scal ? sc.splits : 0, st);
}

}  // namespace msk
