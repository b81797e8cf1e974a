// Device-side control of the projected Polak-Ribiere CG (Eq. minproblem):
// the conjugate-gradient bookkeeping, the line-search state machine and the
// loop conditions run on the device, so that a whole solve is one launch of a
// CUDA graph whose loops are conditional WHILE nodes (the host reads the results
// once, at the end).
//
// A small problem's solve is a chain of kernels of a few microseconds each, so
// its time is their number.  Every control step therefore runs in the last block
// of the reduction that feeds it: the dot products and the vector update before
// them are one launch with the decision per image (k_cg_beta, k_cg_direction),
// the scalar reduction of a probe feeds the line search and, at its end, accepts
// the step (k_scalars_ls).  64 x 64 with 10,260 visibilities, five iterations with 60
// probes: 2.06 ms with a launch per step and per reduction stage, 1.67 ms so.
//
// Per iteration (every scalar in FP64):
//   beta_i = max(0, (g - g_prev).g / g_prev.g_prev)  (0 on restarts: the first
//            iteration, every RESTART-th, and when d is not a descent direction)
//   d_i    = -g + beta_i d (bound-projected), slope_i = grad Phi . d
//   alpha0 = -slope / sum w |F(A d)|^2  (the minimiser of chi^2's quadratic
//            model along d), or max I / max |d| without curvature
//   line search on phi(alpha) = Phi(max(I + alpha d, G)): bracketing (shrink by
//            SHRINK until phi < phi(0), else expand by GOLD while phi falls),
//            Brent's method (Brent 1973, ch. 5), then one Newton step on
//            central differences over x -/+ h, h = min(POLISH alpha0, x / 2),
//            clamped to that interval
//   I      = max(I + alpha d, G)
// Images of a cube are independent CGs that share every batched evaluation.
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"
#include "reduce.cuh"
#include "solver.h"

namespace msk {

namespace {

// Constants of this library's reading of the paper's Numerical-Recipes style
// CG (Section 4.2 names the method, not its constants).
constexpr double GOLD = 1.618033988749895;    // bracket expansion ratio
constexpr double CGOLD = 0.3819660112501051;  // golden-section fraction
constexpr double SHRINK = 0.25;               // trial-step reduction
constexpr int LS_MAX_EVALS = 20;              // objective evaluations per line search (+2 for the last step)
constexpr double LS_TOL = 1e-3;               // relative step tolerance (Brent)
constexpr double LS_EPS = 1e-10;              // absolute tolerance / first trial step
constexpr int RESTART = 50;                   // steepest-descent restart period
constexpr double POLISH = 0.2;                // half-width of the final 3-point Newton step / step
constexpr int CTL_THREADS = 256;

__device__ __forceinline__ bool finite(double x) { return isfinite(x); }

// Line search on phi(alpha), alpha >= 0, as a resumable state machine: start()
// sets the first request, feed() takes phi(req) and sets the next request
// until the phase is DONE (alpha = the accepted step, 0 when no decrease was
// found within the budget).
__device__ void ls_finish(LineSearchState& s, double al, double f) {
    if (al > 0.0) {
        s.px = al;
        s.pfx = f;
        s.ph = fmin(POLISH * s.a0, 0.5 * al);
        s.req = s.px + s.ph;
        s.phase = LS_POL_P;
        return;
    }
    s.alpha = al;
    s.phase = LS_DONE;
}

__device__ void ls_brent_step(LineSearchState& s) {
    if (s.nb >= s.budget) {
        s.evals += s.nb;
        ls_finish(s, s.x, s.fx);
        return;
    }
    const double xm = 0.5 * (s.lo + s.hi);
    const double tol1 = LS_TOL * fabs(s.x) + s.eps;
    const double tol2 = 2.0 * tol1;
    if (fabs(s.x - xm) <= tol2 - 0.5 * (s.hi - s.lo)) {
        s.evals += s.nb;
        ls_finish(s, s.x, s.fx);
        return;
    }
    bool golden = true;
    if (fabs(s.e) > tol1) {
        // parabola through (v, fv), (w, fw), (x, fx)
        const double r = (s.x - s.w) * (s.fx - s.fv);
        double q = (s.x - s.v) * (s.fx - s.fw);
        double p = (s.x - s.v) * q - (s.x - s.w) * r;
        q = 2.0 * (q - r);
        if (q > 0.0) p = -p;
        else q = -q;
        const double e_prev = s.e;
        s.e = s.d;
        if (fabs(p) < fabs(0.5 * q * e_prev) && p > q * (s.lo - s.x) && p < q * (s.hi - s.x)) {
            s.d = p / q;
            const double t = s.x + s.d;
            if ((t - s.lo) < tol2 || (s.hi - t) < tol2) s.d = (xm >= s.x) ? tol1 : -tol1;
            golden = false;
        }
    }
    if (golden) {
        s.e = (s.x >= xm) ? (s.lo - s.x) : (s.hi - s.x);
        s.d = CGOLD * s.e;
    }
    s.req = (fabs(s.d) >= tol1) ? s.x + s.d : s.x + (s.d >= 0.0 ? tol1 : -tol1);
}

__device__ void ls_brent_start(LineSearchState& s) {
    s.lo = s.a;
    s.hi = s.c;
    s.x = s.w = s.v = s.b;
    s.fx = s.fw = s.fv = s.fb;
    s.d = s.e = 0.0;
    s.nb = 0;
    s.budget = LS_MAX_EVALS - s.evals;
    s.phase = LS_BRENT;
    ls_brent_step(s);
}

__device__ void ls_shrink_check(LineSearchState& s) {
    if (s.fb >= s.fa && s.evals < LS_MAX_EVALS) {
        s.c = s.b;
        s.fc = s.fb;
        s.b = s.b * SHRINK;
        s.req = s.b;
        s.phase = LS_SHRINK;
    } else if (s.fb >= s.fa) {
        ls_finish(s, 0.0, s.f0);
    } else {
        ls_brent_start(s);
    }
}

__device__ void ls_expand_check(LineSearchState& s) {
    if (s.fc < s.fb && s.evals < LS_MAX_EVALS) {
        s.a = s.b;
        s.fa = s.fb;
        s.b = s.c;
        s.fb = s.fc;
        s.c = s.b + GOLD * (s.b - s.a);
        s.req = s.c;
        s.phase = LS_EXPAND;
    } else if (s.fc < s.fb) {
        ls_finish(s, s.c, s.fc);
    } else {
        ls_brent_start(s);
    }
}

__device__ void ls_start(LineSearchState& s, double phi0, double alpha0) {
    s.a0 = alpha0;
    s.f0 = phi0;
    s.eps = LS_EPS * alpha0;
    s.a = 0.0;
    s.fa = phi0;
    s.b = alpha0;
    s.req = s.b;
    s.evals = 0;
    s.alpha = 0.0;
    s.phase = LS_INIT;
}

__device__ void ls_feed(LineSearchState& s, double f) {
    switch (s.phase) {
        case LS_INIT:
            s.fb = f;
            s.evals = 1;
            if (s.fb >= s.fa) {
                s.c = s.b;
                s.fc = s.fb;
                ls_shrink_check(s);
            } else {
                s.c = s.b + GOLD * (s.b - s.a);
                s.req = s.c;
                s.phase = LS_EXPAND;
            }
            break;
        case LS_SHRINK:
            s.fb = f;
            s.evals += 1;
            ls_shrink_check(s);
            break;
        case LS_EXPAND:
            s.fc = f;
            s.evals += 1;
            ls_expand_check(s);
            break;
        case LS_BRENT: {
            const double t = s.req, ft = f;
            s.nb += 1;
            if (ft <= s.fx) {
                if (t >= s.x) s.lo = s.x;
                else s.hi = s.x;
                s.v = s.w;
                s.fv = s.fw;
                s.w = s.x;
                s.fw = s.fx;
                s.x = t;
                s.fx = ft;
            } else {
                if (t < s.x) s.lo = t;
                else s.hi = t;
                if (ft <= s.fw || s.w == s.x) {
                    s.v = s.w;
                    s.fv = s.fw;
                    s.w = t;
                    s.fw = ft;
                } else if (ft <= s.fv || s.v == s.x || s.v == s.w) {
                    s.v = t;
                    s.fv = ft;
                }
            }
            ls_brent_step(s);
            break;
        }
        case LS_POL_P:
            s.pfp = f;
            s.evals += 1;
            s.req = s.px - s.ph;
            s.phase = LS_POL_M;
            break;
        case LS_POL_M: {
            const double fm = f;
            s.evals += 1;
            double x = s.px;
            const double curv = s.pfp - 2.0 * s.pfx + fm;
            if (curv > 0.0) {
                const double t = s.px - s.ph * (s.pfp - fm) / (2.0 * curv);
                x = fmin(fmax(t, s.px - s.ph), s.px + s.ph);
            }
            s.alpha = x;
            s.phase = LS_DONE;
            break;
        }
        default:
            break;
    }
}

// Block-wide OR of a flag; every thread gets the result.
__device__ int block_any(int x) { return __syncthreads_or(x); }

// The loop condition: written to ctl (read by the host when graphs are off)
// and, inside a graph, to the conditional node's handle.
__device__ void set_cond(CgControl* ctl, int which, int value, unsigned long long handle) {
    if (threadIdx.x != 0) return;
    if (which == 0) ctl->outer = value;
    else ctl->inner = value;
    if (handle) cudaGraphSetConditional((cudaGraphConditionalHandle)handle, value ? 1u : 0u);
}

__device__ void hist_row(const CgControl* ctl, double* hist, int i, int k, double phi, double chi, double S,
                         double alpha, double beta, double evals) {
    double* h = hist + ((int64_t)i * ctl->hist_stride + k) * 6;
    h[0] = phi;
    h[1] = chi;
    h[2] = S;
    h[3] = alpha;
    h[4] = beta;
    h[5] = evals;
}

// After the first objective + gradient: per-image state and history row 0.
__global__ void __launch_bounds__(CTL_THREADS) k_cg_init(int NI, CgImage* st, CgControl* ctl, const double* scal,
                                                         double* hist, const int* dstatus,
                                                         unsigned long long h_outer) {
    int any = 0, bad = 0;
    for (int i = threadIdx.x; i < NI; i += CTL_THREADS) {
        CgImage& s = st[i];
        s.phi = scal[3 + 3 * i];
        s.chi = scal[4 + 3 * i];
        s.S = scal[5 + 3 * i];
        s.beta = s.slope = s.alpha = 0.0;
        s.iters = s.evals = 0;
        s.ls.phase = LS_DONE;
        s.active = 1;
        if (!(finite(s.phi) && finite(s.chi) && finite(s.S))) {
            bad = 1;
            s.active = 0;
        }
        hist_row(ctl, hist, i, 0, s.phi, s.chi, s.S, 0.0, 0.0, 0.0);
        any |= s.active;
    }
    any = block_any(any);
    bad = block_any(bad);
    if (threadIdx.x == 0) {
        if (bad) ctl->status |= CG_NONFINITE;
        if (*dstatus) ctl->status |= CG_DEVICE;
    }
    __syncthreads();
    set_cond(ctl, 0, any && ctl->k < ctl->n_iter && ctl->status == 0, h_outer);
}

// ---------------------------------------------------------------------------
// Sums of x0, x1 and maxima of m0, m1 over an image's pixels: a block's result
// goes to part, and the image's last block to finish (count[i], zero between
// launches) combines the blocks' results in order.  True in the threads of that
// block, which hold the totals in thread 0.
// ---------------------------------------------------------------------------
struct Totals {
    double x0, x1, m0, m1;
};

__device__ __forceinline__ void block_max2(double& x, double& y, double (*sh)[2]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x = fmax(x, __shfl_down_sync(0xffffffffu, x, o));
        y = fmax(y, __shfl_down_sync(0xffffffffu, y, o));
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
        sh[w][0] = x;
        sh[w][1] = y;
    }
    __syncthreads();
    if (w == 0) {
        x = sh[l % (CTL_THREADS / 32)][0];
        y = sh[l % (CTL_THREADS / 32)][1];
#pragma unroll
        for (int o = CTL_THREADS / 64; o > 0; o >>= 1) {
            x = fmax(x, __shfl_down_sync(0xffffffffu, x, o));
            y = fmax(y, __shfl_down_sync(0xffffffffu, y, o));
        }
    }
    __syncthreads();
}

template <bool MAXIMA>
__device__ bool image_totals(int i, double& x0, double& x1, double& m0, double& m1, Totals* part, unsigned* count) {
    __shared__ double sh[CTL_THREADS / 32][2];
    __shared__ bool last;
    const int nblk = gridDim.x;
    block_sum2<CTL_THREADS>(x0, x1, sh);
    if (MAXIMA) block_max2(m0, m1, sh);
    if (threadIdx.x == 0) {
        part[(int64_t)i * nblk + blockIdx.x] = {x0, x1, m0, m1};
        __threadfence();
        last = atomicAdd(count + i, 1u) == (unsigned)nblk - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    x0 = x1 = m0 = m1 = 0.0;
    for (int b = threadIdx.x; b < nblk; b += CTL_THREADS) {
        const double* p = (const double*)(part + (int64_t)i * nblk + b);
        x0 += __ldcg(p);
        x1 += __ldcg(p + 1);
        if (MAXIMA) {
            m0 = fmax(m0, __ldcg(p + 2));
            m1 = fmax(m1, __ldcg(p + 3));
        }
    }
    block_sum2<CTL_THREADS>(x0, x1, sh);
    if (MAXIMA) block_max2(m0, m1, sh);
    if (threadIdx.x == 0) count[i] = 0;
    return true;
}

// Polak-Ribiere beta from g_prev.g_prev and (g - g_prev).g; direction mode 1
// (d = -g + beta d) or 2 (d = -g) for active images, 0 keep.
__global__ void __launch_bounds__(CTL_THREADS) k_cg_beta(DevData d, const double* __restrict__ g,
                                                         const double* __restrict__ g_prev, CgImage* st,
                                                         const CgControl* ctl, double* beta, int* mode,
                                                         Totals* part, unsigned* count) {
    const int64_t NN = (int64_t)d.N * d.N;
    const int i = blockIdx.y;
    const int64_t p = (int64_t)blockIdx.x * CTL_THREADS + threadIdx.x;
    double x0 = 0.0, x1 = 0.0, m0 = 0.0, m1 = 0.0;
    if (p < NN) {
        const double a = g[i * NN + p], b = g_prev[i * NN + p];
        x0 = b * b;
        x1 = (a - b) * a;
    }
    if (!image_totals<false>(i, x0, x1, m0, m1, part, count) || threadIdx.x != 0) return;
    const int k = ctl->k;
    double b = 0.0;
    if (k > 0 && k % RESTART != 0 && x0 > 0.0) b = fmax(0.0, x1 / x0);
    st[i].beta = b;
    beta[i] = b;
    mode[i] = st[i].active ? (b == 0.0 ? 2 : 1) : 0;
}

// Search direction per image (mode 0 keep, 1 d = -g + beta d, 2 d = -g; a pixel
// at I = G cannot move down), its slope grad Phi . d, max I and max |d| (dots).
// An active image whose d is not a descent direction gets mode 2 and beta 0, the
// others mode 0; the second launch (again) takes the former only, and stops an
// image still without descent.
__global__ void __launch_bounds__(CTL_THREADS) k_cg_direction(DevData d, bool again, const double* __restrict__ I,
                                                              const double* __restrict__ g,
                                                              const double* __restrict__ gfull, CgImage* st,
                                                              CgControl* ctl, double* beta, int* mode, double* dir,
                                                              double* dots, Totals* part, unsigned* count) {
    const int64_t NN = (int64_t)d.N * d.N;
    const int i = blockIdx.y, md = mode[i];
    if (again && md == 0) return;
    const int64_t p = (int64_t)blockIdx.x * CTL_THREADS + threadIdx.x;
    double x0 = 0.0, x1 = 0.0, m0 = 0.0, m1 = 0.0;
    if (p < NN) {
        const int64_t q = i * NN + p;
        double nd;
        if (md == 0) {
            nd = dir[q];
        } else {
            nd = md == 2 ? -g[q] : -g[q] + beta[i] * dir[q];
            if (I[q] <= d.G && nd < 0.0) nd = 0.0;
            dir[q] = nd;
        }
        x0 = gfull[q] * nd;
        m0 = I[q];
        m1 = fabs(nd);
    }
    if (!image_totals<true>(i, x0, x1, m0, m1, part, count) || threadIdx.x != 0) return;
    CgImage& s = st[i];
    s.slope = x0;
    dots[2 * i] = m0;
    dots[2 * i + 1] = m1;
    const bool uphill = s.active && s.slope >= 0.0;
    if (again) {
        if (uphill) {
            s.active = 0;
            ctl->stopped_early = 1;
        }
    } else {
        mode[i] = uphill ? 2 : 0;
        if (uphill) {
            s.beta = 0.0;
            beta[i] = 0.0;
        }
    }
}

// Accepted steps: alpha per image (0 for images that stop: no decrease found).
__device__ void accept_steps(int NI, CgImage* st, CgControl* ctl, double* alpha) {
    int stopped = 0;
    const int fail = ctl->status != 0;
    for (int i = threadIdx.x; i < NI; i += CTL_THREADS) {
        CgImage& s = st[i];
        double a = 0.0;
        if (s.active) {
            if (fail || s.ls.phase != LS_DONE || !(s.ls.alpha > 0.0)) {
                s.active = 0;
                stopped = 1;
            } else {
                a = s.ls.alpha;
            }
        }
        s.alpha = a;
        alpha[i] = a;
    }
    stopped = block_any(stopped);
    if (threadIdx.x == 0 && stopped && !fail) ctl->stopped_early = 1;
}

// The scalar reduction, then in its last block one step of the line searches.
// START: scal holds 1/2 sum w |F(A d)|^2 per image in its chi^2 slot (curvature
// pass), dots = (max I, max |d|): first trial step and line-search start.
// Otherwise one probe was evaluated: scal holds Phi(max(I + alpha d, G)) - Phi(I).
// When no image asks for another probe, the steps are accepted.
template <bool START>
__global__ void __launch_bounds__(CTL_THREADS) k_scalars_ls(DevData d, ScalarArgs sc, CgImage* st, CgControl* ctl,
                                                            const double* dots, double* alpha, const int* dstatus,
                                                            unsigned long long h_inner) {
    // The state machine runs on a copy whose loads are all in flight during the
    // reduction: in place, every branch would wait for its own.
    const int NI = d.n_images;
    chain_next();
    chain_wait();
    CgImage mine;
    if ((int)threadIdx.x < NI) mine = st[threadIdx.x];
    if (!scalars_block<CTL_THREADS>(d, sc, blockIdx.x, blockIdx.y)) return;
    __syncthreads();
    int run = 0, bad = 0;
    for (int i = threadIdx.x; i < NI; i += CTL_THREADS) {
        if (i != (int)threadIdx.x) mine = st[i];
        bool r = false;
        if (START) {
            mine.ls.phase = LS_DONE;
            if (mine.active) {
                const double curv = 2.0 * __ldcg(sc.scal + 4 + 3 * i);
                if (!finite(curv)) bad = 1;
                double a0 = curv > 0.0 ? -mine.slope / curv : 0.0;
                if (!(a0 > 0.0)) a0 = dots[2 * i] / dots[2 * i + 1];
                ls_start(mine.ls, mine.phi, a0);
                r = true;
            }
        } else if (mine.active && mine.ls.phase != LS_DONE) {
            const double f = mine.phi + __ldcg(sc.scal + 3 + 3 * i);
            if (!finite(f)) bad = 1;
            ls_feed(mine.ls, f);
            r = mine.ls.phase != LS_DONE;
        }
        st[i].ls = mine.ls;
        alpha[i] = r ? mine.ls.req : 0.0;
        run |= r;
    }
    run = block_any(run);
    bad = block_any(bad);
    if (threadIdx.x == 0) {
        if (START) {
            ctl->rounds = 0;
        } else {
            ctl->rounds += 1;
            ctl->probes += 1;
        }
        if (bad) ctl->status |= CG_NONFINITE;
        if (*dstatus) ctl->status |= CG_DEVICE;
        // every line search ends within LS_MAX_EVALS + 2 probes; the cap only
        // guards the loop against a state that should not occur
        if (!START && ctl->rounds >= LS_MAX_EVALS + 8) ctl->status |= CG_LOOP;
    }
    __syncthreads();
    const bool more = run && ctl->status == 0;
    if (!more) accept_steps(NI, st, ctl, alpha);
    set_cond(ctl, 1, more, h_inner);
}

// After the step's objective + gradient: history row k + 1, counters and the
// outer loop condition.
__global__ void __launch_bounds__(CTL_THREADS) k_cg_record(int NI, CgImage* st, CgControl* ctl, const double* scal,
                                                           double* hist, const int* dstatus,
                                                           unsigned long long h_outer) {
    const int k = ctl->k;
    int any = 0, bad = 0;
    for (int i = threadIdx.x; i < NI; i += CTL_THREADS) {
        CgImage& s = st[i];
        if (s.alpha > 0.0) {
            const double ev = (double)(s.ls.evals + 2);
            s.iters = k + 1;
            s.evals += s.ls.evals + 2;
            s.phi = scal[3 + 3 * i];
            s.chi = scal[4 + 3 * i];
            s.S = scal[5 + 3 * i];
            if (!(finite(s.phi) && finite(s.chi) && finite(s.S))) bad = 1;
            hist_row(ctl, hist, i, k + 1, s.phi, s.chi, s.S, s.alpha, s.beta, ev);
        } else {
            hist_row(ctl, hist, i, k + 1, s.phi, s.chi, s.S, 0.0, 0.0, 0.0);
        }
        any |= s.active;
    }
    any = block_any(any);
    bad = block_any(bad);
    if (threadIdx.x == 0) {
        ctl->k = k + 1;
        if (bad) ctl->status |= CG_NONFINITE;
        if (*dstatus) ctl->status |= CG_DEVICE;
    }
    __syncthreads();
    set_cond(ctl, 0, any && k + 1 < ctl->n_iter && ctl->status == 0, h_outer);
}

}  // namespace

void launch_cg_init(int NI, CgImage* st, CgControl* ctl, const double* scal, double* hist, const int* dstatus,
                    unsigned long long h_outer, cudaStream_t s) {
    k_cg_init<<<1, CTL_THREADS, 0, s>>>(NI, st, ctl, scal, hist, dstatus, h_outer);
}
void launch_cg_beta(const DevData& d, const double* g, const double* g_prev, CgImage* st, const CgControl* ctl,
                    double* beta, int* mode, double* part, unsigned* count, cudaStream_t s) {
    k_cg_beta<<<dim3(prep_blocks(d.N), d.n_images), CTL_THREADS, 0, s>>>(d, g, g_prev, st, ctl, beta, mode,
                                                                        (Totals*)part, count);
}
void launch_cg_direction(const DevData& d, bool again, const double* I, const double* g, const double* gfull,
                         CgImage* st, CgControl* ctl, double* beta, int* mode, double* dir, double* dots,
                         double* part, unsigned* count, cudaStream_t s) {
    k_cg_direction<<<dim3(prep_blocks(d.N), d.n_images), CTL_THREADS, 0, s>>>(
        d, again, I, g, gfull, st, ctl, beta, mode, dir, dots, (Totals*)part, count);
}
void launch_scalars_ls(const DevData& d, const ScalarArgs& sc, bool start, CgImage* st, CgControl* ctl,
                       const double* dots, double* alpha, const int* dstatus, unsigned long long h_inner,
                       cudaStream_t s) {
    const dim3 grid(d.n_images, sc.splits);
    launch_chained(start ? k_scalars_ls<true> : k_scalars_ls<false>, grid, CTL_THREADS, 0, s, d.chain, 1, d, sc, st, ctl,
                   dots, alpha, dstatus, h_inner);
}
void launch_cg_record(int NI, CgImage* st, CgControl* ctl, const double* scal, double* hist, const int* dstatus,
                      unsigned long long h_outer, cudaStream_t s) {
    k_cg_record<<<1, CTL_THREADS, 0, s>>>(NI, st, ctl, scal, hist, dstatus, h_outer);
}

}  // namespace msk
