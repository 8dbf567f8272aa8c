// paper_kernel.cu -- RSWR exactly as the paper states it (arXiv 2203.10477,
// Sec. 2.3-2.6, Sec. 3), on the GPU: adaptive spans chosen from the data.
//
// One span:
//   rswr_iface_kernel  (one CTA per interface i | i+1, Sec. 2.3-2.4): predicts
//       subdomains i and i+1 on the part of their windows that can reach the
//       overlap within the predictive span tau (zero input-flux guess at
//       their input boundaries), records the predicted output flux waveforms
//       both neighbours need for the update (Sec. 2.5), compares the two
//       predictions on the overlap and takes, as the pair's maximum span,
//       the largest number of leading steps over which they agree exactly at
//       some overlap point; the global span is the minimum over pairs (Sec. 3,
//       atomicMin).
//   paper_select_kernel: caps the span by the Waveform Time Span Theorem
//       (Sec. 2.4), records it, and copies the span's boundary samples for the
//       span kernel.
//   rswr_resolve_kernel (tiles of each subdomain's part of the combined
//       solution, Sec. 2.5): solves the subdomain again over the span with
//       its input flux set to the neighbour's predicted output flux
//       (Neumann ghost u_{L-1} = u_{L+1} - 2 dx g, u_{R+1} = u_{R-1} + 2 dx g)
//       and writes the points of Omega_i not covered by a window further left.
//   paper_advance_kernel: the next span starts span levels later, with the
//       predictive span ceil((1 + beta) * span) (Sec. 2.6).
// The run's progress lives on the device (PaperState), so the host queues the
// kernels of many spans and reads the state back once per batch.  The bulk of
// every span runs on the span kernel.
//
// FP32 runs whose windows fit a warp's registers (overlap + two predictive
// spans at most 32 P points) are one cooperative launch, paper_run_kernel; see
// there.

#include <algorithm>

#include "rswr_internal.h"
#include "resident.cuh"

namespace rswr {

namespace {

template <typename Real>
__device__ __forceinline__ void upd(int form, Real c2, Real k, Real uL, Real uC, Real uR, Real w, Real& un, Real& wn)
{
    if (form == kCanonical) {
        un = rfma(c2, radd(uL, uR), rfma(k, uC, -w));
        wn = uC;
    } else {
        const Real v = rfma(c2, radd(rsub(uL, uC), rsub(uR, uC)), w);
        un = radd(uC, v);
        wn = v;
    }
}

template <typename Real>
__device__ __forceinline__ Real dir_w(int form, Real f_old, Real f_new)
{
    return form == kCanonical ? f_old : rsub(f_new, f_old);
}

__device__ __forceinline__ int64_t win_l(int64_t i, int64_t nx, int64_t N, int64_t el)
{
    const int64_t b0 = i * nx / N;
    return b0 - el < 0 ? 0 : b0 - el;
}

__device__ __forceinline__ int64_t win_r(int64_t i, int64_t nx, int64_t N, int64_t er)
{
    const int64_t b1 = (i + 1) * nx / N;
    return b1 - 1 + er > nx - 1 ? nx - 1 : b1 - 1 + er;
}

// One step of a window [lo, hi] of subdomain `sub` held in shared memory.
// Edge rules: Dirichlet at the grid ends; at the subdomain's input boundaries
// either the zero-flux guess (g == nullptr) or the Neumann ghost from g[s];
// a cut that is not a subdomain boundary gets the mirror (its points are
// outside the part of the window that is kept).
template <typename Real>
__device__ void window_step(int form, Real c2, Real k, Real two_dx, int64_t nx, int64_t lo, int64_t hi, int64_t Lsub,
                            int64_t Rsub, const Real* gL, const Real* gR, int s, const Real* fA, const Real* fB,
                            int64_t n, const Real* u, const Real* w, Real* un, Real* wn)
{
    for (int64_t j = lo + threadIdx.x; j <= hi; j += blockDim.x) {
        const int64_t o = j - lo;
        if (j == 0) {
            const Real a0 = fA ? fA[n] : Real(0), a1 = fA ? fA[n + 1] : Real(0);
            un[o] = a1;
            wn[o] = dir_w<Real>(form, a0, a1);
            continue;
        }
        if (j == nx - 1) {
            const Real b0 = fB ? fB[n] : Real(0), b1 = fB ? fB[n + 1] : Real(0);
            un[o] = b1;
            wn[o] = dir_w<Real>(form, b0, b1);
            continue;
        }
        Real uL, uR;
        if (j == lo) {
            if (j == Lsub && gL) uL = rsub(u[o + 1], rmul(two_dx, gL[s]));
            else uL = u[o + 1];
        } else {
            uL = u[o - 1];
        }
        if (j == hi) {
            if (j == Rsub && gR) uR = radd(u[o - 1], rmul(two_dx, gR[s]));
            else uR = u[o - 1];
        } else {
            uR = u[o + 1];
        }
        upd<Real>(form, c2, k, uL, u[o], uR, w[o], un[o], wn[o]);
    }
}

template <typename Real>
__global__ void rswr_iface_kernel(const __grid_constant__ PaperParams<Real> p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t i = blockIdx.x;  // interface between subdomains i and i+1
    const int64_t nx = p.nx, N = p.N;
    const int64_t Li = win_l(i, nx, N, p.el), Ri = win_r(i, nx, N, p.er);
    const int64_t Ln = win_l(i + 1, nx, N, p.el), Rn = win_r(i + 1, nx, N, p.er);
    if (p.st && p.st->done) return;  // (every thread reads the same word)
    const int steps = p.st ? p.st->steps : p.steps;
    const int64_t n0 = p.st ? p.st->n0 : p.n0;
    const int64_t a0 = Ln - steps > Li ? Ln - steps : Li;  // prediction of i: [a0, Ri]
    const int64_t b1 = Ri + steps < Rn ? Ri + steps : Rn;  // prediction of i+1: [Ln, b1]
    const int64_t na = Ri - a0 + 1, nb = b1 - Ln + 1, nov = Ri - Ln + 1;
    Real* s = reinterpret_cast<Real*>(smem_raw);
    Real* ua = s;
    Real* wa = ua + na;
    Real* ua2 = wa + na;
    Real* wa2 = ua2 + na;
    Real* ub = wa2 + na;
    Real* wb = ub + nb;
    Real* ub2 = wb + nb;
    Real* wb2 = ub2 + nb;
    int* agree = reinterpret_cast<int*>(wb2 + nb);  // [nov]: leading steps of exact agreement, -1 = stopped
    for (int64_t o = threadIdx.x; o < na; o += blockDim.x) {
        ua[o] = p.u[a0 + o];
        wa[o] = p.w[a0 + o];
    }
    for (int64_t o = threadIdx.x; o < nb; o += blockDim.x) {
        ub[o] = p.u[Ln + o];
        wb[o] = p.w[Ln + o];
    }
    for (int64_t o = threadIdx.x; o < nov; o += blockDim.x) agree[o] = 0;
    __syncthreads();
    for (int st = 0; st < steps; ++st) {
        const int64_t n = n0 + st;
        // output flux waveforms at level n: subdomain i at Ln (for i+1), i+1 at Ri (for i)
        if (threadIdx.x == 0) {
            p.gL[(i + 1) * p.tau_stride + st] = rdiv(rsub(ua[Ln + 1 - a0], ua[Ln - 1 - a0]), p.two_dx);
            p.gR[i * p.tau_stride + st] = rdiv(rsub(ub[Ri + 1 - Ln], ub[Ri - 1 - Ln]), p.two_dx);
        }
        window_step<Real>(p.form, p.c2, p.k, p.two_dx, nx, a0, Ri, Li, Ri, nullptr, nullptr, st, p.fA, p.fB, n, ua, wa,
                          ua2, wa2);
        window_step<Real>(p.form, p.c2, p.k, p.two_dx, nx, Ln, b1, Ln, Rn, nullptr, nullptr, st, p.fA, p.fB, n, ub, wb,
                          ub2, wb2);
        __syncthreads();
        for (int64_t o = threadIdx.x; o < nov; o += blockDim.x) {
            if (agree[o] >= 0) {
                if (ua2[Ln + o - a0] == ub2[o]) agree[o] = st + 1;
                else agree[o] = -(agree[o] + 1);  // stop, remembering the count
            }
        }
        Real* t;
        t = ua; ua = ua2; ua2 = t;
        t = wa; wa = wa2; wa2 = t;
        t = ub; ub = ub2; ub2 = t;
        t = wb; wb = wb2; wb2 = t;
        __syncthreads();
    }
    // the pair's maximum span: largest agreement over the overlap
    __shared__ int best;
    if (threadIdx.x == 0) best = 0;
    __syncthreads();
    for (int64_t o = threadIdx.x; o < nov; o += blockDim.x) {
        const int a = agree[o] >= 0 ? agree[o] : -agree[o] - 1;
        atomicMax(&best, a);
    }
    __syncthreads();
    if (threadIdx.x == 0) atomicMin(p.span_min, best);
}

template <typename Real>
__global__ void rswr_resolve_kernel(const __grid_constant__ PaperParams<Real> p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t t = blockIdx.x;
    const int64_t i = p.tile_sub[t], c0 = p.tile_lo[t], c1 = p.tile_hi[t];  // owned [c0, c1) of subdomain i
    const int64_t nx = p.nx, N = p.N;
    const int64_t Li = win_l(i, nx, N, p.el), Ri = win_r(i, nx, N, p.er);
    const int span = p.st ? p.st->span : p.steps;
    const int64_t n0 = p.st ? p.st->n0 : p.n0;
    if (span <= 0) return;  // the run is complete (every thread reads the same word)
    const int64_t lo = c0 - span > Li ? c0 - span : Li;
    const int64_t hi = c1 - 1 + span < Ri ? c1 - 1 + span : Ri;
    const int64_t nw = hi - lo + 1;
    Real* s = reinterpret_cast<Real*>(smem_raw);
    Real* u = s;
    Real* w = u + nw;
    Real* u2 = w + nw;
    Real* w2 = u2 + nw;
    for (int64_t o = threadIdx.x; o < nw; o += blockDim.x) {
        u[o] = p.u[lo + o];
        w[o] = p.w[lo + o];
    }
    __syncthreads();
    const Real* gL = (i > 0 && Li > 0) ? p.gL + i * p.tau_stride : nullptr;
    const Real* gR = (i + 1 < N && Ri < nx - 1) ? p.gR + i * p.tau_stride : nullptr;
    for (int st = 0; st < span; ++st) {
        window_step<Real>(p.form, p.c2, p.k, p.two_dx, nx, lo, hi, Li, Ri, gL, gR, st, p.fA, p.fB, n0 + st, u, w,
                          u2, w2);
        __syncthreads();
        Real* tt;
        tt = u; u = u2; u2 = tt;
        tt = w; w = w2; w2 = tt;
    }
    for (int64_t j = c0 + threadIdx.x; j < c1; j += blockDim.x) {
        p.uo[j] = u[j - lo];
        p.wo[j] = w[j - lo];
    }
}

// The re-solved zones into the combined state: points [tile_lo, tile_hi) of
// every zone tile, from the scratch pair (plain arrays) to the state pair.
template <typename Real>
__global__ void paper_scatter_kernel(const Real* su, const Real* sw, Real* du, Real* dw, const int64_t* lo,
                                     const int64_t* hi, const PaperState* st)
{
    if (st && st->span <= 0) return;  // the run is complete: nothing was re-solved
    const int64_t t = blockIdx.x;
    for (int64_t j = lo[t] + threadIdx.x; j < hi[t]; j += blockDim.x) {
        du[j] = su[j];
        dw[j] = sw[j];
    }
}

// The select step's end (Sec. 2.4, Sec. 3): the global span is the minimum
// over the pairs (the word the interface CTAs lowered), at most the
// predictive steps and the Theorem's cap, at least 1; recorded as span number
// `count`.  Then the span kernel's boundary samples: levels n0 .. n0+nsamp-1
// of fA and fB (0 past level T) into fAs, fBs.
template <typename Real>
__global__ void paper_select_kernel(PaperState* st, const int* word, int cap, const Real* fA, const Real* fB,
                                    Real* fAs, Real* fBs, int nsamp, int64_t T, int64_t* spans, int64_t spans_cap)
{
    __shared__ int s_span;
    __shared__ int64_t s_n0;
    if (threadIdx.x == 0) {
        int span = 0;
        if (!st->done) {
            span = *word < st->steps ? *word : st->steps;
            if (span > cap) span = cap;
            if (span < 1) span = 1;
            if (spans && st->count < spans_cap) spans[st->count] = span;
        }
        st->span = span;
        s_span = span;
        s_n0 = st->n0;
    }
    __syncthreads();
    if (s_span <= 0) return;
    for (int i = threadIdx.x; i < nsamp; i += blockDim.x) {
        const int64_t lv = s_n0 + i;
        fAs[i] = (fA && lv <= T) ? fA[lv] : Real(0);
        fBs[i] = (fB && lv <= T) ? fB[lv] : Real(0);
    }
}

// The next span (Sec. 2.6): n0 advances by the span, the predictive span
// becomes ceil((1 + beta) span) (beta in thousandths, exact integer
// arithmetic) capped at tau_max, the predictive steps min(tau, T - n0).
__global__ void paper_advance_kernel(PaperState* st, int64_t T, int64_t beta_m, int64_t tau_max)
{
    if (st->done || st->span <= 0) return;
    const int64_t span = st->span;
    st->n0 += span;
    st->count += 1;
    int64_t tau = (span * (1000 + beta_m) + 999) / 1000;
    if (tau > tau_max) tau = tau_max;
    st->tau = (int32_t)tau;
    const int64_t rem = T - st->n0;
    st->steps = (int32_t)(tau < rem ? tau : rem);
    st->done = st->n0 >= T ? 1 : 0;
}

// ---- the whole run in one launch (FP32) ---------------------------------------

using span::kFull;

// u and w of one update (upd with the form known)
template <int FORM>
__device__ __forceinline__ void upd1(float c2, float k, float ul, float uc, float ur, float& u, float& w)
{
    if constexpr (FORM == kCanonical) {
        u = rfma(c2, radd(ul, ur), rfma(k, uc, -w));
        w = uc;
    } else {
        w = rfma(c2, radd(rsub(ul, uc), rsub(ur, uc)), w);
        u = radd(uc, w);
    }
}

// One step of a window whose ends are registers el / er (-1: not on this
// lane): their outer neighbour is the mirror, or the Neumann ghost (gl, gr: 2 dx g).
template <int FORM, int P>
__device__ __forceinline__ void window_step1(float (&u)[P], float (&w)[P], float c2, float k, int el, int er,
                                             bool ghost_l, float gl, bool ghost_r, float gr)
{
    float ul = __shfl_up_sync(kFull, u[P - 1], 1);
    const float rgt = __shfl_down_sync(kFull, u[0], 1);
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const float uc = u[i], ur = i < P - 1 ? u[i + 1] : rgt;
        const float out_l = ghost_l ? rsub(ur, gl) : ur, out_r = ghost_r ? radd(ul, gr) : ul;
        upd1<FORM>(c2, k, el == i ? out_l : ul, uc, er == i ? out_r : ur, u[i], w[i]);
        ul = uc;
    }
}

template <int P>
__device__ __forceinline__ void warp_set(float (&u)[P], float (&w)[P], int r, float x, float y)
{
#pragma unroll
    for (int i = 0; i < P; ++i)
        if (r == i) {
            u[i] = x;
            w[i] = y;
        }
}

// Leading steps on which the two predictions agree at some overlap point still
// `alive` (a bit per register): false once there is none.
template <int P>
__device__ __forceinline__ bool agree(const float (&ua)[P], const float (&ub)[P], uint32_t& alive)
{
    uint32_t same = 0;
#pragma unroll
    for (int q = 0; q < P; ++q) same |= ua[q] == ub[q] ? 1u << q : 0u;
    alive &= same;
    return __any_sync(kFull, alive != 0);
}

// Predict + select of interface i (Sec. 2.3, 2.4): both predictions in one
// register layout, so that the overlap is compared point by point.  Returns the
// pair's span; rows: room for 2 * steps values.
template <int FORM, int P>
__device__ int warp_iface(const PaperParams<float>& p, const float* gu, const float* gw, int64_t i, int steps,
                          int64_t n0, float* rows, int lane)
{
    const int64_t nx = p.nx, N = p.N;
    const int64_t Li = win_l(i, nx, N, p.el), Ri = win_r(i, nx, N, p.er);
    const int64_t Ln = win_l(i + 1, nx, N, p.el), Rn = win_r(i + 1, nx, N, p.er);
    const int64_t a0 = Ln - steps > Li ? Ln - steps : Li;  // prediction of i: [a0, Ri]
    const int64_t b1 = Ri + steps < Rn ? Ri + steps : Rn;  // prediction of i+1: [Ln, b1]
    // neither prediction reaches the far end of its subdomain: its cut end needs no
    // rule (what comes from there arrives after the last step), and the window
    // starts so that Ln is a lane's first register
    const bool cut = Ln - steps >= Li + P && Ri + steps < Rn;
    const int64_t lo = cut ? Ln - (Ln - a0 + P - 1) / P * P : a0;
    const int p_l = (int)(Ln - lo), p_r = (int)(Ri - lo), p_e = (int)(b1 - lo);
    auto reg = [&](int pos) { return lane == pos / P ? pos % P : -1; };
    float ua[P], wa[P], ub[P], wb[P];
    uint32_t alive = 0;
#pragma unroll
    for (int q = 0; q < P; ++q) {
        const int64_t j = lo + lane * P + q;
        const bool in = j <= b1;
        ua[q] = ub[q] = in ? __ldcg(gu + j) : 0.f;
        wa[q] = wb[q] = in ? __ldcg(gw + j) : 0.f;
        if (j >= Ln && j <= Ri) alive |= 1u << q;
    }
    const int r_l = reg(p_l), r_r = reg(p_r);
    int best = 0, done = 0;
    if (cut) {
        for (int st = 0; st < steps; ++st) {
            float al = __shfl_up_sync(kFull, ua[P - 1], 1), bl = __shfl_up_sync(kFull, ub[P - 1], 1);
            const float ar = __shfl_down_sync(kFull, ua[0], 1), br = __shfl_down_sync(kFull, ub[0], 1);
            const float fl = rsub(ua[1], al);  // (at Ln; times 2 dx) output flux of i, level n
            bl = r_l == 0 ? ub[1] : bl;        // zero flux into i + 1
            float fm = 0.f, fp = 0.f;
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const float ac = ua[q], bc = ub[q];
                const float an = q < P - 1 ? ua[q + 1] : ar, bn = q < P - 1 ? ub[q + 1] : br;
                const bool e = r_r == q;
                fm = e ? bl : fm;
                fp = e ? bn : fp;
                upd1<FORM>(p.c2, p.k, al, ac, e ? al : an, ua[q], wa[q]);  // zero flux into i at Ri
                upd1<FORM>(p.c2, p.k, bl, bc, bn, ub[q], wb[q]);
                al = ac;
                bl = bc;
            }
            if (r_l >= 0) rows[2 * st] = fl;
            if (r_r >= 0) rows[2 * st + 1] = rsub(fp, fm);  // output flux of i + 1 at Ri
            done = st + 1;
            if (!agree<P>(ua, ub, alive)) break;  // (no later step is selected: its fluxes are not needed)
            best = st + 1;
        }
    } else {
        const int r_0 = reg(0), r_e = reg(p_e);
        const bool dir_a = a0 == 0, dir_b = b1 == nx - 1;  // Dirichlet nodes
        auto flux = [&](const float(&u)[P], int r, float* out) {
            const float l = __shfl_up_sync(kFull, u[P - 1], 1), rr = __shfl_down_sync(kFull, u[0], 1);
            float d = 0.f;
#pragma unroll
            for (int q = 0; q < P; ++q)
                if (r == q) d = rsub(q < P - 1 ? u[q + 1] : rr, q > 0 ? u[q - 1] : l);
            if (r >= 0) *out = d;
        };
        for (int st = 0; st < steps; ++st) {
            const int64_t n = n0 + st;
            flux(ua, r_l, rows + 2 * st);
            flux(ub, r_r, rows + 2 * st + 1);
            window_step1<FORM, P>(ua, wa, p.c2, p.k, r_0, r_r, false, 0.f, false, 0.f);
            window_step1<FORM, P>(ub, wb, p.c2, p.k, r_l, r_e, false, 0.f, false, 0.f);
            if (dir_a) {
                const float x0 = p.fA ? p.fA[n] : 0.f, x1 = p.fA ? p.fA[n + 1] : 0.f;
                warp_set<P>(ua, wa, r_0, x1, dir_w<float>(FORM, x0, x1));
            }
            if (dir_b) {
                const float x0 = p.fB ? p.fB[n] : 0.f, x1 = p.fB ? p.fB[n + 1] : 0.f;
                warp_set<P>(ub, wb, r_e, x1, dir_w<float>(FORM, x0, x1));
            }
            done = st + 1;
            if (!agree<P>(ua, ub, alive)) break;
            best = st + 1;
        }
    }
    __syncwarp();
    for (int st = lane; st < done; st += 32) {
        p.gL[(i + 1) * p.tau_stride + st] = rdiv(rows[2 * st], p.two_dx);
        p.gR[i * p.tau_stride + st] = rdiv(rows[2 * st + 1], p.two_dx);
    }
    __syncwarp();
    return best;
}

// Update of a piece near an input boundary of a subdomain (Sec. 2.5), or near an
// end of the grid (sub < 0); of two short ones with `pair`, half a warp each
// (what the shuffles carry between the halves arrives after the span, as from any
// cut end).  rows: room for 4 * span values.
template <int FORM, int P>
__device__ void warp_resolve(const PaperParams<float>& p, const float* gu, const float* gw, float* du, float* dw,
                             const PaperPiece* pieces, bool pair, int span, int64_t n0, float* rows, int warp_lane)
{
    const int lanes = pair ? 16 : 32, half = pair ? warp_lane >> 4 : 0, lane = warp_lane & (lanes - 1);
    const PaperPiece piece = pieces[half];
    const int64_t i = piece.sub, c0 = piece.lo, c1 = c0 + piece.len;
    rows += half * 2 * span;
    const int64_t nx = p.nx, N = p.N;
    const int64_t Li = i < 0 ? 0 : win_l(i, nx, N, p.el), Ri = i < 0 ? nx - 1 : win_r(i, nx, N, p.er);
    const int64_t lo = c0 - span > Li ? c0 - span : Li;
    const int64_t hi = c1 - 1 + span < Ri ? c1 - 1 + span : Ri;
    auto reg = [&](int64_t pos) { return lane == pos / P ? (int)(pos % P) : -1; };
    float u[P], w[P];
#pragma unroll
    for (int q = 0; q < P; ++q) {
        const int64_t j = lo + lane * P + q;
        u[q] = j <= hi ? __ldcg(gu + j) : 0.f;
        w[q] = j <= hi ? __ldcg(gw + j) : 0.f;
    }
    const bool dir_a = lo == 0, dir_b = hi == nx - 1;
    const bool gl = i > 0 && Li > 0 && lo == Li, gr = i >= 0 && i + 1 < N && Ri < nx - 1 && hi == Ri;
    // per step: what the end's rule needs (2 dx g, or the node's next sample)
    for (int st = lane; st < span; st += lanes) {
        float a = 0.f, b = 0.f;
        if (dir_a) a = p.fA ? p.fA[n0 + st + 1] : 0.f;
        else if (gl) a = rmul(p.two_dx, __ldcg(p.gL + i * p.tau_stride + st));
        if (dir_b) b = p.fB ? p.fB[n0 + st + 1] : 0.f;
        else if (gr) b = rmul(p.two_dx, __ldcg(p.gR + i * p.tau_stride + st));
        rows[2 * st] = a;
        rows[2 * st + 1] = b;
    }
    __syncwarp();
    const int r_l = reg(0), r_r = reg(hi - lo);
    float fa = dir_a && p.fA ? p.fA[n0] : 0.f, fb = dir_b && p.fB ? p.fB[n0] : 0.f;
    for (int st = 0; st < span; ++st) {
        const float a = rows[2 * st], b = rows[2 * st + 1];
        window_step1<FORM, P>(u, w, p.c2, p.k, r_l, r_r, gl, a, gr, b);
        if (dir_a) {
            warp_set<P>(u, w, r_l, a, dir_w<float>(FORM, fa, a));
            fa = a;
        }
        if (dir_b) {
            warp_set<P>(u, w, r_r, b, dir_w<float>(FORM, fb, b));
            fb = b;
        }
    }
#pragma unroll
    for (int q = 0; q < P; ++q) {
        const int64_t j = lo + lane * P + q;
        if (j >= c0 && j < c1) {
            du[j] = u[q];
            dw[j] = w[q];
        }
    }
    __syncwarp();
}

// Window points [0, 32 P) of one component from src (16-byte aligned; points j0 +
// position, zero from nx on) through shared memory: whole lines on the way in.
template <int P>
__device__ __forceinline__ void warp_load(const float* src, float (&v)[P], float* sm, int lane, int64_t j0, int64_t nx)
{
    float4 x[P / 4];
#pragma unroll
    for (int k = 0; k < P / 4; ++k) {
        const int64_t at = 4 * (lane + 32 * k);
        const float* s = src + at;
        if (j0 + at + 4 <= nx) {
            x[k] = __ldcg(reinterpret_cast<const float4*>(s));
        } else {
            const int64_t left = nx - j0 - at;
            x[k].x = left > 0 ? __ldcg(s) : 0.f;
            x[k].y = left > 1 ? __ldcg(s + 1) : 0.f;
            x[k].z = left > 2 ? __ldcg(s + 2) : 0.f;
            x[k].w = 0.f;
        }
    }
#pragma unroll
    for (int k = 0; k < P / 4; ++k)
        *reinterpret_cast<float4*>(sm + resident::unit_place<float>(lane + 32 * k)) = x[k];
    __syncwarp();
    resident::get_units<float, P>(sm, v, lane);
    __syncwarp();
}

// Update of a piece [c0, c1) that no input boundary and no grid end reaches
// within a span: the bare stencil.
template <int FORM, int P>
__device__ __forceinline__ void warp_bulk(const PaperParams<float>& p, const float* gu, const float* gw, float* du,
                                          float* dw, int64_t c0, int64_t c1, int cap, int span, float* sm, int lane)
{
    const int64_t lo = (c0 - cap) & ~(int64_t)3;
    float u[P], w[P];
    warp_load<P>(gu + lo, u, sm, lane, lo, p.nx);
    warp_load<P>(gw + lo, w, sm, lane, lo, p.nx);
    resident::Stream<float> none;
    resident::run_steps<float, FORM, P, resident::kPlain>(
        u, w, p.c2, p.k, 0, span, false, none, [](const float(&)[P], float, float, int) {},
        [](float(&)[P], float(&)[P], const float(&)[P], int) {});
    resident::store_owned<float, P>(du + lo, u, sm, lane, (int)(c0 - lo), (int)(c1 - c0));
    resident::store_owned<float, P>(dw + lo, w, sm, lane, (int)(c0 - lo), (int)(c1 - c0));
}

constexpr int kRunWarps = 4;

// All spans of a run (a cooperative launch).  One warp per interface predicts
// and selects; behind a grid barrier every warp knows the global span; one
// warp per piece then updates the grid from one state buffer to the other --
// pieces near input boundaries with the paper's rule in windows of 32 PI
// points, all others with the bare stencil in windows of 32 PB -- and behind
// another barrier the next span starts.  Last-span pieces go straight to the
// caller's arrays.
//
// What bounds it: at 4,194,304 points (256 subdomains, overlap 64, spans of 34) a
// span takes 5 us for the predictions (a chain of 38 steps of 260 clocks), 2 x 2
// us of barriers and 26 us of updates, two rounds of windows on every warp slot,
// bound by instruction issue (the state stays in L2).  500 steps took 2064 us
// launched span by span -- shared-memory windows with a block barrier per step
// at the interfaces, two passes of the span kernel, eight launches a span -- and
// take 800 us here.  More CTAs per SM with fewer registers spill (940 us).
template <int FORM, int PI, int PB>
__global__ void __launch_bounds__(32 * kRunWarps, 4) paper_run_kernel(const __grid_constant__ PaperParams<float> p,
                                                                      const __grid_constant__ PaperRun q)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_ok;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* const sm = reinterpret_cast<float*>(smem_raw) + (size_t)warp * q.warp_values;
    // (neighbouring warp numbers in different CTAs: few interfaces spread over all SMs)
    const int64_t gw = (int64_t)warp * gridDim.x + blockIdx.x, nw = (int64_t)gridDim.x * kRunWarps;
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    unsigned target = 0;
    int barriers = 0;
    auto barrier = [&](int count, int side) {
        target += gridDim.x;
        __syncthreads();
        const int no = barriers++;
        if (threadIdx.x == 0) {
            __threadfence();
            if ((int)blockIdx.x != q.inject_cta || no < q.inject_barrier) atomicAdd(q.arrived, 1u);
            long long t0 = 0;
            int ok = 1;
            unsigned spins = 0;
            while ((unsigned)ld_acquire(reinterpret_cast<const int*>(q.arrived)) - target > 0x7fffffffu) {
                if ((++spins & 63u) != 0u) continue;
                const long long now = global_ns();
                if (t0 == 0) t0 = now;
                if (*(volatile int*)&q.err->code != 0) ok = 0;
                else if (now - t0 > q.wait_ns) {
                    latch_error(q.err, kDevTimeoutFlag, (int)blockIdx.x, count, side);
                    ok = 0;
                }
                if (!ok) break;
            }
            s_ok = ok;
        }
        __syncthreads();
        return s_ok != 0;
    };
    int64_t n0 = 0;
    int steps = q.steps, count = 0;
    while (n0 < q.T) {
        const float* const gu = p.u + (count & 1) * q.swap_u;
        const float* const gv = p.w + (count & 1) * q.swap_w;
        int* const word = p.span_min + (count & 1);  // (the other one is for the next span)
        for (int64_t i = gw; i < p.N - 1; i += nw) {
            const int best = warp_iface<FORM, PI>(p, gu, gv, i, steps, n0, sm, lane);
            if (lane == 0) atomicMin(word, best);
        }
        if (!barrier(count, 1)) return;
        const int w0 = *(volatile int*)word;
        int span = w0 < steps ? w0 : steps;
        if (span > q.cap) span = q.cap;
        if (span < 1) span = 1;
        const bool last = n0 + span >= q.T;
        if (first) {
            p.span_min[(count + 1) & 1] = 0x7f7f7f7f;  // (last read before the previous barrier)
            if (q.spans && count < q.spans_cap) q.spans[count] = span;
        }
        float* const du = last ? p.uo : const_cast<float*>(p.u) + (~count & 1) * q.swap_u;
        float* const dw = last ? p.wo : const_cast<float*>(p.w) + (~count & 1) * q.swap_w;
        for (int64_t t = gw; t < q.npiece - q.npair; t += nw) {
            const bool pair = t < q.npair;
            const PaperPiece* const c = q.pieces + (pair ? 2 * t : t + q.npair);
            if (c->sub == kPieceBulk)
                warp_bulk<FORM, PB>(p, gu, gv, du, dw, c->lo, c->lo + c->len, q.cap, span, sm, lane);
            else
                warp_resolve<FORM, PI>(p, gu, gv, du, dw, c, pair, span, n0, sm, lane);
        }
        n0 += span;
        ++count;
        int64_t tau = ((int64_t)span * (1000 + q.beta_m) + 999) / 1000;
        if (tau > p.tau_stride) tau = p.tau_stride;
        steps = (int)(tau < q.T - n0 ? tau : q.T - n0);
        if (!last && !barrier(count, 2)) return;
    }
    if (first) {
        q.st->n0 = n0;
        q.st->count = count;
        q.st->done = 1;
    }
}

}  // namespace

cudaError_t paper_select_launch(int dtype, PaperState* st, const int* word, int cap, const void* fA, const void* fB,
                                void* fAs, void* fBs, int nsamp, int64_t T, int64_t* spans, int64_t spans_cap,
                                cudaStream_t s)
{
    if (dtype == kF64)
        paper_select_kernel<double><<<1, 256, 0, s>>>(st, word, cap, static_cast<const double*>(fA),
                                                      static_cast<const double*>(fB), static_cast<double*>(fAs),
                                                      static_cast<double*>(fBs), nsamp, T, spans, spans_cap);
    else
        paper_select_kernel<float><<<1, 256, 0, s>>>(st, word, cap, static_cast<const float*>(fA),
                                                     static_cast<const float*>(fB), static_cast<float*>(fAs),
                                                     static_cast<float*>(fBs), nsamp, T, spans, spans_cap);
    return cudaGetLastError();
}

cudaError_t paper_advance_launch(PaperState* st, int64_t T, int64_t beta_m, int64_t tau_max, cudaStream_t s)
{
    paper_advance_kernel<<<1, 1, 0, s>>>(st, T, beta_m, tau_max);
    return cudaGetLastError();
}

cudaError_t paper_scatter_launch(int dtype, const void* su, const void* sw, void* du, void* dw, const int64_t* lo,
                                 const int64_t* hi, int ntiles, const PaperState* st, cudaStream_t s)
{
    if (ntiles <= 0) return cudaSuccess;
    if (dtype == kF64)
        paper_scatter_kernel<double><<<ntiles, 128, 0, s>>>(static_cast<const double*>(su),
                                                            static_cast<const double*>(sw), static_cast<double*>(du),
                                                            static_cast<double*>(dw), lo, hi, st);
    else
        paper_scatter_kernel<float><<<ntiles, 128, 0, s>>>(static_cast<const float*>(su), static_cast<const float*>(sw),
                                                           static_cast<float*>(du), static_cast<float*>(dw), lo, hi, st);
    return cudaGetLastError();
}

cudaError_t paper_iface_launch(int dtype, const void* params, int n_iface, size_t smem, cudaStream_t s)
{
    if (n_iface <= 0) return cudaSuccess;
    void* args[] = {const_cast<void*>(params)};
    const void* fn = dtype == kF64 ? reinterpret_cast<const void*>(&rswr_iface_kernel<double>)
                                   : reinterpret_cast<const void*>(&rswr_iface_kernel<float>);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // (measured: 256 threads per interface 51 us per span on the c2 grid, 32 threads 62 us)
    return cudaLaunchKernel(fn, dim3(n_iface), dim3(256), args, smem, s);
}

cudaError_t paper_resolve_launch(int dtype, const void* params, int ntiles, size_t smem, cudaStream_t s)
{
    void* args[] = {const_cast<void*>(params)};
    const void* fn = dtype == kF64 ? reinterpret_cast<const void*>(&rswr_resolve_kernel<double>)
                                   : reinterpret_cast<const void*>(&rswr_resolve_kernel<float>);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // zone tiles are a few span lengths wide: two warps per tile (measured on
    // the c2 grid: 34 us per span against 41 us with 256 threads)
    return cudaLaunchKernel(fn, dim3(ntiles), dim3(64), args, smem, s);
}

namespace {

struct RunEntry {
    int form, PI, PB;
    const void* fn;
};

#define RSWR_PAPER_RUN(FORM, PI, PB) {FORM, PI, PB, reinterpret_cast<const void*>(&paper_run_kernel<FORM, PI, PB>)}
const RunEntry kRuns[] = {
    RSWR_PAPER_RUN(kIncrement, 8, 32),  RSWR_PAPER_RUN(kIncrement, 8, 8),  RSWR_PAPER_RUN(kIncrement, 16, 32),
    RSWR_PAPER_RUN(kCanonical, 8, 32),  RSWR_PAPER_RUN(kCanonical, 8, 8),  RSWR_PAPER_RUN(kCanonical, 16, 32),
};

size_t run_smem(const PaperRunChoice& c) { return sizeof(float) * kRunWarps * (size_t)c.warp_values; }

}  // namespace

bool paper_run_choose(int form, int64_t nx, int64_t ov, int64_t cap, int64_t tau_max, int num_sms, PaperRunChoice* out)
{
    // a prediction window (its start rounded down by up to P - 1 points) and a
    // re-solve window that keeps 64 points beside its halos fit 32 PI points
    int PI = 0;
    for (int P = 8; P <= 16 && !PI; P *= 2)
        if (ov + 2 * tau_max + P <= 32 * P && 2 * cap + 64 <= 32 * P) PI = P;
    if (!PI) return false;
    // Windows of 256 points for the bulk while every scheduler has at most two of
    // them (a chain of spans: fewer points per lane, shorter steps), of 1024
    // beyond (twice the cap of a window is recomputed)
    const int64_t small = 32 * 8 - 2 * cap - 4;
    const int PB = PI == 8 && nx <= small * 8 * num_sms ? 8 : 32;
    for (int v = 0; v < (int)(sizeof(kRuns) / sizeof(kRuns[0])); ++v)
        if (kRuns[v].form == form && kRuns[v].PI == PI && kRuns[v].PB == PB) {
            out->v = v;
            out->edge = 32 * PI - 2 * cap;
            out->half = 16 * PI - 2 * cap;
            out->bulk = 32 * PB - 2 * cap - 4;
            const int64_t need = std::max<int64_t>(4 * tau_max, 32 * PB + 32);  // (a moved window: 3 points more)
            out->warp_values = (int)((need + 31) / 32 * 32);
            return true;
        }
    return false;
}

cudaError_t paper_run_launch(const PaperRunChoice& c, const PaperParams<float>& p, const PaperRun& q, int num_sms,
                             cudaStream_t s)
{
    const void* fn = kRuns[c.v].fn;
    const size_t smem = run_smem(c);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * kRunWarps, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int64_t work = std::max<int64_t>(q.npiece - q.npair, p.N - 1);
    const int64_t want = (work + kRunWarps - 1) / kRunWarps;
    const int grid = (int)std::min<int64_t>(want, (int64_t)per_sm * num_sms);
    void* args[] = {const_cast<PaperParams<float>*>(&p), const_cast<PaperRun*>(&q)};
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)grid), dim3(32 * kRunWarps), args, smem, s);
}

}  // namespace rswr
