// resident.cuh -- resident warp windows: the whole run of a grid that fits on
// the chip in one cooperative launch, sm_103a.
//
// Every warp owns a contiguous piece of one problem and keeps the piece plus a
// halo of H points on each side in registers (P consecutive points per lane)
// for the whole run.  A chunk of up to H steps runs with shuffles only; the two
// window ends take a guess whose influence travels one point per step, so the
// owned points stay exact for H steps (the Waveform Time Span Theorem,
// Sec. 2.4, with the warp's window as the subdomain and 2H shared points).
// Then the H owned points next to each end, both components, go to the
// neighbouring warps, whose halos they are: through shared memory with an
// mbarrier per warp and side inside a CTA, through L2 across CTAs.
//
// What bounds it: small grids are a chain of T steps, each a shuffle and four
// dependent FP32 operations (two FP64 ones, at 64 cycles of a scheduler's pipe
// per warp instruction), plus one exchange per chunk.  So
//   * no warp ever waits for a CTA-wide barrier: a warp waits for its two
//     neighbours only, and runs ahead of the others by up to one chunk;
//   * a grid of up to 16 CTAs is one thread-block cluster: an exchange across
//     CTAs is a few st.async into the neighbour's shared memory, counted by an
//     mbarrier there;
//   * on a larger grid an exchange across CTAs is one 16-byte store per point that carries its
//     own launch and chunk number (16-byte accesses are single-copy atomic), so a reader
//     polls the data itself and no flag follows it;
//   * a window is placed so that a Dirichlet node is the neighbour of its
//     outermost point (one select a step) and a point source sits on a lane's
//     first register (two); other cases take compares per register;
//   * a probe's window is placed so that its point is a lane's first or last
//     register; the lane drops the value into a shared buffer every step, and the
//     warp turns 32 levels into one coalesced store (elsewhere: rows of all the
//     lane's registers; more than two probes: a record per lane).
// The initial state comes straight from the caller's arrays and the final state
// goes straight to them, unless it would land on what the run still reads.
//
// Measured, whole runs, against the ticketed kernels (the last: against one CTA
// per resident tile): 1001 FP64 points, 2000 steps 4636 -> 694 us; 8001 FP32, 2000
// steps 1890 -> 198; 60001 FP32, 5000 steps 4388 -> 604; 200003 FP64, 512 steps
// 1635 -> 740; 2^20 FP32, 2048 steps 839 -> 402.

#pragma once

#include "rswr_internal.h"
#include "span_common.cuh"

namespace rswr {
namespace resident {

using span::kFull;

constexpr int kRing = 16;      // levels of a probe row buffer
constexpr int kFastRing = 32;  // levels of a buffer of probes on end registers

// ---- 16-byte single-copy-atomic accesses at gpu scope ------------------------
__device__ __forceinline__ void st_pair(ulonglong2* p, unsigned long long lo, unsigned long long hi)
{
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
                 "l"(lo), "l"(hi)
                 : "memory");
}

__device__ __forceinline__ void ld_pair(const ulonglong2* p, unsigned long long& lo, unsigned long long& hi)
{
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p)
                 : "memory");
}

// Words per exchanged point in a global slot: FP32 {u, w | chunk}, FP64 {u | chunk}, {w | chunk}.
template <typename Real>
constexpr int slot_words = sizeof(Real) == 4 ? 1 : 2;

// Stores of one lane without a branch (a branch that one lane takes costs a
// reconvergence, some 100 clocks a step on a lone warp).
__device__ __forceinline__ void st_shared_if(bool on, const float* d, float a, float b)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.shared.v2.f32 [%1], {%2, %3};\n\t}" ::"r"((uint32_t)on),
                 "r"(smem_addr(d)), "f"(a), "f"(b)
                 : "memory");
}
__device__ __forceinline__ void st_shared_if(bool on, const double* d, double a, double b)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.shared.v2.f64 [%1], {%2, %3};\n\t}" ::"r"((uint32_t)on),
                 "r"(smem_addr(d)), "d"(a), "d"(b)
                 : "memory");
}

__device__ __forceinline__ void st_shared_if16(bool on, const float* d, const float* x)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t"
                 "@p st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n\t"
                 "@p st.shared.v4.f32 [%1 + 16], {%6, %7, %8, %9};\n\t"
                 "@p st.shared.v4.f32 [%1 + 32], {%10, %11, %12, %13};\n\t"
                 "@p st.shared.v4.f32 [%1 + 48], {%14, %15, %16, %17};\n\t}" ::"r"((uint32_t)on),
                 "r"(smem_addr(d)), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "f"(x[4]), "f"(x[5]), "f"(x[6]),
                 "f"(x[7]), "f"(x[8]), "f"(x[9]), "f"(x[10]), "f"(x[11]), "f"(x[12]), "f"(x[13]), "f"(x[14]),
                 "f"(x[15])
                 : "memory");
}

__device__ __forceinline__ void st_global_if(bool on, float* d, float a)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.global.f32 [%1], %2;\n\t}" ::"r"((uint32_t)on), "l"(d),
                 "f"(a)
                 : "memory");
}
__device__ __forceinline__ void st_global_if(bool on, double* d, double a)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.global.f64 [%1], %2;\n\t}" ::"r"((uint32_t)on), "l"(d),
                 "d"(a)
                 : "memory");
}

// Warps of a CTA at most: 16 (one CTA then holds an SM's whole register file),
// 8 where a lane's points fill more than 64 registers.
template <typename Real>
__host__ __device__ constexpr int max_warps(int P) { return P * sizeof(Real) > 64 ? 8 : 16; }

// Lanes of a probe row: the probed point's lane and a neighbour of it.
template <typename Real>
__host__ __device__ constexpr int kRowLanes(int P) { return P == 1 ? 3 : 2; }

// Shared memory of one warp, in values: the window as the last two chunks left
// it [parity][component][32 P], inbox [side][parity][component][H], probe rows.
template <typename Real>
__host__ __device__ inline size_t warp_values(int H, int P, int probe_rows)
{
    size_t n = (size_t)128 * P + 8 * H;
    const int row = kRing * kRowLanes<Real>(P) * P;
    n += (size_t)probe_rows * (row > 2 * kFastRing ? row : 2 * kFastRing);
    return (n + 3) / 4 * 4;
}

// A probe on one of a lane's own points, where a warp has more than two.
template <typename Real>
struct LaneProbe {
    Real* out;
    int64_t stride;
    Real scale;
    int32_t nmax;
    int32_t code;  // 2 (register + 1) + kind; a node beside the window: register -1 or P; -1: none
};

// Records of every lane that the row buffers of two probes hold.
template <typename Real>
__host__ __device__ constexpr int max_rounds(int P)
{
    const int row = kRing * kRowLanes<Real>(P) * P;
    return 2 * (row > 2 * kFastRing ? row : 2 * kFastRing) * (int)sizeof(Real) / (32 * (int)sizeof(LaneProbe<Real>));
}

// The samples of a warp's one special point (a node's value, a source's
// addend), held across the warp: cur is the coming step's; lane l has the sample
// of step 32 m + 1 + l in c0 and of the 32 steps after in c1, which is loaded 32
// steps before it is needed.
template <typename Real>
struct Stream {
    const Real* p;  // this lane's next sample to load
    int64_t step;   // 32 samples on
    int level, top; // its level, the last level there is
    Real cur, c0, c1;
    __device__ __forceinline__ Real load()
    {
        const Real v = (p != nullptr && level <= top) ? *p : Real(0);
        if (p != nullptr) p += step;
        level += 32;
        return v;
    }
    // the sample of step 0 is the one of level `first`
    __device__ __forceinline__ void open(const Real* samples, int64_t stride, int first, int lane, int last)
    {
        cur = (samples && first <= last) ? samples[first * stride] : Real(0);
        level = first + 1 + lane;
        p = samples ? samples + level * stride : nullptr;
        step = 32 * stride;
        top = last;
        c0 = load();
        c1 = load();
    }
    __device__ __forceinline__ void next()
    {
        c0 = c1;
        c1 = load();
    }
    // the sample of the step after step n
    __device__ __forceinline__ Real after(int n) const { return __shfl_sync(kFull, c0, n & 31); }
};

// What a warp's window holds besides plain points.  A grid's end window is
// placed so that the Dirichlet node is the neighbour of its outermost point:
// the node is then not a point of the window, its samples take the place of
// the shuffle from outside (one select a step).
enum : int {
    kPlain = 0,
    kNodeLeft = 1,   // j = 0 next to lane 0's first register
    kNodeRight = 2,  // j = nx - 1 next to lane 31's last register
    kSource = 3,     // one point source, on the first register of a lane
    kAny = 4         // nodes inside the window, several sources: patched after the step
};

// `steps` leapfrog steps of the window from level lv on.  mine: this lane's
// shuffle (node) or register (source) takes the stream's samples.
// rec(u, lft, rgt, s) sees level lv + s before it is advanced (it must not shuffle
// inside a divergent branch); patch(u, w, u_old, s)
// patches the special points after the step (kAny).
template <typename Real, int FORM, int P, int SPEC, typename Rec, typename Patch>
__device__ __forceinline__ void run_steps(Real (&u)[P], Real (&w)[P], Real c2, Real k, int lv, int steps, bool mine,
                                          Stream<Real>& st, Rec&& rec, Patch&& patch)
{
    // (a lone warp pays for every branch; FP64 is bound by its pipe)
    constexpr int kUnroll = sizeof(Real) == 8 || SPEC == kAny ? 1 : (P <= 8 ? 4 : (P <= 16 ? 2 : 1));
    constexpr bool kStream = SPEC == kNodeLeft || SPEC == kNodeRight || SPEC == kSource;
    Real lft = __shfl_up_sync(kFull, u[P - 1], 1);
    Real rgt = __shfl_down_sync(kFull, u[0], 1);
    auto take = [&]() {
        if constexpr (SPEC == kNodeLeft) lft = mine ? st.cur : lft;
        if constexpr (SPEC == kNodeRight) rgt = mine ? st.cur : rgt;
    };
    take();
    for (int s0 = 0; s0 < steps;) {
        int s1 = steps;
        if constexpr (kStream) {
            const int left = 32 - ((lv + s0) & 31);  // samples in c0
            s1 = s0 + left < steps ? s0 + left : steps;
        }
#pragma unroll kUnroll
        for (int s = s0; s < s1; ++s) {
            const Real l_old = lft, r_old = rgt;
            Real nxt = Real(0);
            if constexpr (kStream) nxt = st.after(lv + s);  // (in time for the end of this step)
            if constexpr (SPEC == kAny) {
                rec(u, l_old, r_old, s);
                Real uo[P];  // level n
#pragma unroll
                for (int i = 0; i < P; ++i) uo[i] = u[i];
                span::leap_step<Real, FORM, P>(u, w, lft, rgt, c2, k);
                patch(u, w, uo, s);
                lft = __shfl_up_sync(kFull, u[P - 1], 1);
                rgt = __shfl_down_sync(kFull, u[0], 1);
                continue;
            }
            Real n0 = Real(0), v0 = Real(0);  // the first point's new values
            auto add_source = [&]() {
                if constexpr (SPEC == kSource) {
                    if constexpr (FORM == kIncrement) {
                        const Real vs = radd(v0, st.cur);
                        v0 = mine ? vs : v0;
                        n0 = mine ? radd(u[0], vs) : n0;
                    } else {
                        n0 = mine ? radd(n0, st.cur) : n0;
                    }
                }
            };
            if constexpr (P == 1) {
                if constexpr (FORM == kIncrement) {
                    v0 = rfma(c2, rsub(rsub(rgt, u[0]), rsub(u[0], lft)), w[0]);
                    n0 = radd(u[0], v0);
                } else {
                    n0 = rfma(c2, radd(lft, rgt), rfma(k, u[0], -w[0]));
                    v0 = u[0];
                }
                add_source();
                lft = __shfl_up_sync(kFull, n0, 1);
                rgt = __shfl_down_sync(kFull, n0, 1);
                rec(u, l_old, r_old, s);
                u[0] = n0;
                w[0] = v0;
            } else if constexpr (FORM == kIncrement) {
                // the two end points first, so that the shuffles of their new
                // values pass while the points between are updated
                const Real d0 = rsub(u[1], u[0]);
                const Real dm = P > 2 ? rsub(u[P - 1], u[P - 2]) : d0;
                v0 = rfma(c2, rsub(d0, rsub(u[0], lft)), w[0]);
                n0 = radd(u[0], v0);
                add_source();
                const Real vl = rfma(c2, rsub(rsub(rgt, u[P - 1]), dm), w[P - 1]);
                const Real nl = radd(u[P - 1], vl);
                lft = __shfl_up_sync(kFull, nl, 1);
                rgt = __shfl_down_sync(kFull, n0, 1);
                rec(u, l_old, r_old, s);
                Real dprev = d0;
#pragma unroll
                for (int i = 1; i < P - 1; ++i) {
                    const Real d = i < P - 2 ? rsub(u[i + 1], u[i]) : dm;
                    const Real v = rfma(c2, rsub(d, dprev), w[i]);
                    dprev = d;
                    w[i] = v;
                    u[i] = radd(u[i], v);
                }
                u[0] = n0;
                w[0] = v0;
                u[P - 1] = nl;
                w[P - 1] = vl;
            } else {
                n0 = rfma(c2, radd(lft, u[1]), rfma(k, u[0], -w[0]));
                v0 = u[0];
                add_source();
                const Real nl = rfma(c2, radd(u[P - 2], rgt), rfma(k, u[P - 1], -w[P - 1]));
                lft = __shfl_up_sync(kFull, nl, 1);
                rgt = __shfl_down_sync(kFull, n0, 1);
                rec(u, l_old, r_old, s);
                Real ul = u[0];
#pragma unroll
                for (int i = 1; i < P - 1; ++i) {
                    const Real uc = u[i];
                    u[i] = rfma(c2, radd(ul, u[i + 1]), rfma(k, uc, -w[i]));
                    w[i] = uc;
                    ul = uc;
                }
                w[P - 1] = u[P - 1];
                u[P - 1] = nl;
                u[0] = n0;
                w[0] = v0;
            }
            if constexpr (kStream) {
                st.cur = nxt;
                take();
            }
        }
        if constexpr (kStream)
            if (((lv + s1) & 31) == 0) st.next();
        s0 = s1;
    }
}

// One value into the inbox of a neighbouring CTA of the cluster (an address in
// the cluster's shared-memory window), counted by the mbarrier beside it.
__device__ __forceinline__ void st_async(uint32_t a, uint32_t bar, float x)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a),
                 "r"(__float_as_uint(x)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_async(uint32_t a, uint32_t bar, double x)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(a),
                 "l"(__double_as_longlong(x)), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ bool inbox_arrived(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint32_t cluster_addr(uint32_t a, int rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

// A window (one component) in shared memory as 16-byte units, the low bits of a
// unit's place mixed with the next ones: neither a lane's own P points nor
// consecutive points of the window meet bank conflicts.
template <typename Real>
__device__ __forceinline__ int unit_place(int unit)
{
    return (unit ^ ((unit >> 3) & 7)) * (int)(16 / sizeof(Real));
}

// unit_place(u0 + i), u0 = lane * (P / N): with up to 8 units per lane the mixing
// term is the same for all of them (one exclusive-or per unit)
template <typename Real, int P>
__device__ __forceinline__ int lane_unit(uint32_t u0, int i)
{
    constexpr int N = 16 / sizeof(Real);
    if constexpr (P / N <= 8 && (P / N & (P / N - 1)) == 0)
        return (int)(((u0 & ~7u) + (((u0 & 7u) + i) ^ ((u0 >> 3) & 7u))) * N);
    else
        return unit_place<Real>((int)u0 + i);
}

template <typename Real, int P>
__device__ __forceinline__ void put_units(Real* sm, const Real (&v)[P], int lane)
{
    constexpr int N = 16 / sizeof(Real);
    if constexpr (P % N == 0) {
        using V = typename span::Vec<Real, P>::T;
        const uint32_t u0 = (uint32_t)(lane * (P / N));
#pragma unroll
        for (int i = 0; i < P / N; ++i) {
            V x;
            x.x = v[N * i];
            x.y = v[N * i + 1];
            if constexpr (N == 4) {
                x.z = v[N * i + 2];
                x.w = v[N * i + 3];
            }
            *reinterpret_cast<V*>(sm + lane_unit<Real, P>(u0, i)) = x;
        }
    } else {  // (FP64, one point per lane)
        sm[unit_place<Real>(lane / N) + lane % N] = v[0];
    }
}

template <typename Real, int P>
__device__ __forceinline__ void get_units(const Real* sm, Real (&v)[P], int lane)
{
    constexpr int N = 16 / sizeof(Real);
    static_assert(P % N == 0, "whole units");
    using V = typename span::Vec<Real, P>::T;
    const uint32_t u0 = (uint32_t)(lane * (P / N));
#pragma unroll
    for (int i = 0; i < P / N; ++i) {
        const V x = *reinterpret_cast<const V*>(sm + lane_unit<Real, P>(u0, i));
        v[N * i] = x.x;
        v[N * i + 1] = x.y;
        if constexpr (N == 4) {
            v[N * i + 2] = x.z;
            v[N * i + 3] = x.w;
        }
    }
}

// The window's points [a, a + n) to a global array (dst: window position 0)
// through shared memory, so that a warp's stores cover whole lines (straight
// from the registers a store touches a 16-byte piece of 32 lines: 1.4 TB/s
// measured).  In shared memory the window is moved up by the 0 .. N - 1 points
// that put its units on the array's 16-byte boundaries.
template <typename Real, int P>
__device__ __forceinline__ void store_owned(Real* dst, const Real (&v)[P], Real* sm, int lane, int a, int n)
{
    constexpr int N = 16 / sizeof(Real);
    const int off = (int)((reinterpret_cast<uintptr_t>(dst) / sizeof(Real)) & (N - 1));
    if (off == 0 && P % N == 0) {
        put_units<Real, P>(sm, v, lane);
    } else {
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const int p = lane * P + i + off;
            sm[unit_place<Real>(p / N) + p % N] = v[i];
        }
    }
    __syncwarp();
    dst -= off;
    const int b = a + off, e = b + n;                    // positions in shared memory
    const int u0 = (b + N - 1) / N, u1 = e / N;          // whole units [u0, u1)
    if (u0 < u1) {
        using V = typename span::Vec<Real, P>::T;
        // 32 units on, the mixing term changes in its third bit: two places in turn
        const int u = u0 + lane;
        const Real* s0 = sm + unit_place<Real>(u);
        const Real* s1 = sm + unit_place<Real>(u + 32);
        Real* d = dst + u * N;
        constexpr int K = (P + N - 1) / N;
#pragma unroll
        for (int k = 0; k < K; k += 2) {
            if (u + 32 * k < u1) *reinterpret_cast<V*>(d + 32 * N * k) = *reinterpret_cast<const V*>(s0 + 32 * N * k);
            if (k + 1 < K && u + 32 * k + 32 < u1)
                *reinterpret_cast<V*>(d + 32 * N * (k + 1)) = *reinterpret_cast<const V*>(s1 + 32 * N * k);
        }
    }
    // the points before the first and after the last whole unit
    if (u0 > u1 || u0 * N != b || u1 * N != e) {
        const int h = u0 <= u1 ? u0 * N : e;
        if (b + lane < h) dst[b + lane] = sm[unit_place<Real>((b + lane) / N) + (b + lane) % N];
        const int t = u0 <= u1 ? u1 * N : e;
        if (t + lane < e) dst[t + lane] = sm[unit_place<Real>((t + lane) / N) + (t + lane) % N];
    }
    __syncwarp();
}

template <typename Real, int P>
__device__ __forceinline__ void load_window(const Real* src, Real (&v)[P], int j0, int nx)
{
    constexpr int N = 16 / sizeof(Real);
    if constexpr (P % N == 0) {
        if (j0 >= 0 && j0 + P <= nx && (reinterpret_cast<uintptr_t>(src + j0) & 15) == 0) {
            span::smem_to_regs<Real, P>(src + j0, v);
            return;
        }
    }
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = (j0 + i >= 0 && j0 + i < nx) ? src[j0 + i] : Real(0);
}

// The exchange between a warp and its two neighbours: the H owned points next
// to each end become the neighbours' halos.
template <typename Real, int P>
struct Exchange {
    Real* area;           // this warp's shared memory: window [parity][component][32 P], inbox
    uint64_t (*bar)[2][2];  // warp, side, parity: the neighbour's points are there
    int H, warp, lane, a0, len;
    bool left, right, ext_l, ext_r, cluster, by_bar, vec;
    // what this lane's registers [hb, he) take from a neighbour, and where from
    // for parity 0 (the neighbour's window in the CTA, or the inbox)
    int hb, he, hstep;
    const Real *hu, *hw;
    ulonglong2 *out_l, *out_r;
    const ulonglong2 *in_l, *in_r;
    uint32_t box_l, box_r, bar_l, bar_r;
    int words;

    // inbox (side, parity) of a warp's area: both components, H values each
    __device__ __forceinline__ Real* inbox(Real* a, int side, int par) const
    {
        return a + 128 * P + (side * 2 + par) * 2 * H;
    }

    __device__ __forceinline__ void init(const ResExchange& x, const ResWarp* warps, const ResWarp& wd, int g,
                                         Real* area0, uint64_t (*bars)[2][2])
    {
        lane = threadIdx.x & 31;
        warp = threadIdx.x >> 5;
        const int nwarp = blockDim.x >> 5;
        H = x.H;
        cluster = x.cluster;
        bar = bars;
        area = area0 + (size_t)warp * x.warp_values;
        a0 = wd.lo - wd.start;
        len = wd.len;
        left = wd.links & 1;
        right = wd.links & 2;
        ext_l = wd.links & 4;
        ext_r = wd.links & 8;
        by_bar = cluster || !(ext_l | ext_r);  // (no side is polled in global memory)
        hb = he = hstep = 0;
        hu = hw = area;
        bool v = true;
        auto clampP = [](int t) { return t < 0 ? 0 : (t > P ? P : t); };
        const int p0 = lane * P;
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            if (!(side ? right : left)) continue;
            const int a = side ? a0 + len : a0 - H;  // window positions [a, a + H)
            const int b = clampP(a - p0), e = clampP(a + H - p0);
            if (e <= b) continue;
            hb = b;
            he = e;
            const Real* src;
            if (side ? ext_r : ext_l) {
                src = inbox(area, side, 0) + (p0 - a);
                hw = src + H;
                hstep = 2 * H;
            } else {
                // the neighbour's position of this window's position p0
                const int nb = warp + (side ? 1 : -1);
                src = area0 + (size_t)nb * x.warp_values + (wd.start + p0 - warps[g + (side ? 1 : -1)].start);
                hw = src + 32 * P;
                hstep = 64 * P;
            }
            hu = src;
            constexpr int N = 16 / sizeof(Real);
            if (b != 0 || e != P || P % N != 0 || ((src - area0) & (N - 1)) != 0 || ((hw - area0) & (N - 1)) != 0)
                v = false;
        }
        vec = __all_sync(kFull, v);
        // across CTAs: the slots, or in a cluster the neighbours' inboxes and their barriers
        out_l = out_r = nullptr;
        in_l = in_r = nullptr;
        box_l = box_r = bar_l = bar_r = 0;
        words = H * slot_words<Real>;  // of a slot; parity 1 follows parity 0
        if (cluster) {
            if (ext_l) {
                box_l = cluster_addr(smem_addr(inbox(area0 + (size_t)(nwarp - 1) * x.warp_values, 1, 0)), blockIdx.x - 1);
                bar_l = cluster_addr(smem_addr(&bars[nwarp - 1][1][0]), blockIdx.x - 1);
            }
            if (ext_r) {
                box_r = cluster_addr(smem_addr(inbox(area0, 0, 0)), blockIdx.x + 1);
                bar_r = cluster_addr(smem_addr(&bars[0][0][0]), blockIdx.x + 1);
            }
        } else {
            ulonglong2* s = x.xbuf + (int64_t)blockIdx.x * 4 * words;  // [CTA][side][parity]
            out_l = s;
            out_r = s + 2 * words;
            in_l = s - 2 * words;  // the CTA before, its right side
            in_r = s + 4 * words;  // the CTA after, its left side
        }
    }

    // The k-th exchange of the run.  false: a wait ran out (or another warp's
    // did).  mute: this warp publishes nothing (test hook).
    __device__ __forceinline__ bool swap(const ResExchange& x, Real (&u)[P], Real (&w)[P], int k, bool mute)
    {
        // the H owned points next to each end to shared memory, and those next to
        // an end that has its neighbour in another CTA onwards
        const int par = k & 1;
        const unsigned long long tag = (x.epoch << 32) | (unsigned)(k + 1);
        Real* const win = area + par * 64 * P;
        // (with 64 bytes and more to a lane, from the few lanes that hold them only: 32
        // lanes at that stride meet in the same banks; 1,048,576 FP32 points, 2048
        // steps, 439 -> 402 us.  Below, the branch costs more than the conflicts.)
        const int p0 = lane * P;
        if (P * sizeof(Real) < 64 || (left && p0 < a0 + H && p0 + P > a0) || (right && p0 < a0 + len && p0 + P > a0 + len - H)) {
            if constexpr (P * sizeof(Real) % 16 == 0) {
                span::regs_to_smem<Real, P>(win + lane * P, u);
                span::regs_to_smem<Real, P>(win + 32 * P + lane * P, w);
            } else {
#pragma unroll
                for (int i = 0; i < P; ++i) {
                    win[lane * P + i] = u[i];
                    win[32 * P + lane * P + i] = w[i];
                }
            }
        }
        __syncwarp();
        if (lane < 2 && !mute) {
            const bool has = lane ? right : left, ext = lane ? ext_r : ext_l;
            // this warp's points are there, for the neighbour in the CTA; what
            // the inbox waits for, from the neighbour in the cluster
            if (has && !ext) mbar_arrive(&bar[lane ? warp + 1 : warp - 1][lane ^ 1][par]);
            else if (has && cluster)
                mbar_arrive_expect_tx(&bar[warp][lane][par], (uint32_t)(2 * H * sizeof(Real)));
        }
        if (ext_l | ext_r) {
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                if (!(side ? ext_r : ext_l) || mute) continue;
                const Real* src = win + (side ? a0 + len - H : a0);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int p = lane + 32 * h;
                    if (p >= H) continue;
                    const Real a = src[p], b = src[32 * P + p];
                    if (cluster) {
                        const uint32_t box = (side ? box_r : box_l) + (uint32_t)((par * 2 * H + p) * sizeof(Real));
                        const uint32_t nbar = (side ? bar_r : bar_l) + par * 8u;
                        st_async(box, nbar, a);
                        st_async(box + (uint32_t)(H * sizeof(Real)), nbar, b);
                    } else {
                        ulonglong2* out = (side ? out_r : out_l) + par * words;
                        if constexpr (sizeof(Real) == 4) {
                            st_pair(out + p, (unsigned long long)__float_as_uint(a) |
                                                 ((unsigned long long)__float_as_uint(b) << 32), tag);
                        } else {
                            st_pair(out + 2 * p, (unsigned long long)__double_as_longlong(a), tag);
                            st_pair(out + 2 * p + 1, (unsigned long long)__double_as_longlong(b), tag);
                        }
                    }
                }
            }
        }
        bool ok = true;
        // (every so many polls: the time limit, and whether another warp gave up)
        long long t0 = 0;
        unsigned spins = 0;
        auto late = [&]() {
            if ((++spins & 63u) != 0u) return false;
            const long long now = global_ns();
            if (t0 == 0) t0 = now;
            return now - t0 > x.wait_ns || *(volatile int*)&x.err->code != 0;
        };
        if (!by_bar) {
            // both sides are polled together: a poll of L2 is a long round trip
            bool want[2] = {ext_l, ext_r};
            for (;;) {
                unsigned long long y[2][2][4];  // [side][half]: u word, tag, (FP64: w word, tag)
#pragma unroll
                for (int side = 0; side < 2; ++side)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int p = lane + 32 * h;
                        if (!want[side] || p >= H) continue;
                        const ulonglong2* in = (side ? in_r : in_l) + par * words;
                        if constexpr (sizeof(Real) == 4) {
                            ld_pair(in + p, y[side][h][0], y[side][h][1]);
                        } else {
                            ld_pair(in + 2 * p, y[side][h][0], y[side][h][1]);
                            ld_pair(in + 2 * p + 1, y[side][h][2], y[side][h][3]);
                        }
                    }
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    if (!want[side]) continue;
                    bool all = true;
                    Real* box = inbox(area, side, par);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int p = lane + 32 * h;
                        if (p >= H) continue;
                        if constexpr (sizeof(Real) == 4) {
                            all = all && y[side][h][1] == tag;
                            box[p] = __uint_as_float((unsigned)y[side][h][0]);
                            box[H + p] = __uint_as_float((unsigned)(y[side][h][0] >> 32));
                        } else {
                            all = all && y[side][h][1] == tag && y[side][h][3] == tag;
                            box[p] = __longlong_as_double((long long)y[side][h][0]);
                            box[H + p] = __longlong_as_double((long long)y[side][h][2]);
                        }
                    }
                    want[side] = !all;
                }
                if (__all_sync(kFull, !want[0] && !want[1])) break;
                if (__any_sync(kFull, late())) {
                    ok = false;
                    break;
                }
            }
        }
        {
            const uint32_t phase = (uint32_t)(k >> 1) & 1u;
            if (ok && left && (by_bar || !ext_l))
                while (!inbox_arrived(&bar[warp][0][par], phase))
                    if (late()) {
                        ok = false;
                        break;
                    }
            if (ok && right && (by_bar || !ext_r))
                while (!inbox_arrived(&bar[warp][1][par], phase))
                    if (late()) {
                        ok = false;
                        break;
                    }
            ok = __all_sync(kFull, ok);
        }
        if (!ok) {
            // (what this warp sent to a neighbour in the cluster lands while both are there)
            if (cluster) __nanosleep(20000);
            return false;
        }
        __syncwarp();
        {
            const Real *su = hu + par * hstep, *sw = hw + par * hstep;
            if (vec) {
                if (he > 0) {
                    if constexpr (P * sizeof(Real) % 16 == 0) {
                        span::smem_to_regs<Real, P>(su, u);
                        span::smem_to_regs<Real, P>(sw, w);
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < P; ++i)
                    if (i >= hb && i < he) {
                        u[i] = su[i];
                        w[i] = sw[i];
                    }
            }
        }
        return true;
    }
};

// DENSE: compiled with the records of windows that hold many probes (runs without
// such a window pay 2 % for the code: 2^20 points, 406 -> 413 us).
template <typename Real, int FORM, int P, bool DENSE>
__global__ void __launch_bounds__(32 * max_warps<Real>(P), 1) resident_kernel(const __grid_constant__ ResParams<Real> prm)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nwarp = blockDim.x >> 5;
    Real* const area0 = reinterpret_cast<Real*>(smem_raw);
    Real* const area = area0 + (size_t)warp * prm.x.warp_values;
    Real* const ring = area + 128 * P + 8 * prm.x.H;

    __shared__ __align__(8) uint64_t s_bar[16][2][2];  // warp, side, parity: the neighbour's points are there
    if (threadIdx.x < 64) mbar_init(&s_bar[0][0][0] + threadIdx.x, 1);
    if (blockDim.x < 64 && threadIdx.x < 32) mbar_init(&s_bar[0][0][0] + 32 + threadIdx.x, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    // a cluster: every inbox exists before anyone writes to it, and (at the
    // end) no CTA leaves while a neighbour may still write to it
    auto cluster_sync = [&]() {
        if (!prm.x.cluster) return;
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    };
    cluster_sync();

    const int g = blockIdx.x * nwarp + warp;
    if (g >= prm.nwarps) {
        cluster_sync();
        return;
    }
    const ResWarp wd = prm.warps[g];
    const ResProb<Real> pb = prm.problems[wd.problem];
    const int nx = (int)pb.nx;
    const int lo = wd.lo, hi = wd.lo + wd.len;
    const int j0 = wd.start + lane * P;   // this lane's first grid point
    const Real c2 = pb.c2, kk = pb.k;

    // ---- level 0 (the second component at the nodes is "at rest")
    Real u[P], w[P];
    if (prm.in0) load_window<Real, P>(prm.in0 + pb.off, u, j0, nx);
    else
#pragma unroll
        for (int i = 0; i < P; ++i) u[i] = Real(0);
    if (prm.in1) load_window<Real, P>(prm.in1 + pb.off, w, j0, nx);
    else
#pragma unroll
        for (int i = 0; i < P; ++i) w[i] = FORM == kCanonical ? u[i] : Real(0);
    auto node_sample = [&](const Real* f, int64_t n) { return f ? f[n] : Real(0); };
#pragma unroll
    for (int i = 0; i < P; ++i) {  // (nodes inside the window)
        const int j = j0 + i;
        if (j != 0 && j != nx - 1) continue;
        u[i] = node_sample(j == 0 ? pb.fA : pb.fB, 0);
        w[i] = FORM == kCanonical ? u[i] : Real(0);
    }

    // ---- special points (the host places the windows and says which kind)
    const int spec = wd.spec;
    const int src_n = wd.src_end - wd.src_begin;
    const ResSrc<Real>* const srcs = prm.srcs + wd.src_begin;
    Stream<Real> st{};
    bool mine = false;
    if (spec == kNodeLeft) {
        st.open(pb.fA, 1, 0, lane, (int)prm.T);
        mine = lane == 0;
    } else if (spec == kNodeRight) {
        st.open(pb.fB, 1, 0, lane, (int)prm.T);
        mine = lane == 31;
    } else if (spec == kSource) {
        st.open(srcs[0].samples, srcs[0].stride, 1, lane, (int)prm.T);
        mine = srcs[0].j == j0;
    }
    // any special points, after a step from level n (level-n values xo), samples from memory
    auto patch_all = [&](Real(&x)[P], Real(&y)[P], const Real(&xo)[P], int64_t n) {
        auto node = [&](int j, const Real* f) {
            const int r = j - j0;
            if (r < 0 || r >= P) return;
            const Real a = node_sample(f, n), b = node_sample(f, n + 1);
#pragma unroll
            for (int i = 0; i < P; ++i)
                if (i == r) {
                    x[i] = b;
                    if constexpr (FORM == kIncrement) y[i] = rsub(b, a);
                }
        };
        for (int q = 0; q < src_n; ++q) {
            const ResSrc<Real> sr = srcs[q];
            const int r = sr.j - j0;
            if (r < 0 || r >= P) continue;
            const Real a = sr.samples[(n + 1) * sr.stride];
#pragma unroll
            for (int i = 0; i < P; ++i)
                if (i == r) {
                    if constexpr (FORM == kIncrement) {
                        y[i] = radd(y[i], a);
                        x[i] = radd(xo[i], y[i]);
                    } else {
                        x[i] = radd(x[i], a);
                    }
                }
        }
        node(0, pb.fA);
        node(nx - 1, pb.fB);
    };

    // ---- probes whose point this warp owns.  fast: one or two, on a lane's first
    // or last register (the host shifts a window for that): the owner drops the
    // value (flux: both neighbours) into a small buffer every level.  Else the
    // first two through rows of all the registers, further ones directly.
    // DENSE: of more than two every lane holds the records of those on its own
    // points and stores their values each level, all lanes at once: a level costs
    // four instructions per register however many there are.  (One by one from the
    // table, 0.36 us each on a window of 1024 points, they lost to tickets from three
    // on: 2^20 points in 1497 subdomains, all traces, 512 steps 795 us, with tickets
    // 723, this way 488.)  Only where a lane has more than fit are they taken so.
    constexpr int RL = kRowLanes<Real>(P);
    const int np = wd.probe_end - wd.probe_begin;
    const ProbeDev<Real>* const probes = prm.probes + wd.probe_begin;
    int pl[2] = {-64, -64}, pr[2] = {0, 0};  // first lane of the row (-64: none), position of the point in it
    int fl[2] = {-64, -64};                  // the probe's lane, if it is fast
    bool at_first[2] = {true, true}, flux[2] = {false, false};
    bool slow = np > 2, fast = np > 0 && np <= 2;
#pragma unroll
    for (int q = 0; q < 2; ++q)
        if (q < np) {
            const int pos = (int)probes[q].gidx - wd.start;  // gidx: the grid point
            flux[q] = probes[q].kind != 0;
            const int o = pos / P, r = pos % P;
            if (pos < 0 || pos >= 32 * P || (r != 0 && r != P - 1)) fast = false;
            fl[q] = o;
            at_first[q] = r == 0;
            if (pos < (flux[q] ? 1 : 0) || pos + (flux[q] ? 1 : 0) >= 32 * P) {
                slow = true;  // a node that is not in the window, or a flux next to one
                continue;
            }
            pl[q] = r == 0 && o > 0 ? o - 1 : o;
            pr[q] = pos - pl[q] * P;
        }
    if (fast) pl[0] = pl[1] = -64;
    int rounds = 0;  // records of a lane
    LaneProbe<Real>* const recs = reinterpret_cast<LaneProbe<Real>*>(ring) + lane;  // [round][32]
    if (DENSE && slow) {
        // (the probes are sorted by point)
        auto below = [&](int64_t j) {
            int a = 0, b = np;
            while (a < b) {
                const int m = (a + b) >> 1;
                if (probes[m].gidx < j) a = m + 1;
                else b = m;
            }
            return a;
        };
        const int from = below(j0 - (spec == kNodeLeft && lane == 0 ? 1 : 0));
        const int n = below(j0 + P + (spec == kNodeRight && lane == 31 ? 1 : 0)) - from;
        rounds = __reduce_max_sync(kFull, n);
        if (rounds <= max_rounds<Real>(P)) {
            for (int t = 0; t < rounds; ++t) {
                LaneProbe<Real> q{};
                q.code = -1;
                if (t < n) {
                    const ProbeDev<Real> p = probes[from + t];
                    q.out = p.out;
                    q.stride = p.stride;
                    q.scale = p.scale;
                    q.nmax = (int32_t)(p.nmax < 0x7fffffff ? p.nmax : 0x7fffffff);
                    q.code = 2 * ((int)p.gidx - j0 + 1) + (p.kind != 0 ? 1 : 0);
                }
                recs[32 * t] = q;
            }
            slow = false;
            pl[0] = pl[1] = -64;
        } else {
            rounds = 0;
        }
    }
    // level n of the points that have records
    auto put_records = [&](const Real(&x)[P], Real lft, Real rgt, int n) {
        for (int t = 0; t < rounds; ++t) {
            const LaneProbe<Real> q = recs[32 * t];
            const int r = (q.code >> 1) - 1;
            Real um = lft, uc = r < 0 ? lft : rgt, up = rgt;
#pragma unroll
            for (int i = 0; i < P; ++i)
                if (i == r) {
                    uc = x[i];
                    um = i > 0 ? x[i > 0 ? i - 1 : 0] : lft;
                    up = i < P - 1 ? x[i < P - 1 ? i + 1 : 0] : rgt;
                }
            const Real val = q.code & 1 ? rsub(up, um) : uc;
            st_global_if(q.code >= 0 && n <= q.nmax, q.out + n * q.stride, rmul(val, q.scale));
        }
    };
    // level n into the fast probes' buffers [probe][level mod kFastRing]{value or right, left}
    auto put_fast = [&](const Real(&x)[P], Real lft, Real rgt, int n) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            Real a, b;
            if constexpr (P == 1) {
                a = flux[q] ? rgt : x[0];
                b = lft;
            } else {
                a = at_first[q] ? (flux[q] ? x[1] : x[0]) : (flux[q] ? rgt : x[P - 1]);
                b = at_first[q] ? lft : x[P - 2];
            }
            Real* d = ring + (q * kFastRing + (n & (kFastRing - 1))) * 2;
            st_shared_if(lane == fl[q], d, a, b);
            if (np < 2) break;
        }
    };
    // (the writing out reads them every few levels: kept in shared memory)
    __shared__ ProbeDev<Real> s_probe[16][2];
    if (lane < 2 && lane < np) s_probe[warp][lane] = probes[lane];
    __syncwarp();
    // row n mod kRing holds level n; levels from `first` on are not written out yet
    int64_t first = 0;
    auto flush = [&](int64_t end) {
        __syncwarp();
        const int64_t n = first + lane;
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (pl[q] >= 0) {
                const ProbeDev<Real>& p = s_probe[warp][q];
                const Real* row = ring + (q * kRing + (int)(n & (kRing - 1))) * RL * P + pr[q];
                if (n < end && n <= p.nmax) {
                    const Real val = p.kind == 0 ? row[0] : rsub(row[1], row[-1]);
                    p.out[n * p.stride] = rmul(val, p.scale);
                }
            }
        if (fast) {
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (q < np) {
                    const ProbeDev<Real>& p = s_probe[warp][q];
                    const Real* d = ring + (q * kFastRing + (int)(n & (kFastRing - 1))) * 2;
                    if (n < end && n <= p.nmax) p.out[n * p.stride] = rmul(flux[q] ? rsub(d[0], d[1]) : d[0], p.scale);
                }
        }
        first = end;
        __syncwarp();
    };
    // level n of the window into its row; further probes directly
    auto put_rows = [&](const Real(&x)[P], int n) {
        const int s = n & (kRing - 1);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int l = lane - pl[q];
            Real* row = ring + ((q * kRing + s) * RL + l) * P;
            const bool on = l >= 0 && l < RL && pl[q] >= 0;
            if constexpr (P % 16 == 0 && sizeof(Real) == 4) {
#pragma unroll
                for (int i = 0; i < P; i += 16) {
                    float y[16];
#pragma unroll
                    for (int q = 0; q < 16; ++q) y[q] = (float)x[i + q];
                    st_shared_if16(on, reinterpret_cast<const float*>(row + i), y);
                }
            } else if constexpr (P % 2 == 0) {
#pragma unroll
                for (int i = 0; i < P; i += 2) st_shared_if(on, row + i, x[i], x[i + 1]);
            } else {
                if (on) row[0] = x[0];
            }
            if (np < 2) break;
        }
        if (slow) {
            Real lf = __shfl_up_sync(kFull, x[P - 1], 1);
            Real rg = __shfl_down_sync(kFull, x[0], 1);
            if (spec == kNodeLeft && lane == 0) lf = node_sample(pb.fA, n);
            if (spec == kNodeRight && lane == 31) rg = node_sample(pb.fB, n);
            for (int q = 0; q < np; ++q) {
                if (q < 2 && pl[q] >= 0) continue;
                const ProbeDev<Real> p = probes[q];
                const int r = (int)p.gidx - j0;
                if (n > p.nmax) continue;
                if (r == -1 && lane == 0 && spec == kNodeLeft) p.out[n * p.stride] = rmul(lf, p.scale);
                if (r == P && lane == 31 && spec == kNodeRight) p.out[n * p.stride] = rmul(rg, p.scale);
                if (r < 0 || r >= P) continue;
                Real um = lf, uc = x[0], up = rg;
#pragma unroll
                for (int i = 0; i < P; ++i)
                    if (i == r) {
                        uc = x[i];
                        um = i > 0 ? x[i > 0 ? i - 1 : 0] : lf;
                        up = i < P - 1 ? x[i < P - 1 ? i + 1 : 0] : rg;
                    }
                p.out[n * p.stride] = rmul(p.kind == 0 ? uc : rsub(up, um), p.scale);
            }
        }
    };
    // the pair of level n of the owned points (a node outside the window: from
    // its samples); sm: room for one component
    const int w0 = spec == kNodeLeft ? 0 : lo - wd.start;            // owned window positions [w0, w1)
    const int w1 = hi - wd.start - (spec == kNodeRight ? 1 : 0);
    auto store_pair = [&](Real* d0, Real* d1, int64_t n, Real* sm) {
        if (d0) store_owned<Real, P>(d0 + wd.start, u, sm, lane, w0, w1 - w0);
        if (d1) store_owned<Real, P>(d1 + wd.start, w, sm, lane, w0, w1 - w0);
        if ((spec == kNodeLeft && lane == 0) || (spec == kNodeRight && lane == 31)) {
            const Real* f = spec == kNodeLeft ? pb.fA : pb.fB;
            const int j = spec == kNodeLeft ? 0 : nx - 1;
            const Real a = node_sample(f, n - 1), b = node_sample(f, n);
            if (d0) d0[j] = b;
            if (d1) d1[j] = FORM == kCanonical ? a : rsub(b, a);
        }
    };

    Exchange<Real, P> ex;
    ex.init(prm.x, prm.warps, wd, g, area0, s_bar);
    bool ok = true;
    int kept = 0, part_left = 0;  // states kept so far, steps to the next one
    const int probe_levels = fast ? kFastRing : kRing;
    const int Tn = (int)prm.T;
    for (int k = 0; k < prm.nchunks; ++k) {
        const int64_t n0 = (int64_t)k * prm.S;
        const int steps = Tn - n0 < prm.S ? (int)(Tn - n0) : prm.S;
        // (with kept states: a state after every part of ck_steps steps, or of
        // ck_split and ck_steps - ck_split in turn; with probes: the levels up to
        // the end of their buffer)
        for (int d0 = 0; d0 < steps;) {
            const int64_t b0 = n0 + d0;
            int n = steps - d0;
            if (prm.ck0) {
                if (part_left == 0)
                    part_left = prm.ck_split == 0 ? prm.ck_steps : (kept & 1 ? prm.ck_steps - prm.ck_split : prm.ck_split);
                n = n < part_left ? n : part_left;
            }
            if (np) {
                const int room = probe_levels - ((int)b0 & (probe_levels - 1));
                n = n < room ? n : room;
            }
            d0 += n;
            auto patch = [&](Real(&x)[P], Real(&y)[P], const Real(&xo)[P], int s) { patch_all(x, y, xo, b0 + s); };
            auto advance = [&](auto&& rec) {
                switch (spec) {
                    case kPlain:
                        run_steps<Real, FORM, P, kPlain>(u, w, c2, kk, (int)b0, n, mine, st, rec, patch);
                        break;
                    case kNodeLeft:
                        run_steps<Real, FORM, P, kNodeLeft>(u, w, c2, kk, (int)b0, n, mine, st, rec, patch);
                        break;
                    case kNodeRight:
                        run_steps<Real, FORM, P, kNodeRight>(u, w, c2, kk, (int)b0, n, mine, st, rec, patch);
                        break;
                    case kSource:
                        run_steps<Real, FORM, P, kSource>(u, w, c2, kk, (int)b0, n, mine, st, rec, patch);
                        break;
                    default:
                        run_steps<Real, FORM, P, kAny>(u, w, c2, kk, (int)b0, n, mine, st, rec, patch);
                }
            };
            if (np == 0) {
                advance([](const Real(&)[P], Real, Real, int) {});
            } else if (fast) {
                advance([&](const Real(&x)[P], Real l, Real r, int s) { put_fast(x, l, r, (int)b0 + s); });
            } else {
                advance([&](const Real(&x)[P], Real l, Real r, int s) {
                    if (DENSE && rounds) put_records(x, l, r, (int)b0 + s);
                    else put_rows(x, (int)b0 + s);
                });
            }
            if (np && ((int)(b0 + n) & (probe_levels - 1)) == 0) flush(b0 + n);
            if (prm.ck0 && (part_left -= n) == 0) {
                const int64_t o = (int64_t)(++kept) * prm.ck_stride + pb.base;
                // (this exchange's window: free till then)
                store_pair(prm.ck0 + o, prm.ck1 + o, b0 + n, area + (k & 1) * 64 * P);
            }
        }
        if (k + 1 == prm.nchunks) break;

        ok = ex.swap(prm.x, u, w, k, g == prm.inject_warp && k >= prm.inject_chunk);
        if (!ok) {
            latch_error(prm.x.err, kDevTimeoutFlag, g, k, 0);
            break;
        }
    }
    if (!ok) {
        cluster_sync();
        return;
    }

    // ---- level T: probes and the state pair
    if (np > 0) {
        if (fast || (DENSE && rounds)) {
            Real l = __shfl_up_sync(kFull, u[P - 1], 1), r = __shfl_down_sync(kFull, u[0], 1);
            if (spec == kNodeLeft && lane == 0) l = node_sample(pb.fA, prm.T);
            if (spec == kNodeRight && lane == 31) r = node_sample(pb.fB, prm.T);
            if (fast) put_fast(u, l, r, (int)prm.T);
            else put_records(u, l, r, (int)prm.T);
        } else {
            put_rows(u, (int)prm.T);
        }
        flush(prm.T + 1);
    }
    store_pair(prm.out0 ? prm.out0 + pb.off : nullptr, prm.out1 ? prm.out1 + pb.off : nullptr, prm.T,
               area + ((prm.nchunks - 1) & 1) * 64 * P);
    cluster_sync();
}

}  // namespace resident
}  // namespace rswr
