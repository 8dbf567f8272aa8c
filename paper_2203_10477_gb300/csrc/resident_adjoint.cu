// resident_adjoint.cu -- the discrete adjoint sweep with dL/da on grids that fit
// on the chip: every warp keeps its piece of the adjoint variables for the whole
// sweep (resident.cuh: windows, exchange, nodes as neighbours of the outermost
// lanes).
//
// The sweep runs spans of `span` steps, the last first, each in one or two parts
// of at most SA steps.  Per part a warp takes its window of the forward state at
// the part's start from shared memory (copied there a part ahead, cp.async),
// recomputes the part's levels and keeps their Laplacians -- FP32 in tensor
// memory, one lane per thread, SA P columns; FP64 in shared memory -- then steps
// the adjoint variables and pairs every level with its Laplacian.  The halos are
// exchanged every E spans (halo at least E span).  Same operations on the same
// operands as adjoint_kernel.cu, so dL/dfA has the same bits; dL/da sums the
// same products: FP32 in the same chains (eight points from a multiple of eight,
// over the levels of a span), the rest in double.
//
// What bounds it: FP64 its pipe (8 operations per point and level, of 64 clocks
// per warp and scheduler); FP32 the issue slots on full grids (about 12 P + 45
// instructions per warp and level) and the chain of two steps and the exchange
// on small ones.  Measured: 2^20 FP32 points, 2048 levels, 1.43 ms for this sweep;
// a training step with it 4389 .. 4509 (persistent adjoint_kernel) -> 2673 .. 3137 us;
// the gradient of 65539 FP64 points, 2048 levels, 13113 -> 4537 us.

#include "resident.cuh"
#include "tmem.cuh"

namespace rswr {

namespace {

using namespace resident;
using span::kFull;

// shared memory of a warp's exchange set-up, in bytes: the common part, and five
// words of every lane
constexpr size_t kExchangeBytes = (sizeof(Exchange<float, 8>) + 15) / 16 * 16;
static_assert(sizeof(Exchange<float, 16>) <= kExchangeBytes && sizeof(Exchange<double, 8>) <= kExchangeBytes &&
                  sizeof(Exchange<double, 2>) <= kExchangeBytes,
              "one size for all variants");

// columns of tensor memory a CTA allocates: SA P for every four warps, a power of two
__host__ __device__ inline uint32_t radj_columns(int warps, int P, int SA)
{
    uint32_t c = 32;
    while (c < (uint32_t)(((warps + 3) / 4) * SA * P)) c *= 2;
    return c;
}

// warps of a CTA at most (a lane holds two pairs of P points)
template <typename Real>
__host__ __device__ constexpr int radj_max_warps(int P) { return sizeof(Real) == 8 && P >= 4 ? 8 : 16; }

template <typename Real, int FORM, int P, int SA, bool TM>
__global__ void __launch_bounds__(32 * radj_max_warps<Real>(P), 1)
    resident_adjoint_kernel(const __grid_constant__ ResAdjParams<Real> prm)
{
    static_assert(!TM || (sizeof(Real) == 4 && P % 8 == 0), "tensor memory holds FP32 words, 8 columns at a time");
    static_assert(SA <= 32, "a span's samples are held across the warp");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t s_bar[16][2][2];
    __shared__ uint32_t s_tmem;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nwarp = blockDim.x >> 5;
    Real* const area0 = reinterpret_cast<Real*>(smem_raw);
    Real* const area = area0 + (size_t)warp * prm.x.warp_values;
    Real* const laps = area + 128 * P + 8 * prm.x.H;               // [SA][32][P] (not with TM)
    Real* const row = laps + (TM ? 0 : SA * 32 * P);               // the boundary gradient's values of a part
    Real* const fwd = row + 64;                                    // the next part's forward window [component][32 P]

    if constexpr (TM) {
        // (the launch asks for more than half of an SM's shared memory, so one
        // CTA per SM: the allocation never waits)
        if (warp == 0) {
            tmem_alloc(&s_tmem, radj_columns(nwarp, P, SA));
            tmem_relinquish();
        }
        tmem_fence_before_sync();
    }
    if (threadIdx.x < 64) mbar_init(&s_bar[0][0][0] + threadIdx.x, 1);
    if (blockDim.x < 64 && threadIdx.x < 32) mbar_init(&s_bar[0][0][0] + 32 + threadIdx.x, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    auto cluster_sync = [&]() {
        if (!prm.x.cluster) return;
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    };
    cluster_sync();
    uint32_t tm = 0;
    if constexpr (TM) {
        tmem_fence_after_sync();
        tm = tmem_addr(s_tmem, 32u * (uint32_t)(warp & 3), (uint32_t)((warp >> 2) * SA * P));
    }

    const int g = blockIdx.x * nwarp + warp;
    if (g < prm.nwarps) {
        const ResWarp wd = prm.warps[g];
        const ResAdjProb<Real> pb = prm.problems[wd.problem];
        const int nx = (int)pb.nx;
        const int j0 = wd.start + lane * P;
        const Real c2 = pb.c2, kk = pb.k;
        const int T = (int)prm.T;
        // (between the exchanges their set-up waits in shared memory: the levels need
        // the registers)
        using Ex = Exchange<Real, P>;
        Ex* const s_ex = reinterpret_cast<Ex*>(fwd + 64 * P);  // the warp's common part
        int* const s_lane = reinterpret_cast<int*>(reinterpret_cast<char*>(s_ex) + kExchangeBytes) + lane;  // [5][32]
        {
            Ex ex;
            ex.init(prm.x, prm.warps, wd, g, area0, s_bar);
            if (lane == 0) *s_ex = ex;
            s_lane[0] = ex.hb;
            s_lane[32] = ex.he;
            s_lane[64] = ex.hstep;
            s_lane[96] = (int)(ex.hu - area0);
            s_lane[128] = (int)(ex.hw - area0);
            __syncwarp();
        }

        // a Dirichlet node inside the window: of a grid's end piece, on one lane's
        // register nr (the left one always on register 0)
        const bool end_l = !(wd.links & 1), end_r = !(wd.links & 2);
        const int npos = end_l ? -wd.start : nx - 1 - wd.start;
        const int nr = npos % P;
        const bool mine = (end_l || end_r) && lane == npos / P;
        // how the level loops patch it: 1 / 3 first / last register, 4 + r / 4: one of
        // four registers (by compares: a jump on the register costs 100 clocks and more)
        const int node = !(end_l || end_r) ? 0 : (nr == 0 ? 1 : (nr == P - 1 ? 3 : 4 + nr / 4));
        const int nr_l = mine ? nr : -1;
        const Real* const f = end_l ? pb.fA : (end_r ? pb.fB : nullptr);
        // the adjoint's source (the cotangent at the receiver), if this window needs it
        const int spos = pb.js - wd.start;
        const bool has_src = pb.js >= 0 && pb.js >= wd.lo - prm.x.H && pb.js < wd.lo + wd.len + prm.x.H && spos >= 0 &&
                             spos < 32 * P;
        const bool src_mine = has_src && lane == spos / P;
        const int src_r = src_mine ? spos % P : -1;
        const int src = !has_src ? 0 : 4 + (spos % P) / 4;  // as node
        // owned points that are interior grid points, in register indices
        auto clampP = [](int t) { return t < 0 ? 0 : (t > P ? P : t); };
        // (the left node counts: its adjoint is 0, and so are its products)
        const int lo = wd.lo, hi = wd.lo + wd.len < nx - 1 ? wd.lo + wd.len : nx - 1;
        const int ilo = clampP(lo - j0), ihi = clampP(hi - j0);
        const bool owner = ihi > ilo;
        const bool part = __any_sync(kFull, owner && ihi - ilo < P);  // some lane owns some of its points
        const uint32_t mask = (ihi > ilo) ? (uint32_t)(((1ull << (ihi - ilo)) - 1ull) << ilo) : 0u;
        const bool rec = pb.js >= 0 && end_l;  // this warp holds j = 1, on lane 0 (P > 1)

        Real l[P], lw[P];
#pragma unroll
        for (int i = 0; i < P; ++i) l[i] = lw[i] = Real(0);
        if (pb.js >= 0) {
            const Real x = pb.wbar[T];  // lambda at level 1
#pragma unroll
            for (int i = 0; i < P; ++i)
                if (j0 + i == pb.js) {
                    l[i] = x;
                    lw[i] = FORM == kCanonical ? Real(0) : x;
                }
        }
        // part x of the sweep: levels [n0, n0 + len), state x at its start
        const int span = prm.span, split = prm.split;  // split: steps of a span's first part (0: one part)
        auto levels = [&](int x, int& n0, int& len) {
            const int k = split ? x >> 1 : x;
            n0 = k * span + ((split && (x & 1)) ? split : 0);
            const int end = (split && !(x & 1)) ? k * span + split : (k + 1) * span;
            len = (end < T ? end : T) - n0;
        };
        Real cu = Real(0), cs = Real(0);  // the part's node / source samples across the warp
        // the next part to ask for (they come last first): its forward window into
        // shared memory (cp.async; windows start on 16-byte boundaries of the
        // states, whose tail past nx is part of the allocation) and its samples
        constexpr int N = 16 / sizeof(Real);
        const Real* ask0 = prm.uck0 + (int64_t)(prm.parts - 1) * prm.ck_stride + pb.base + wd.start + lane * N;
        const Real* ask1 = ask0 + (prm.uck1 - prm.uck0);
        uint32_t inside = 0;  // units of this lane that are in the grid
#pragma unroll
        for (int q = 0; q < P / N; ++q) {
            const int j = wd.start + (q * 32 + lane) * N;
            if (j >= 0 && j < nx) inside |= 1u << q;
        }
        // (32 units on the mixing term of a unit's place changes in its third bit)
        const uint32_t d0s = smem_addr(fwd + unit_place<Real>(lane));
        const uint32_t d1s = smem_addr(fwd + unit_place<Real>(lane + 32));
        auto ask = [&](int n0, int len) {
#pragma unroll
            for (int q = 0; q < P / N; ++q) {
                if (!((inside >> q) & 1u)) continue;
                const uint32_t d = (q & 1 ? d1s : d0s) + (uint32_t)((q & ~1) * 512);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(ask0 + q * 32 * N) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + (uint32_t)(32 * P * sizeof(Real))),
                             "l"(ask1 + q * 32 * N)
                             : "memory");
            }
            ask0 -= prm.ck_stride;
            ask1 -= prm.ck_stride;
            if (f) cu = n0 + lane <= T ? f[n0 + lane] : Real(0);
            // lambda step s of the part adds wbar[n0 + len - 1 - s]
            const int q = n0 + len - 1 - lane;
            if (has_src) cs = q >= 0 ? pb.wbar[q] : Real(0);
        };
        // (units outside the grid are never copied: zeros)
        for (int i = lane; i < 64 * P; i += 32) fwd[i] = Real(0);
        __syncwarp();
        int n0, len;
        levels(prm.parts - 1, n0, len);
        ask(n0, len);
        // (a span's sums meet in double: the sum over the spans may leave FP32's range)
        double acc = 0.0;
        constexpr int G = sizeof(Real) == 4 && P > 8 ? P / 8 : 1;  // summation groups of a lane
        Real racc[G];
#pragma unroll
        for (int q = 0; q < G; ++q) racc[q] = Real(0);
        bool ok = true;

        for (int x = prm.parts - 1; x >= 0; --x) {
            Real cu_now, cs_now;
            int n0_next = 0, len_next = 0;
            if (x > 0) levels(x - 1, n0_next, len_next);

            // ---- u phase: levels n0 .. n0 + len - 1, their Laplacians kept
            {
                Real u[P], w[P];
                asm volatile("cp.async.wait_all;" ::: "memory");
                __syncwarp();
                get_units<Real, P>(fwd, u, lane);
                get_units<Real, P>(fwd + 32 * P, w, lane);
                __syncwarp();
                cu_now = cu;
                cs_now = cs;
                // the adjoint pair waits in shared memory: the levels need the registers
                put_units<Real, P>(fwd, l, lane);
                put_units<Real, P>(fwd + 32 * P, lw, lane);
                Real f_old = __shfl_sync(kFull, cu_now, 0);
                // (the kept state of level 0 holds no boundary data)
#pragma unroll
                for (int i = 0; i < P; ++i) u[i] = mine && i == nr ? f_old : u[i];
                Real lft = __shfl_up_sync(kFull, u[P - 1], 1);
                Real rgt = __shfl_down_sync(kFull, u[0], 1);
                auto level = [&](auto step_c, auto node_c, int s) {
                    constexpr bool STEP = decltype(step_c)::value;
                    constexpr int NODE = decltype(node_c)::value;
                    Real f_new = Real(0);  // the node's next level
                    if constexpr (STEP && NODE != 0) f_new = __shfl_sync(kFull, cu_now, s + 1);
                    Real lp[P];
                    if constexpr (FORM == kIncrement) {
                        const Real d0 = rsub(u[1], u[0]);
                        const Real dm = P > 2 ? rsub(u[P - 1], u[P - 2]) : d0;
                        lp[0] = rsub(d0, rsub(u[0], lft));
                        lp[P - 1] = rsub(rsub(rgt, u[P - 1]), dm);
                        Real n_0 = u[0], v_0 = w[0], n_l = u[P - 1], v_l = w[P - 1];
                        if constexpr (STEP) {
                            v_0 = rfma(c2, lp[0], w[0]);
                            n_0 = radd(u[0], v_0);
                            v_l = rfma(c2, lp[P - 1], w[P - 1]);
                            n_l = radd(u[P - 1], v_l);
                            if constexpr (NODE == 1) {
                                n_0 = mine ? f_new : n_0;
                                v_0 = mine ? rsub(f_new, f_old) : v_0;
                            }
                            if constexpr (NODE == 3) {
                                n_l = mine ? f_new : n_l;
                                v_l = mine ? rsub(f_new, f_old) : v_l;
                            }
                            lft = __shfl_up_sync(kFull, n_l, 1);
                            rgt = __shfl_down_sync(kFull, n_0, 1);
                        }
                        Real dprev = d0;
#pragma unroll
                        for (int i = 1; i < P - 1; ++i) {
                            const Real d = i < P - 2 ? rsub(u[i + 1], u[i]) : dm;
                            lp[i] = rsub(d, dprev);
                            dprev = d;
                            if constexpr (STEP) {
                                const Real v = rfma(c2, lp[i], w[i]);
                                w[i] = v;
                                u[i] = radd(u[i], v);
                            }
                        }
                        u[0] = n_0;
                        w[0] = v_0;
                        u[P - 1] = n_l;
                        w[P - 1] = v_l;
                    } else {
                        const Real s0 = radd(lft, u[1]), sl = radd(u[P - 2], rgt);
                        lp[0] = rfma(Real(-2), u[0], s0);
                        lp[P - 1] = rfma(Real(-2), u[P - 1], sl);
                        Real n_0 = u[0], n_l = u[P - 1];
                        if constexpr (STEP) {
                            n_0 = rfma(c2, s0, rfma(kk, u[0], -w[0]));
                            n_l = rfma(c2, sl, rfma(kk, u[P - 1], -w[P - 1]));
                            if constexpr (NODE == 1) n_0 = mine ? f_new : n_0;
                            if constexpr (NODE == 3) n_l = mine ? f_new : n_l;
                            lft = __shfl_up_sync(kFull, n_l, 1);
                            rgt = __shfl_down_sync(kFull, n_0, 1);
                        }
                        Real ul = u[0];
#pragma unroll
                        for (int i = 1; i < P - 1; ++i) {
                            const Real uc = u[i];
                            const Real sum = radd(ul, u[i + 1]);
                            lp[i] = rfma(Real(-2), uc, sum);
                            if constexpr (STEP) {
                                u[i] = rfma(c2, sum, rfma(kk, uc, -w[i]));
                                w[i] = uc;
                            }
                            ul = uc;
                        }
                        if constexpr (STEP) {
                            w[0] = u[0];
                            w[P - 1] = u[P - 1];
                        }
                        u[0] = n_0;
                        u[P - 1] = n_l;
                    }
                    if constexpr (STEP && NODE >= 4) {
                        const Real df = rsub(f_new, f_old);
#pragma unroll
                        for (int i = 4 * (NODE - 4); i < 4 * (NODE - 4) + 4 && i < P - 1; ++i) {
                            u[i] = nr_l == i ? f_new : u[i];
                            if constexpr (FORM == kIncrement) w[i] = nr_l == i ? df : w[i];
                        }
                    }
                    f_old = f_new;
                    if constexpr (TM) {
#pragma unroll
                        for (int c = 0; c < P / 8; ++c) {
                            uint32_t b[8];
#pragma unroll
                            for (int q = 0; q < 8; ++q) b[q] = __float_as_uint((float)lp[8 * c + q]);
                            tmem_st8(tm + (uint32_t)(s * P + 8 * c), b);
                        }
                    } else {
                        span::regs_to_smem<Real, P>(laps + (s * 32 + lane) * P, lp);
                    }
                };
                auto all = [&](auto node_c) {
                    for (int s = 0; s + 1 < len; ++s) level(std::true_type{}, node_c, s);
                    level(std::false_type{}, node_c, len - 1);
                };
                switch (node) {
                    case 0: all(std::integral_constant<int, 0>{}); break;
                    case 1: all(std::integral_constant<int, 1>{}); break;
                    case 3: all(std::integral_constant<int, 3>{}); break;
                    case 4: all(std::integral_constant<int, 4>{}); break;
                    case 5: if constexpr (P > 4) all(std::integral_constant<int, 5>{}); break;
                    case 6: if constexpr (P > 8) all(std::integral_constant<int, 6>{}); break;
                    default: if constexpr (P > 12) all(std::integral_constant<int, 7>{});
                }
                if constexpr (TM) tmem_wait_st();
                asm volatile("" ::: "memory");
                get_units<Real, P>(fwd, l, lane);
                get_units<Real, P>(fwd + 32 * P, lw, lane);
                __syncwarp();
                if (x > 0) ask(n0_next, len_next);  // in flight during the adjoint steps
            }
            // ---- lambda phase: levels m0 .. m0 + len - 1 with u levels n0 + len - 1 .. n0
            Real lft = __shfl_up_sync(kFull, l[P - 1], 1);
            Real rgt = __shfl_down_sync(kFull, l[0], 1);
            auto lambda = [&](auto src_c, auto node_c) {
                constexpr int SRC = decltype(src_c)::value;
                constexpr int NODE = decltype(node_c)::value;
                // pairs the level of l with u level r's Laplacians
                [[maybe_unused]] uint32_t lb[TM ? P : 1];
                auto fetch = [&](int r) {
                    if constexpr (TM) {
#pragma unroll
                        for (int c = 0; c < P / 8; ++c)
                            tmem_ld8(tm + (uint32_t)(r * P + 8 * c), *reinterpret_cast<uint32_t(*)[8]>(lb + 8 * c));
                    }
                };
                auto pair = [&](int r) {
                    Real lp[P];
                    if constexpr (TM) {
                        __syncwarp();
#pragma unroll
                        for (int c = 0; c < P / 8; ++c) tmem_wait_ld(*reinterpret_cast<uint32_t(*)[8]>(lb + 8 * c));
#pragma unroll
                        for (int i = 0; i < P; ++i) lp[i] = (Real)__uint_as_float(lb[i]);
                    } else {
                        span::smem_to_regs<Real, P>(laps + (r * 32 + lane) * P, lp);
                    }
                    if (part) {
#pragma unroll
                        for (int i = 0; i < P; ++i)
                            if ((mask >> i) & 1u) racc[i * G / P] = rfma(l[i], lp[i], racc[i * G / P]);
                    } else {
#pragma unroll
                        for (int i = 0; i < P; ++i) racc[i * G / P] = rfma(l[i], lp[i], racc[i * G / P]);
                    }
                };
                fetch(len - 1);
                pair(len - 1);
                for (int s = 0; s < len; ++s) {
                    // (in tensor memory: asked for before the step, needed after it)
                    if (s + 1 < len) fetch(len - 2 - s);
                    if constexpr (NODE == 1 || NODE == 2) st_shared_if(rec && lane == 0, row + 2 * s, l[1], l[1]);
                    Real sv = Real(0);
                    if constexpr (SRC != 0) sv = __shfl_sync(kFull, cs_now, s);
                    // (a source adds to the new increment, or value in the canonical form)
                    auto add_source = [&](int i, Real& x) {
                        if constexpr (SRC != 0)
                            if (SRC == 2 || i / 4 == SRC - 4) {
                                const Real t = radd(x, sv);
                                x = src_r == i ? t : x;
                            }
                    };
                    // the end points first (as in run_steps)
                    Real n_0, v_0, n_l, v_l;
                    [[maybe_unused]] Real d0 = Real(0), dm = Real(0);
                    if constexpr (FORM == kIncrement) {
                        d0 = rsub(l[1], l[0]);
                        dm = P > 2 ? rsub(l[P - 1], l[P - 2]) : d0;
                        v_0 = rfma(c2, rsub(d0, rsub(l[0], lft)), lw[0]);
                        add_source(0, v_0);
                        n_0 = radd(l[0], v_0);
                        v_l = rfma(c2, rsub(rsub(rgt, l[P - 1]), dm), lw[P - 1]);
                        add_source(P - 1, v_l);
                        n_l = radd(l[P - 1], v_l);
                    } else {
                        n_0 = rfma(c2, radd(lft, l[1]), rfma(kk, l[0], -lw[0]));
                        add_source(0, n_0);
                        v_0 = l[0];
                        n_l = rfma(c2, radd(l[P - 2], rgt), rfma(kk, l[P - 1], -lw[P - 1]));
                        add_source(P - 1, n_l);
                        v_l = l[P - 1];
                    }
                    // (zero Dirichlet data)
                    if constexpr (NODE == 1 || NODE == 2) {
                        n_0 = nr_l == 0 ? Real(0) : n_0;
                        v_0 = nr_l == 0 ? Real(0) : v_0;
                    }
                    if constexpr (NODE == 3 || NODE == 2) {
                        n_l = nr_l == P - 1 ? Real(0) : n_l;
                        v_l = nr_l == P - 1 ? Real(0) : v_l;
                    }
                    lft = __shfl_up_sync(kFull, n_l, 1);
                    rgt = __shfl_down_sync(kFull, n_0, 1);
                    if constexpr (FORM == kIncrement) {
                        Real dprev = d0;
#pragma unroll
                        for (int i = 1; i < P - 1; ++i) {
                            const Real d = i < P - 2 ? rsub(l[i + 1], l[i]) : dm;
                            Real v = rfma(c2, rsub(d, dprev), lw[i]);
                            add_source(i, v);
                            dprev = d;
                            lw[i] = v;
                            l[i] = radd(l[i], v);
                        }
                    } else {
                        Real ul = l[0];
#pragma unroll
                        for (int i = 1; i < P - 1; ++i) {
                            const Real uc = l[i];
                            l[i] = rfma(c2, radd(ul, l[i + 1]), rfma(kk, uc, -lw[i]));
                            add_source(i, l[i]);
                            lw[i] = uc;
                            ul = uc;
                        }
                    }
                    l[0] = n_0;
                    lw[0] = v_0;
                    l[P - 1] = n_l;
                    lw[P - 1] = v_l;
                    if constexpr (NODE >= 2 && NODE != 3) {
                        constexpr int i0 = NODE == 2 ? 1 : 4 * (NODE - 4), i1 = NODE == 2 ? P - 1 : i0 + 4;
#pragma unroll
                        for (int i = i0; i < i1 && i < P - 1; ++i) {
                            l[i] = nr_l == i ? Real(0) : l[i];
                            lw[i] = nr_l == i ? Real(0) : lw[i];
                        }
                    }
                    if (s + 1 < len) pair(len - 2 - s);
                }
            };
            using C0 = std::integral_constant<int, 0>;
            if (src && node) {
                // (2: any register)
                lambda(std::integral_constant<int, 2>{}, std::integral_constant<int, 2>{});
            } else if (src) {
                switch (src) {
                    case 4: lambda(std::integral_constant<int, 4>{}, C0{}); break;
                    case 5: if constexpr (P > 4) lambda(std::integral_constant<int, 5>{}, C0{}); break;
                    case 6: if constexpr (P > 8) lambda(std::integral_constant<int, 6>{}, C0{}); break;
                    default: if constexpr (P > 12) lambda(std::integral_constant<int, 7>{}, C0{});
                }
            } else {
                switch (node) {
                    case 0: lambda(C0{}, C0{}); break;
                    case 1: lambda(C0{}, std::integral_constant<int, 1>{}); break;
                    case 3: lambda(C0{}, std::integral_constant<int, 3>{}); break;
                    case 4: lambda(C0{}, std::integral_constant<int, 4>{}); break;
                    case 5: if constexpr (P > 4) lambda(C0{}, std::integral_constant<int, 5>{}); break;
                    case 6: if constexpr (P > 8) lambda(C0{}, std::integral_constant<int, 6>{}); break;
                    default: if constexpr (P > 12) lambda(C0{}, std::integral_constant<int, 7>{});
                }
            }
            const int k = split ? x >> 1 : x;
            const bool span_done = !split || !(x & 1);
            if (span_done) {
#pragma unroll
                for (int q = 0; q < G; ++q) {
                    acc += owner ? (double)racc[q] : 0.0;
                    racc[q] = Real(0);
                }
            }
            if (rec) {
                // dL/dfA[T - m] = c2 lambda at j = 1, levels m = m0 .. m0 + len - 1
                __syncwarp();
                if (lane < len) pb.grad[n0 + len - 1 - lane] = rmul(row[2 * lane], c2);
                __syncwarp();
            }
            const int done = prm.nspans - k;
            if (span_done && k > 0 && done % prm.E == 0) {
                Ex ex = *s_ex;
                ex.lane = lane;
                ex.hb = s_lane[0];
                ex.he = s_lane[32];
                ex.hstep = s_lane[64];
                ex.hu = area0 + s_lane[96];
                ex.hw = area0 + s_lane[128];
                const int x_no = done / prm.E - 1;
                ok = ex.swap(prm.x, l, lw, x_no, g == prm.inject_warp && x_no >= prm.inject_exchange);
                if (!ok) {
                    latch_error(prm.x.err, kDevTimeoutFlag, g, k, 1);
                    break;
                }
            }
            n0 = n0_next;
            len = len_next;
        }
        // (a sweep that was given up has a part's copies on the way)
        asm volatile("cp.async.wait_all;" ::: "memory");
        double sum = acc;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(kFull, sum, o);
        if (lane == 0) prm.sums[g] = sum;
    }
    cluster_sync();
    if constexpr (TM) {
        tmem_fence_before_sync();
        __syncthreads();
        if (warp == 0) {
            tmem_fence_after_sync();
            tmem_dealloc(s_tmem, radj_columns(nwarp, P, SA));
        }
    }
}

struct Entry {
    int dtype, form, P, SA;
    bool tm;
    int warps;
    const void* fn;
};

template <typename Real, int FORM, int P, int SA, bool TM>
Entry entry()
{
    return Entry{sizeof(Real) == 8 ? kF64 : kF32, FORM, P, SA, TM, radj_max_warps<Real>(P),
                 reinterpret_cast<const void*>(&resident_adjoint_kernel<Real, FORM, P, SA, TM>)};
}

const Entry* table(int* n)
{
    static const Entry entries[] = {
        entry<float, kIncrement, 8, 16, true>(),  entry<float, kIncrement, 16, 8, true>(),
        entry<double, kCanonical, 2, 8, false>(), entry<double, kCanonical, 4, 8, false>(),
        entry<double, kCanonical, 8, 8, false>(),
    };
    *n = (int)(sizeof(entries) / sizeof(entries[0]));
    return entries;
}

}  // namespace

int radj_variants()
{
    int n;
    table(&n);
    return n;
}

void radj_info(int v, int* dtype, int* form, int* P, int* SA, int* max_warps)
{
    int n;
    const Entry& e = table(&n)[v];
    *dtype = e.dtype;
    *form = e.form;
    *P = e.P;
    *SA = e.SA;
    *max_warps = e.warps;
}

size_t radj_smem_bytes(int v, int H, int warps, int* values)
{
    int n;
    const Entry& e = table(&n)[v];
    const size_t es = e.dtype == kF64 ? 8 : 4;
    const size_t one = ((size_t)128 * e.P + 8 * H + (e.tm ? 0 : (size_t)e.SA * 32 * e.P) + 64 + 64 * e.P +
                        (kExchangeBytes + 5 * 32 * sizeof(int)) / es + 3) / 4 * 4;
    *values = (int)one;
    size_t b = one * warps * es;
    // more than half of an SM's: one CTA per SM (its tensor memory allocation never waits)
    if (e.tm && b < (size_t)120 * 1024) b = (size_t)120 * 1024;
    return b;
}

cudaError_t radj_fits(int v, size_t smem, bool* ok)
{
    int n;
    const Entry& e = table(&n)[v];
    *ok = false;
    int dev = 0, per_block = 0;
    cudaError_t st = cudaGetDevice(&dev);
    if (st == cudaSuccess) st = cudaDeviceGetAttribute(&per_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (st != cudaSuccess) return st;
    per_block -= 2048;
    if (smem > (size_t)per_block) return cudaSuccess;
    st = cudaFuncSetAttribute(e.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, per_block);
    *ok = st == cudaSuccess;
    return st;
}

cudaError_t radj_launch(int v, const void* params, int grid, int threads, size_t smem, bool cluster, cudaStream_t s)
{
    int n;
    const Entry& e = table(&n)[v];
    return res_launch_kernel(e.fn, params, grid, threads, smem, cluster, s);
}

cudaError_t radj_clusters(int v, int grid, int threads, size_t smem, int* clusters)
{
    int n;
    const Entry& e = table(&n)[v];
    return res_kernel_clusters(e.fn, grid, threads, smem, clusters);
}

}  // namespace rswr
