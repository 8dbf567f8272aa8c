"""The paper-literal run of FP32 plans in one launch (csrc/paper_kernel.cu) at the
sizes where its windows change -- the widest overlaps of 8 and 16 points per
lane and the first beyond, spans that leave a re-solve window 64 points, one
subdomain, the smallest cores, bulk windows of 256 and 1024 points, more
pieces than warps -- bit for bit against the paper's rule written out in
NumPy, every window solved whole, with correctly rounded FP32 operations."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2203_10477_gb300 import inputs

CAN, INC = 1, 2
f32, f64 = np.float32, np.float64


def fma32(a, b, c):
    """round32(a b + c): the product is exact in FP64; the sum is rounded to odd
    there (its last bit set when inexact), so that rounding it again is harmless."""
    p, c = f64(a) * np.asarray(b, f64), np.asarray(c, f64)
    s = p + c
    t = s - p
    err = (p - (s - t)) + (c - t)
    even = (np.ascontiguousarray(s).view(np.int64) & 1) == 0
    toward = np.nextafter(s, np.where(err > 0, np.inf, -np.inf))
    return np.where((err != 0) & even, toward, s).astype(f32)


class Rule:
    def __init__(self, form, nx, c2, k, two_dx, fA, fB):
        self.__dict__.update(locals())

    def solve(self, u, w, lo, hi, n0, steps, gL=None, gR=None, seen=None):
        """The window [lo, hi] from the state (u, w) over `steps` steps; gL / gR:
        input fluxes (None: zero-flux mirror); seen(s, u, w) before each step."""
        u, w = u[lo:hi + 1].copy(), w[lo:hi + 1].copy()
        for s in range(steps):
            if seen:
                seen(s, u, w)
            ul, ur = np.concatenate([u[1:2], u[:-1]]), np.concatenate([u[1:], u[-2:-1]])
            if gL is not None:
                ul[0] = u[1] - self.two_dx * gL[s]
            if gR is not None:
                ur[-1] = u[-2] + self.two_dx * gR[s]
            if self.form == CAN:
                un = fma32(self.c2, ul + ur, fma32(self.k, u, -w))
                wn = u.copy()
            else:
                wn = fma32(self.c2, (ul - u) + (ur - u), w)
                un = u + wn
            for at, j, f in ((0, lo, self.fA), (-1, hi, self.fB)):
                if j == (0 if at == 0 else self.nx - 1):
                    un[at] = f[n0 + s + 1]
                    wn[at] = f[n0 + s] if self.form == CAN else f[n0 + s + 1] - f[n0 + s]
            u, w = un, wn
        if seen:
            seen(steps, u, w)
        return u, w


def paper_rule(rule, N, ov, cfl, T, u, w):
    nx, el, er = rule.nx, (ov + 1) // 2, ov // 2
    L = [max(i * nx // N - el, 0) for i in range(N)]
    R = [min((i + 1) * nx // N - 1 + er, nx - 1) for i in range(N)]
    cap = max(1, math.ceil((ov - 1) / (2 * cfl)) - 1)
    n0, tau, spans = 0, ov, []
    while n0 < T:
        steps = min(tau, T - n0)
        gL, gR, span = [None] * N, [None] * N, steps
        rec = []
        for i in range(N):
            x = []
            rule.solve(u, w, L[i], R[i], n0, steps, seen=lambda s, a, b: x.append(a.copy()))
            rec.append(np.array(x))
        for i in range(N - 1):
            a, b = rec[i], rec[i + 1]
            gL[i + 1] = (a[:, L[i + 1] + 1 - L[i]] - a[:, L[i + 1] - 1 - L[i]]) / rule.two_dx
            gR[i] = (b[:, R[i] + 1 - L[i + 1]] - b[:, R[i] - 1 - L[i + 1]]) / rule.two_dx
            same = a[1:, L[i + 1] - L[i]:] == b[1:, :R[i] - L[i + 1] + 1]
            span = min(span, int(np.logical_and.accumulate(same, axis=0).sum(axis=0).max()))
        span = max(1, min(span, cap))
        nu, nw = np.empty_like(u), np.empty_like(w)
        start = 0
        for i in range(N):
            a, b = rule.solve(u, w, L[i], R[i], n0, span, gL[i], gR[i])
            nu[start:R[i] + 1], nw[start:R[i] + 1] = a[start - L[i]:], b[start - L[i]:]
            start = R[i] + 1
        u, w = nu, nw
        spans.append(span)
        n0 += span
        tau = (span * 1100 + 999) // 1000
    return u, w, spans


@pytest.mark.gpu
@pytest.mark.parametrize("nx,N,ov,cfl,T", [
    (900, 4, 76, 0.9, 100),
    (900, 4, 77, 0.9, 100),
    (1801, 4, 154, 0.9, 200),
    (1801, 4, 155, 0.9, 200),     # (beyond: the span-by-span kernels)
    (2001, 8, 12, 0.057, 300),
    (2001, 8, 13, 0.057, 300),
    (301, 1, 16, 0.5, 50),
    (50, 25, 2, 0.9, 30),
    (9001, 3, 64, 0.9, 35),       # a run of one full span and one step
    (40001, 400, 33, 0.7, 60),
    (250001, 9, 40, 0.9, 50),     # bulk windows of 1024 points
    (2000001, 300, 48, 0.9, 27),  # more pieces than warps
])
@pytest.mark.parametrize("form", [CAN, INC])
def test_run_follows_the_rule(form, nx, N, ov, cfl, T):
    from paper_2203_10477_gb300 import build, rswr

    build.build()
    dt = cfl / (nx - 1)
    r = inputs.rng(nx + ov)
    fA, fB = r.standard_normal(T + 1).astype(f32), r.standard_normal(T + 1).astype(f32)
    q0, q1 = r.standard_normal(nx).astype(f32), r.standard_normal(nx).astype(f32)
    plan = rswr.Plan(0.0, 1.0, 1.0, nx, dt, N, ov, dtype=rswr.F32, form=form)
    got = plan.run_paper(fA, fB, T, q0=q0, q1=q1)
    info = plan.info()
    dx = 1.0 / (nx - 1)
    rule = Rule(form, nx, f32(info["c2f"]), f32(info["kf"]), f32(2.0 * dx), fA, fB)
    u, w = q0.copy(), q1.copy()
    u[0], u[-1] = fA[0], fB[0]
    w[0], w[-1] = (u[0], u[-1]) if form == CAN else (0, 0)
    u, w, spans = paper_rule(rule, N, ov, info["c"], T, u, w)
    assert list(got["spans"]) == spans
    assert np.array_equal(got["u"].cpu().numpy(), u)
    assert np.array_equal(got["w"].cpu().numpy(), w)
