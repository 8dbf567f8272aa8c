"""The work that a user of this library has it do, as timed cases.

A case is a dict of plain values:

  kind      "run"         Plan.run: the forward problem (states, receiver, interface waveforms, point sources)
            "grad_fA"     Plan.adjoint / Batch.adjoint: the boundary-waveform gradient of a receiver misfit
            "grad"        Plan.adjoint with dL/da
            "train"       RSWRFunction: a forward run and the gradients of f_A and a through torch.autograd
            "paper"       Plan.run_paper: the paper-literal method, spans chosen from the data
            "batch"       Batch.run: many uneven problems in one call
  dtype     "f32" / "f64"
  nx, n_sub, overlap, cfl, a, T
  problems, nx_lo, nx_hi, table   (batches) problem count, range of the grid sizes, seed of the table of sizes
  state     a smooth wave field on the whole grid as the initial state (else zero data, as the paper's problem)
  fB        a driven right end (else f_B = 0)
  traces    the interface output waveforms, recv: a receiver trace, sources: so many interior pulse sources
  tune      autotune(tune) once when the plan is made, as the library's bench does for its large workloads
            (0: the plan as it is created)

Sizes are those of the library's own workloads (inputs.py) and tests, with the
step counts of the large ones cut down (the work is the same every step).
"""
import math

import numpy as np
import torch

from paper_2203_10477_gb300 import rswr

SUB_LEN = 2048  # points per subdomain of the batch workloads


def listed():
    base = {"kind": "run", "dtype": "f32", "cfl": 0.9, "a": 1.0, "state": False, "fB": False, "traces": False,
            "recv": False, "sources": 0, "tune": 0}

    def case(name, **kw):
        return dict(base, name=name, **kw)

    return [
        # the two-subdomain verification problem (nx = 1001, overlap 16, FP64) with everything recorded:
        # the smallest call, made often (parameter studies, checks); latency counts
        case("c1_f64", dtype="f64", nx=1001, n_sub=2, overlap=16, cfl=0.5, T=2000, traces=True, recv=True),
        # one shot of a small FP32 model, both ends driven, receiver recorded (inner loop of an inversion)
        case("shot_8k_f32", nx=8001, n_sub=4, overlap=32, T=2000, state=True, fB=True, recv=True),
        # a medium odd-sized grid, long run, interface waveforms on (the FP32 accuracy workload of the tests)
        case("line_60k_f32", nx=60001, n_sub=30, overlap=64, T=5000, state=True, traces=True),
        # the same kind of run in FP64 on a ragged grid (S = 24), resumed from a state, right end driven
        case("line_200k_f64", dtype="f64", nx=200003, n_sub=48, overlap=48, T=512, state=True, fB=True, recv=True),
        # the one-million-point grid of the gradient workload, forward only, tuned as its bench does
        case("grid_1m_f32", nx=1 << 20, n_sub=256, overlap=64, a=1.3, T=2048, state=True, recv=True, tune=512),
        # the large workload in both precisions: 2^24 points, 1024 subdomains, all interface waveforms
        case("c2_f64", dtype="f64", nx=1 << 24, n_sub=1024, overlap=64, T=320, state=True, traces=True, tune=96),
        case("c2_f32", nx=(1 << 24) - 3, n_sub=1024, overlap=64, T=1280, state=True, traces=True, tune=96),
        # ten pulse sources inside the domain (the paper's second experiment), FP32
        case("pulse10_f32", nx=1 << 22, n_sub=10, overlap=64, T=1000, sources=10, recv=True),
        # the paper-literal method on a 4M-point grid
        case("paper_4m_f32", kind="paper", nx=1 << 22, n_sub=256, overlap=64, T=500, state=True),
        # many uneven independent problems in one call (overlap 32), receivers recorded
        case("batch_512_f32", kind="batch", problems=512, nx_lo=1 << 10, nx_hi=1 << 18, table=10477, overlap=32,
             cfl=0.8, T=512, state=True, recv=True, tune=64),
        # one training step: forward run, then the gradients of the boundary waveform and the wave speed
        case("train_1m_f32", kind="train", nx=1 << 20, n_sub=256, overlap=64, a=1.3, T=2048, tune=512),
        # the same gradients in FP64 on a ragged grid
        case("grad_64k_f64", kind="grad", dtype="f64", nx=65539, n_sub=32, overlap=64, a=1.3, T=2048),
    ]


# ---- drawn cases --------------------------------------------------------------

_CAP = {"f32": 3.0e10, "f64": 5.0e9}  # grid-point updates of a drawn case (the largest listed ones hold more)


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "batch", "grad_fA", "grad", "train", "paper"])
    dtype = rng.choice(["f32", "f32", "f64"])
    c = {"kind": kind, "dtype": dtype, "cfl": round(rng.uniform(0.5, 0.95), 3), "a": round(rng.uniform(0.5, 2.0), 3),
         "overlap": rng.randint(16, 64), "state": False, "fB": False, "traces": False, "recv": False, "sources": 0,
         "tune": 0}
    if kind == "batch" or (kind == "grad_fA" and rng.random() < 0.5):
        c["problems"] = _logint(rng, 8, 512)
        c["nx_lo"], c["nx_hi"] = 1 << 10, _logint(rng, 1 << 13, 1 << 18)
        c["table"] = rng.randint(0, 1 << 30)
        points = c["problems"] * (c["nx_lo"] + c["nx_hi"]) / 2
        c["T"] = _logint(rng, 128, max(128, min(2048, _CAP[dtype] / 2 / points)))
        c["state"] = kind == "batch" and rng.random() < 0.7
        c["recv"] = kind == "batch" and rng.random() < 0.5
        return c
    top = {"run": 1 << 24, "paper": 1 << 22, "grad_fA": 1 << 20, "grad": 1 << 19, "train": 1 << 20}[kind]
    low = 4001 if kind == "paper" else 1001
    c["nx"] = _logint(rng, low, top)
    work = _CAP[dtype] / (4 if kind in ("grad", "train", "paper") else 1)
    c["T"] = _logint(rng, 100, max(101, min(5000 if kind == "run" else 2048, work / c["nx"])))
    c["n_sub"] = max(1, c["nx"] // _logint(rng, 500, 16384))
    if kind == "run":
        c["state"] = rng.random() < 0.7
        c["fB"] = rng.random() < 0.5
        c["recv"] = rng.random() < 0.5
        c["traces"] = c["n_sub"] > 1 and rng.random() < 0.5 and (c["n_sub"] - 1) * c["T"] < 8e6
        c["sources"] = rng.choice([0, 0, rng.randint(1, 10)])
        c["tune"] = 64 if c["nx"] >= 1 << 22 and rng.random() < 0.5 else 0
    elif kind == "paper":
        c["state"] = rng.random() < 0.7
    return c


# ---- inputs ---------------------------------------------------------------------

def _td(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _waveform(rows, T, g, scale=1.0):
    """Band-limited waveforms (bins above a tenth of Nyquist removed), starting at 0."""
    x = torch.randn(rows, T + 1, dtype=torch.float64, device="cuda", generator=g)
    F = torch.fft.rfft(x)
    F[:, F.shape[1] // 10 + 1:] = 0
    w = torch.fft.irfft(F, n=T + 1)
    ramp = 1.0 - torch.exp(-(torch.arange(T + 1, dtype=torch.float64, device="cuda") / 20.0) ** 2)
    return scale * 3.0 * w * ramp


def _sizes(case):
    r = np.random.Generator(np.random.PCG64(case["table"]))
    nx = r.integers(case["nx_lo"], case["nx_hi"], size=case["problems"], endpoint=True)
    a = r.uniform(0.5, 2.0, size=case["problems"])
    return [int(n) for n in nx], [float(x) for x in a]


class _Problem:
    def __init__(self, nx, a, dt, n_sub, overlap):
        self.nx, self.a, self.dt, self.n_sub, self.overlap, self.xa, self.xb = nx, a, dt, n_sub, overlap, 0.0, 1.0


def _problems(case):
    """The problems of a case (one for a plan), unit interval, dt from the Courant number."""
    if "problems" in case:
        nxs, speeds = _sizes(case)
        subs = [max(1, n // SUB_LEN) for n in nxs]
    else:
        nxs, speeds, subs = [case["nx"]], [case["a"]], [case["n_sub"]]
    return [_Problem(n, a, case["cfl"] / (n - 1) / a, s, case["overlap"]) for n, a, s in zip(nxs, speeds, subs)]


def _field(nx, cfl, g):
    """A packet-free smooth wave field (wavelengths of 60 to 600 points) at two consecutive levels, 0 at both ends."""
    x = torch.arange(nx, dtype=torch.float64, device="cuda")
    env = torch.clamp(torch.minimum(x, nx - 1 - x) / min(200.0, nx / 4), max=1.0)
    u, um = torch.zeros_like(x), torch.zeros_like(x)
    wl = 60.0 * 10.0 ** torch.rand(4, dtype=torch.float64, device="cuda", generator=g)
    ph = 2 * math.pi * torch.rand(4, dtype=torch.float64, device="cuda", generator=g)
    for q in range(4):
        k = 2 * math.pi / wl[q]
        s = cfl if q % 2 else -cfl  # right- and left-going parts
        u += 0.5 * torch.sin(k * x + ph[q])
        um += 0.5 * torch.sin(k * (x + s) + ph[q])
    return env * u, env * um


def _inputs(case, seed):
    g = _gen(seed)
    T, td = case["T"], _td(case)
    probs = _problems(case)
    n, d = len(probs), {}
    d["fA"] = _waveform(n, T, g).to(td)
    d["fB"] = _waveform(n, T, g, 0.7).to(td) if case["fB"] else None
    d["q0"] = d["q1"] = None
    if case["state"]:
        if n == 1:
            u, um = _field(probs[0].nx, case["cfl"], g)
        else:
            # one field per size would be slow to make: cut the problems out of one long field
            lens = [p.nx for p in probs]
            u, um = _field(sum(lens), case["cfl"], g)
        d["q0"] = u.to(td)
        # second component: u at the level before (FP64, canonical form), the increment (FP32, increment form)
        d["q1"] = (um if case["dtype"] == "f64" else u - um).to(td)
    r = np.random.Generator(np.random.PCG64(int(seed)))
    reach = max(1, int(T * 0.4))
    d["j_r"] = [int(r.integers(1, max(2, min(p.nx - 1, reach if "grad" in case["kind"] or case["kind"] == "train"
                                             else p.nx - 1)))) for p in probs]
    d["wbar"] = _waveform(n, T, g).to(td) if case["kind"] in ("grad_fA", "grad", "train") else None
    if case["sources"]:
        K, nx = case["sources"], probs[0].nx
        s, A = r.uniform(0.0, 1.0, K), r.uniform(-1.0, 1.0, K)
        lv = np.arange(T + 1, dtype=np.float64)
        d["src_j"] = [int((2 * q + 1) * (nx - 1) // (2 * K)) for q in range(K)]
        if not case["state"]:  # a receiver that the first source's waves reach
            d["j_r"] = [min(nx - 2, d["src_j"][0] + int(r.integers(1, reach + 1)))]
        d["src"] = torch.as_tensor(np.stack([A[q] / 30.0 * np.exp(-((lv - (4 + 2 * s[q]) * 30.0) / 30.0) ** 2)
                                             for q in range(K)]), device="cuda").to(td)
    return probs, d


def prepare(case, seed):
    probs, d = _inputs(case, seed)
    dt = rswr.F64 if case["dtype"] == "f64" else rswr.F32
    if "problems" in case:
        h = rswr.Batch(probs, dtype=dt)
    else:
        h = rswr.Plan.from_problem(probs[0], dtype=dt)
    if case["tune"]:
        h.autotune(case["tune"])
    if case["sources"]:
        h.set_sources(d["src_j"], d["src"])
    st = {"case": case, "h": h, "d": d}
    if "problems" not in case:
        d["fA"] = d["fA"][0].contiguous()
        d["fB"] = None if d["fB"] is None else d["fB"][0].contiguous()
        d["wbar"] = None if d["wbar"] is None else d["wbar"][0].contiguous()
    if case["kind"] == "train":
        st["fA"] = d["fA"].clone().requires_grad_(True)
        st["a"] = torch.tensor([case["a"]], dtype=torch.float64, device="cuda", requires_grad=True)
        st["fn"] = rswr.rswr_function()
    return st


def run(st):
    c, h, d = st["case"], st["h"], st["d"]
    k, T = c["kind"], c["T"]
    if k == "run":
        r = h.run(d["fA"], d["fB"], T, q0=d["q0"], q1=d["q1"], traces=c["traces"], j_r=d["j_r"][0] if c["recv"] else None)
        return [r["u"], r["w"], r["traces"], r["recv"]]
    if k == "batch":
        r = h.run(d["fA"], d["fB"], T, q0=d["q0"], q1=d["q1"], j_r=d["j_r"] if c["recv"] else None)
        return [r["u"], r["w"], r["recv"]]
    if k == "paper":
        r = h.run_paper(d["fA"], d["fB"], T, q0=d["q0"], q1=d["q1"])
        return [r["u"], r["w"], r["spans"]]
    if k in ("grad_fA", "grad"):
        r = h.adjoint(d["fA"], d["fB"], T, d["j_r"] if "problems" in c else d["j_r"][0], d["wbar"], want_a=k == "grad")
        return [r["grad_fA"], r["grad_a"]]
    y = st["fn"].apply(st["fA"], st["a"], h, T, d["j_r"][0])
    gf, ga = torch.autograd.grad(y, (st["fA"], st["a"]), d["wbar"])
    return [y.detach(), gf, ga]


def work(case):
    nxs = _sizes(case)[0] if "problems" in case else [case["nx"]]
    es, T, k = (8 if case["dtype"] == "f64" else 4), case["T"], case["kind"]
    points = sum(nxs)
    rows = len(nxs)
    flops = 5.0 * points * T  # one update: five operations in either form
    if k in ("grad_fA", "grad"):
        by = 2.0 * es * rows * (T + 1)
        if k == "grad":
            by += es * rows * (T + 1)
            flops = 13.0 * points * T  # forward and adjoint updates, the Laplacian's own operation and the pairing
    elif k == "train":
        by, flops = 4.0 * es * (T + 1), 13.0 * points * T
    else:
        by = es * ((4.0 if case["state"] else 2.0) * points + rows * (T + 1) * (2 if case["fB"] else 1))
        if case["traces"]:
            by += es * 2.0 * (case["n_sub"] - 1) * (T + 1)
        if case["recv"]:
            by += es * float(rows) * (T + 1)
        by += es * float(case["sources"]) * (T + 1)
    return {"bytes": by, "flops": flops}


# ---- the same results in plain 64-bit torch -------------------------------------------

def _leapfrog(nxs, c2s, fA, fB, T, q0=None, um=None, rec=None, src=None, keep_lap=False):
    """u^T, u^{T-1}, the levels 0..T of the points `rec` (packed indices) and, if asked, the Laplacians of levels 0..T-1."""
    dev, off = "cuda", np.concatenate([[0], np.cumsum(nxs)])
    L = torch.as_tensor(off[:-1], device=dev)
    R = torch.as_tensor(off[1:] - 1, device=dev)
    n = int(off[-1])
    u = torch.zeros(n, dtype=torch.float64, device=dev) if q0 is None else q0.clone()
    p = u.clone() if um is None else um.clone()
    zero = torch.zeros_like(fA)
    fB = zero if fB is None else fB
    u[L], u[R] = fA[:, 0], fB[:, 0]
    p[L], p[R] = fA[:, 0], fB[:, 0]
    one = len(nxs) == 1
    c2 = c2s[0] if one else torch.repeat_interleave(torch.tensor(c2s, dtype=torch.float64, device=dev),
                                                    torch.as_tensor(np.asarray(nxs), device=dev))[1:-1]
    out = None if rec is None else torch.empty(T + 1, len(rec), dtype=torch.float64, device=dev)
    laps = []
    for t in range(T + 1):
        if out is not None:
            out[t] = u[rec]
        if t == T:
            break
        lap = u[2:] + u[:-2]
        lap.sub_(u[1:-1], alpha=2.0)
        if keep_lap:
            laps.append(lap)
        m = p[1:-1]
        m.neg_().add_(u[1:-1], alpha=2.0)
        if one:
            m.add_(lap, alpha=c2)
        else:
            m.addcmul_(c2, lap)
        p[L], p[R] = fA[:, t + 1], fB[:, t + 1]
        if src is not None:
            p.index_add_(0, src[0], src[1][:, t + 1])
        u, p = p, u
    return u, p, out, laps


def _adjoint(nxs, c2s, wbar, j_r, T, laps=None):
    """grad_fA per problem and, with the forward Laplacians of one problem, dL/dc2."""
    off = np.concatenate([[0], np.cumsum(nxs)])
    n, dev = int(off[-1]), "cuda"
    L = torch.as_tensor(off[:-1], device=dev)
    R = torch.as_tensor(off[1:] - 1, device=dev)
    at = torch.as_tensor(off[:-1] + np.asarray(j_r), device=dev)
    c2v = torch.tensor(c2s, dtype=torch.float64, device=dev)
    c2 = torch.repeat_interleave(c2v, torch.as_tensor(np.asarray(nxs), device=dev))
    lam, nxt = torch.zeros(n, dtype=torch.float64, device=dev), torch.zeros(n, dtype=torch.float64, device=dev)
    lam.index_add_(0, at, wbar[:, T])  # level T
    lam[L], lam[R] = 0, 0
    g = torch.zeros(len(nxs), T + 1, dtype=torch.float64, device=dev)
    dc2 = torch.zeros((), dtype=torch.float64, device=dev)
    for t in range(T - 1, -1, -1):
        g[:, t] = c2v * lam[L + 1]
        if laps is not None:
            dc2 += torch.dot(lam[1:-1], laps[t])
        lap = lam[2:] + lam[:-2]
        lap.sub_(lam[1:-1], alpha=2.0)
        m = nxt[1:-1]
        m.neg_().add_(lam[1:-1], alpha=2.0).addcmul_(c2[1:-1], lap)
        nxt.index_add_(0, at, wbar[:, t])
        nxt[L], nxt[R] = 0, 0
        lam, nxt = nxt, lam
    return g, dc2


def exact(case, seed):
    probs, d = _inputs(case, seed)
    T, k = case["T"], case["kind"]
    nxs, c2s = [p.nx for p in probs], [(p.a * p.dt * (p.nx - 1)) ** 2 for p in probs]
    D = lambda x: None if x is None else x.double()  # noqa: E731
    fA, fB = D(d["fA"]), D(d["fB"])
    if k in ("grad_fA", "grad", "train"):
        # zero data and a quiet right end: nothing beyond what the cone of T steps reaches enters the gradients
        cut = [min(p.nx, j + T + 8) for p, j in zip(probs, d["j_r"])]
        laps, recv = None, None
        if k != "grad_fA":
            _, _, out, laps = _leapfrog(cut, c2s, fA, None, T, rec=torch.tensor(d["j_r"], device="cuda"), keep_lap=True)
            recv = out[:, 0]
        g, dc2 = _adjoint(cut, c2s, D(d["wbar"]), d["j_r"], T, laps)
        one = g if "problems" in case else g[0]
        if k == "grad_fA":
            return [one, None]
        ga = (dc2 * 2.0 * c2s[0] / case["a"]).reshape(1)
        return [one, ga] if k == "grad" else [recv, one, ga]
    q0, um = D(d["q0"]), None
    if q0 is not None:
        um = D(d["q1"]) if case["dtype"] == "f64" else q0 - D(d["q1"])
    off = np.concatenate([[0], np.cumsum(nxs)])
    rec, ntr = [], 0
    if case["traces"]:
        n, N, ov = nxs[0], case["n_sub"], case["overlap"]
        for i in range(N - 1):
            b = (i + 1) * n // N
            for j in (max(b - (ov + 1) // 2, 0), min(b - 1 + ov // 2, n - 1)):
                rec += [j - 1, j + 1]
        ntr = len(rec)
    if case["recv"]:
        rec += [int(o) + j for o, j in zip(off[:-1], d["j_r"])]
    src = None
    if case["sources"]:
        src = (torch.tensor(d["src_j"], device="cuda"), D(d["src"]))
    u, p, out, _ = _leapfrog(nxs, c2s, fA, fB, T, q0, um, torch.tensor(rec, device="cuda") if rec else None, src)
    w = p if case["dtype"] == "f64" else u - p
    if k == "paper":
        return [u, w, None]
    recv = None
    if case["recv"]:
        recv = out[:, ntr:].T.contiguous()
        recv = recv if k == "batch" else recv[0]
    if k == "batch":
        return [u, w, recv]
    tr = None
    if case["traces"]:
        flux = (out[:, 1:ntr:2] - out[:, 0:ntr:2]) * (0.5 * (nxs[0] - 1))
        tr = flux.T.reshape(case["n_sub"] - 1, 2, T + 1)
    return [u, w, tr, recv]
