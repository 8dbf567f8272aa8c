"""Free warp windows of the span kernel (csrc/span_kernel.cuh): a node, a source
and probes where a warp's window begins and ends, on a lane's first and last
registers, in halos only, two of them in one window, more probes than a warp
records by itself; spans off and on the record buffer's eight levels; bit for bit
against the CPU oracle on every such variant."""
from types import SimpleNamespace

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2203_10477_gb300 import inputs

pytestmark = pytest.mark.gpu

F32 = 0


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_10477_gb300 import build, rswr

    build.build()
    return rswr


def free_variants(R):
    return [v for v in R.variants() if v["dtype"] == F32 and not v.get("resident") and v["max_span"] > 0]


# nx relative to the tile's core: the last tile holds a few points, one warp's, nearly all
@pytest.mark.parametrize("tail", [3, 31, 705, -1])
@pytest.mark.parametrize("form", [1, 2])
def test_special_points_equal_oracle(R, oracle_mod, form, tail):
    todo = [v for v in free_variants(R) if v["form"] == form]
    assert todo
    for v in todo:
        P, KH = v["P"], v["KH"]
        S = min(KH, 32) - (5 if tail == 31 else 0)
        H = (S + 3) // 4 * 4
        core, cw = v["window"] - 2 * H, 32 * P - 2 * KH
        nx = 2 * core + tail
        N, T = 40, 3 * S + 7
        dt = 0.9 / (nx - 1)
        r = inputs.rng(nx + P)
        fA, fB = (r.standard_normal(T + 1).astype(np.float32) for _ in range(2))
        q0, q1 = (r.standard_normal(nx).astype(np.float32) for _ in range(2))
        at = core - H + cw  # the first point of the second tile's second warp
        for js in ([1], [nx - 2], [at], [at - 1], [at + 32 * P - 1], [at + KH + P], [core, core + 1],
                   [3, core + cw // 2, nx - 40]):
            js = [j for j in js if 0 < j < nx - 1]
            s = r.standard_normal((len(js), T + 1)).astype(np.float32)
            jr = min(max(js[0] + 1, 0), nx - 1)
            plan = R.Plan(0.0, 1.0, 1.0, nx, dt, N, 64, dtype=F32, form=form)
            plan.set_span(S)
            plan.set_variant(v["variant"])
            plan.set_sources(js, s)
            got = plan.run(fA, fB, T, q0=q0, q1=q1, traces=True, j_r=jr)
            ref = oracle_mod.rswr_mask(nx, T, 1.0, dt, fA, fB, N, 64, q0=q0, q1=q1, form=form - 1, prec="f32", src_j=js,
                                       src=s)
            mono = oracle_mod.leapfrog(nx, T, 1.0, dt, fA, fB, q0=q0, q1=q1, form=form - 1, prec="f32", rec_j=[jr],
                                       src_j=js, src=s)
            for a, b in (("u", ref["u"]), ("w", ref["w"]), ("traces", ref["traces"]), ("recv", mono["rec"][0])):
                bad = np.flatnonzero(got[a].cpu().numpy().ravel() != np.asarray(b).ravel())
                assert bad.size == 0, (v, js, a, bad[:5])


@pytest.mark.parametrize("ov", [4, 11, 16, 21, 32, 33, 63, 64])
def test_passes_of_several_spans_equal_oracle(R, oracle_mod, ov):
    """Overlaps below 64: a pass holds as many whole spans as 32 steps (ov // 2 steps
    each) for plans whose span the caller did not choose; tuned, batched, with
    a fault injected (one span to a pass again) and taken back."""
    nx, N, T = 9001, 40, 150
    dt = 0.9 / (nx - 1)
    r = inputs.rng(ov)
    fA, fB = (r.standard_normal(T + 1).astype(np.float32) for _ in range(2))
    q0, q1 = (r.standard_normal(nx).astype(np.float32) for _ in range(2))
    ref = oracle_mod.rswr_mask(nx, T, 1.0, dt, fA, fB, N, ov, q0=q0, q1=q1, form=1, prec="f32")
    S = ov // 2
    plan = R.Plan(0.0, 1.0, 1.0, nx, dt, N, ov, dtype=F32)
    plan.set_mode(1)  # (not the resident path)
    plan.set_variant(0)
    halos = []
    for step in range(3):
        plan.inject_missing_flag(2 if step == 1 else -1, 1 << 30)  # (a span that the run does not reach)
        halos.append(plan.info()["halo"])
        assert plan.info()["span_steps"] == S
        got = plan.run(fA, fB, T, q0=q0, q1=q1, traces=True)
        plan.check()
        for k in ("u", "w", "traces"):
            assert np.array_equal(got[k].cpu().numpy(), ref[k]), (k, step)
    assert halos == [(m + 3) // 4 * 4 for m in (32 // S * S, S, 32 // S * S)]
    plan.set_span(S)
    assert plan.info()["halo"] == (S + 3) // 4 * 4


@pytest.mark.parametrize("dtype", [0, 1])
def test_packing_of_uneven_problems(R, dtype):
    """No step: the initial pair comes back, for problems shorter than, as long as and
    longer than a block's 2048 points, with ends inside and on a block's edge."""
    sizes = [64, 1984, 2048, 3, 2045, 40000, 65, 6144, 2047, 2049, 5, 100000]
    probs = [SimpleNamespace(nx=n, xa=0.0, xb=1.0, a=1.0, dt=0.9 / (n - 1), n_sub=1, overlap=2) for n in sizes]
    b = R.Batch(probs, dtype=dtype)
    td = np.float64 if dtype else np.float32
    r = inputs.rng(2)
    q0, q1 = (r.standard_normal(sum(sizes)).astype(td) for _ in range(2))
    f = r.standard_normal((len(sizes), 1)).astype(td)
    got = b.run(f, f, 0, q0=q0, q1=q1)
    u, w = q0.copy(), q1.copy()
    at = 0
    for n in sizes:
        for j in (at, at + n - 1):
            u[j] = f[sizes.index(n), 0]
            w[j] = u[j] if dtype else 0
        at += n
    assert np.array_equal(got["u"].cpu().numpy(), u)
    assert np.array_equal(got["w"].cpu().numpy(), w)
