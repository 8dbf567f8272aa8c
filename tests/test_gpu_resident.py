"""Resident warp windows (csrc/resident.cuh): grids that fit on the chip, at the
sizes where the cut into pieces can go wrong, bit for bit against the CPU
oracle: one piece, two pieces, a ragged last piece, pieces of the smallest
length, one cluster and several CTAs through L2, chunks of several spans, run
lengths on and off a chunk's end, probes on the nodes, next to them and on the
pieces' ends, sources alone in a window, next to a node and several at once."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2203_10477_gb300 import inputs

pytestmark = pytest.mark.gpu

F32, F64 = 0, 1


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_10477_gb300 import build, rswr

    build.build()
    return rswr


def host(t):
    return t.detach().cpu().numpy()


def same(a, b, what):
    bad = np.flatnonzero(np.asarray(a).ravel() != np.asarray(b).ravel())
    assert bad.size == 0, f"{what}: {bad.size} values differ, first at {bad[:5]}"


def problem(oracle_mod, dtype, nx, T, seed=3):
    dt_ = np.float64 if dtype == F64 else np.float32
    dt = 0.9 / (nx - 1)
    r = inputs.rng(seed)
    fA = (0.5 + r.standard_normal(T + 1)).astype(dt_)
    fB = (r.standard_normal(T + 1) - 0.3).astype(dt_)
    q0 = r.standard_normal(nx).astype(dt_)
    q1 = (0.1 * r.standard_normal(nx)).astype(dt_)
    return dt, fA, fB, q0, q1, dict(form=0 if dtype == F64 else 1, prec="f64" if dtype == F64 else "f32")


# overlaps 16, 33, 48, 64: chunks of several spans, odd spans, one span
@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("nx,ov,T", [
    (5, 2, 9), (40, 16, 64), (63, 16, 65), (64, 16, 1), (65, 33, 48), (193, 33, 33), (255, 48, 128), (257, 64, 64),
    (449, 64, 97), (1001, 16, 129), (4099, 48, 200), (8001, 64, 131), (20011, 33, 70), (60001, 64, 96),
])
def test_plan_as_created_equals_oracle(R, oracle_mod, dtype, nx, ov, T):
    dt, fA, fB, q0, q1, kw = problem(oracle_mod, dtype, nx, T)
    N = 3 if nx // 3 >= ov else 1
    plan = R.Plan(0.0, 1.0, 1.0, nx, dt, N, ov, dtype=dtype)
    rs = oracle_mod.rswr_mask(nx, T, 1.0, dt, fA, fB, N, ov, q0=q0, q1=q1, **kw) if N > 1 else None
    for jr in sorted({0, 1, nx // 2, nx - 2, nx - 1}):
        ref = oracle_mod.leapfrog(nx, T, 1.0, dt, fA, fB, q0=q0, q1=q1, rec_j=[jr], **kw)
        out = plan.run(fA, fB, T, q0=q0, q1=q1, traces=N > 1, j_r=jr)
        plan.check()
        same(host(out["u"]), ref["u"], f"u (receiver {jr})")
        same(host(out["w"]), ref["w"], "w")
        same(host(out["recv"]), ref["rec"][0], f"receiver {jr}")
        if N > 1:
            same(host(out["traces"]), rs["traces"], "traces")


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("S", [1, 5, 14, 30, 32])
def test_every_resident_variant_and_probe_position(R, oracle_mod, dtype, S):
    """A receiver on every point around the pieces' ends (a window of 300 points
    covers the ends of several pieces of the narrow variants)."""
    nx, T = 2003, 67
    dt, fA, fB, q0, q1, kw = problem(oracle_mod, dtype, nx, T, seed=S)
    js = list(range(0, 300, 7)) + [1, 2, nx - 3, nx - 2, nx - 1]
    ref = oracle_mod.leapfrog(nx, T, 1.0, dt, fA, fB, q0=q0, q1=q1, rec_j=js, **kw)
    for v in [v for v in R.variants() if v["dtype"] == dtype and v["resident"] and v["max_span"] >= S]:
        plan = R.Plan(0.0, 1.0, 1.0, nx, dt, 1, 64, dtype=dtype)
        plan.set_span(S)
        plan.set_variant(v["variant"])
        for i, j in enumerate(js):
            if i % 8 and j not in (0, 1, nx - 2, nx - 1):
                continue
            out = plan.run(fA, fB, T, q0=q0, q1=q1, j_r=j)
            same(host(out["recv"]), ref["rec"][i], f"variant {v['variant']} receiver {j}")
        plan.check()
        same(host(out["u"]), ref["u"], f"variant {v['variant']} u")
        same(host(out["w"]), ref["w"], f"variant {v['variant']} w")


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("places", [[700], [1], [2001], [3, 1500], [700, 700, 701], list(range(690, 700)), [0, 2002, 900]])
def test_sources_in_resident_windows(R, oracle_mod, dtype, places):
    nx, T = 2003, 97
    dt, fA, fB, q0, q1, kw = problem(oracle_mod, dtype, nx, T, seed=8)
    s = inputs.rng(4).standard_normal((len(places), T + 1)).astype(q0.dtype)
    plan = R.Plan(0.0, 1.0, 1.0, nx, dt, 1, 48, dtype=dtype)
    plan.set_sources(places, s)
    out = plan.run(fA, fB, T, q0=q0, q1=q1, j_r=places[0])
    plan.check()
    ref = oracle_mod.leapfrog(nx, T, 1.0, dt, fA, fB, q0=q0, q1=q1, rec_j=[places[0]],
                              src_j=np.asarray(places, np.int64), src=s, **kw)
    same(host(out["u"]), ref["u"], "u")
    same(host(out["w"]), ref["w"], "w")
    same(host(out["recv"]), ref["rec"][0], "receiver")


def test_grids_just_above_the_capacity_still_run(R, oracle_mod):
    """A resident variant chosen by the caller, or remembered from a smaller grid of
    the same size class by the autotuner, on a grid that does not fit at once."""
    nx, T = 1400003, 40
    dt, fA, fB, q0, q1, kw = problem(oracle_mod, F32, nx, T)
    ref = oracle_mod.leapfrog(nx, T, 1.0, dt, fA, fB, q0=q0, q1=q1, **kw)
    R.Plan(0.0, 1.0, 1.0, 1 << 20, dt, 64, 60, dtype=F32).autotune(64)
    for v in [None] + [v["variant"] for v in R.variants() if v["dtype"] == F32 and v["resident"]]:
        plan = R.Plan(0.0, 1.0, 1.0, nx, dt, 64, 60, dtype=F32)
        plan.set_span(30)
        if v is None:
            plan.autotune(64)
        else:
            plan.set_variant(v)
        out = plan.run(fA, fB, T, q0=q0, q1=q1)
        plan.check()
        same(host(out["u"]), ref["u"], f"variant {v} u")
        same(host(out["w"]), ref["w"], f"variant {v} w")
