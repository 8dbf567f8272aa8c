"""Plans whose tiling changes between runs with the same arguments: a captured
run is not replayed on the arrays of an earlier tiling, and a plan on a resident
variant whose grid does not fit runs on a tiling of its own.  Bit for bit
against the CPU oracle."""
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


class Call:
    """The same tensors for every run, and the oracle's state."""

    def __init__(self, oracle_mod, dtype, nx, T, cfl=0.9):
        dt_ = np.float64 if dtype == F64 else np.float32
        r = inputs.rng(nx)
        self.dt, self.T = cfl / (nx - 1), T
        fA, q0, q1 = (r.standard_normal(n).astype(dt_) for n in (T + 1, nx, nx))
        kw = dict(form=0 if dtype == F64 else 1, prec="f64" if dtype == F64 else "f32")
        ref = oracle_mod.leapfrog(nx, T, 1.0, self.dt, fA, np.zeros(T + 1, dt_), q0=q0, q1=q1, **kw)
        dev = lambda x: torch.as_tensor(x, device="cuda")
        self.fA, self.q0, self.q1, self.u, self.w = map(dev, (fA, q0, q1, ref["u"], ref["w"]))
        self.out = (torch.empty_like(self.q0), torch.empty_like(self.q0))

    def run(self, plan, what):
        for o in self.out:
            o.fill_(7.0)
        plan.run(self.fA, None, self.T, q0=self.q0, q1=self.q1, out=self.out)
        plan.check()
        assert torch.equal(self.out[0], self.u) and torch.equal(self.out[1], self.w), what


@pytest.mark.parametrize("dtype", [F32, F64])
def test_no_replay_after_a_new_tiling(R, oracle_mod, dtype):
    nx = 300007
    c = Call(oracle_mod, dtype, nx, 40)
    plan = R.Plan(0.0, 1.0, 1.0, nx, c.dt, 16, 48, dtype=dtype)
    own = [v for v in R.variants() if v["dtype"] == dtype and v["form"] == plan.info()["form"]]
    S = plan.info()["span_steps"]
    own = [v for v in own if v["max_span"] == 0 or v["max_span"] >= S]
    tick = [v["variant"] for v in own if not v["resident"]]
    plan.set_variant(tick[0])  # (off the resident path: runs are captured)
    for rnd in range(2):
        c.run(plan, f"{rnd}: captured")
        c.run(plan, f"{rnd}: replayed")
        # to a narrower tiling (more tiles: larger tables) and back
        plan.set_variant(min(own, key=lambda v: v["window"])["variant"])
        plan.set_variant(tick[0])
        c.run(plan, f"{rnd}: after another variant")
        plan.set_span(1)
        plan.set_span(S)
        c.run(plan, f"{rnd}: after another span")
        plan.inject_missing_flag(0, 1 << 20)
        plan.inject_missing_flag(-1, 0)
        c.run(plan, f"{rnd}: after the hook was set and cleared")


def test_no_replay_after_a_resident_variant_that_does_not_fit(R, oracle_mod):
    nx = 1400003
    c = Call(oracle_mod, F32, nx, 40)
    plan = R.Plan(0.0, 1.0, 1.0, nx, c.dt, 64, 60, dtype=F32)
    c.run(plan, "as created")
    for v in [v["variant"] for v in R.variants() if v["dtype"] == F32 and v["resident"]]:
        plan.set_variant(v)
        c.run(plan, f"variant {v}")
        c.run(plan, f"variant {v} again")
    plan.set_variant(0)
    c.run(plan, "the first variant again")


@pytest.mark.parametrize("dtype", [F32, F64])
def test_resident_variant_runs_what_its_kernel_does_not_cover(R, oracle_mod, dtype):
    """A plan on a resident variant: spans longer than its windows take (FP64),
    probes over the initial state, a continued paper-literal run, and the plan's
    own runs between them, on one tiling that stays."""
    import ctypes

    nx, T, jr = 30011, 150, 15000
    c = Call(oracle_mod, dtype, nx, T)
    ov = 64 if dtype == F32 else 160
    plan = R.Plan(0.0, 1.0, 1.0, nx, c.dt, 3, ov, dtype=dtype)
    tiles = plan.info()["ntiles"]
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    ref = plan.run(c.fA, None, T, q0=c.q0, q1=c.q1, j_r=jr)["recv"]
    paper = plan.run_paper(c.fA, None, T, q0=c.q0, q1=c.q1)
    todo = [v for v in R.variants() if v["dtype"] == dtype and v["resident"] and v["max_span"] >= ov // 2]
    assert todo
    for v in todo:
        plan.set_variant(v["variant"])
        assert plan.info()["variant"] == v["variant"] and plan.info()["ntiles"] == tiles
        c.run(plan, v)
        u = c.q0.clone()
        rec = u[jr:jr + T + 1]
        R.check(R.lib().rswr_run(plan.h, p(c.fA), None, T, p(u), p(c.q1), p(c.out[0]), p(c.out[1]), None, jr, p(rec),
                                 torch.cuda.current_stream().cuda_stream))
        plan.check()
        assert torch.equal(rec, ref) and torch.equal(c.out[0], c.u), v
        got = plan.run_paper(c.fA, None, T, q0=c.q0, q1=c.q1)
        assert torch.equal(got["u"], paper["u"]) and list(got["spans"]) == list(paper["spans"]), v
        c.run(plan, v)


def test_grids_whose_windows_have_no_room_to_shift(R, oracle_mod):
    """Windows that fit the chip only without room to put a source or a probe on
    an end register."""
    nx, T = 1150001, 70
    c = Call(oracle_mod, F32, nx, T)
    plan = R.Plan(0.0, 1.0, 1.0, nx, c.dt, 64, 64, dtype=F32)
    c.run(plan, "nothing special")
    js = [1, 333333, nx // 2, nx - 2]
    s = inputs.rng(3).standard_normal((len(js), T + 1)).astype(np.float32)
    h = lambda t: t.cpu().numpy()
    for src in (None, js):
        plan.set_sources(src, s if src else None)
        kw = dict(src_j=np.asarray(js, np.int64), src=s) if src else {}
        ref = oracle_mod.leapfrog(nx, T, 1.0, c.dt, h(c.fA), np.zeros(T + 1, np.float32), q0=h(c.q0), q1=h(c.q1), form=1,
                                  prec="f32", rec_j=[0, 1, 333330, 333333, nx // 2 + 1, nx - 2, nx - 1], **kw)
        for i, jr in enumerate([0, 1, 333330, 333333, nx // 2 + 1, nx - 2, nx - 1]):
            got = plan.run(c.fA, None, T, q0=c.q0, q1=c.q1, j_r=jr)
            plan.check()
            assert np.array_equal(h(got["recv"]), ref["rec"][i]), (src, jr)
        assert np.array_equal(h(got["u"]), ref["u"]) and np.array_equal(h(got["w"]), ref["w"]), src


def test_fp64_resident_variants_take_every_span(R, oracle_mod):
    """Spans of up to 256 steps are accepted whether the variant or the span comes
    first."""
    nx = 9001
    c = Call(oracle_mod, F64, nx, 300)
    for v in [v["variant"] for v in R.variants() if v["dtype"] == F64 and v["resident"]]:
        plan = R.Plan(0.0, 1.0, 1.0, nx, c.dt, 2, 512, dtype=F64)
        assert plan.info()["span_steps"] == 256
        plan.set_variant(v)
        for S in (256, 63, 200):
            plan.set_span(S)
            assert plan.info()["variant"] == v and plan.info()["span_steps"] == S
            c.run(plan, (v, S))
