"""Timing events (rswr_*_set_kernel_events) on every kind of run: captured and
replayed, launched directly, resident, monolithic and paper-literal, and calls
that are no runs (a gradient with dL/da) with the events set."""
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


def events():
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()  # (torch makes the event at its first record)
    b.record()
    return a, b


def timed(h, call):
    """The same results with the events set as without, and a time between them
    that is positive and no longer than the whole call."""
    ref = [t.clone() for t in call()]
    a, b = events()
    h.set_kernel_events(a, b)
    for _ in range(2):  # (a captured run: recorded, then replayed)
        c, d = events()
        torch.cuda.synchronize()
        c.record()
        got = call()
        d.record()
        torch.cuda.synchronize()
        assert 0.0 < a.elapsed_time(b) <= c.elapsed_time(d)
        for x, y in zip(got, ref):
            assert torch.equal(x, y)
    h.set_kernel_events(None, None)


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("graph", [True, False])
def test_runs(R, dtype, graph):
    nx, T, N = 20001, 100, 8
    td = torch.float64 if dtype == F64 else torch.float32
    fA = torch.as_tensor(inputs.rng(1).standard_normal(T + 1), device="cuda").to(td)
    plan = R.Plan(0.0, 1.0, 1.0, nx, 0.9 / (nx - 1), N, 64, dtype=dtype)
    plan.set_graph(graph)

    def state(r):
        return r["u"], r["w"]

    timed(plan, lambda: state(plan.run(fA, None, T)))  # as created: resident
    timed(plan, lambda: state(plan.mono(fA, None, T)))
    timed(plan, lambda: state(plan.run_paper(fA, None, T)))
    timed(plan, lambda: (plan.adjoint(fA, None, T, 40, fA)["grad_fA"],))
    for v in [v for v in R.variants() if v["dtype"] == dtype and v["form"] == plan.info()["form"]]:
        if 0 < v["max_span"] < 32:
            continue
        plan.set_variant(v["variant"])
        timed(plan, lambda: state(plan.run(fA, None, T)))
        if v["resident"]:
            timed(plan, lambda: state(plan.run_paper(fA, None, T)))


@pytest.mark.parametrize("dtype", [F32, F64])
def test_gradients_leave_the_events_alone(R, dtype):
    nx, T = 20001, 200
    td = torch.float64 if dtype == F64 else torch.float32
    fA = torch.as_tensor(inputs.rng(2).standard_normal(T + 1), device="cuda").to(td)
    plan = R.Plan(0.0, 1.0, 1.0, nx, 0.9 / (nx - 1), 8, 64, dtype=dtype)
    ref = plan.adjoint(fA, None, T, 40, fA, want_a=True)
    kept = plan.run_keep(fA, None, T, j_r=40)
    a, b = events()
    torch.cuda.synchronize()
    before = a.elapsed_time(b)
    plan.set_kernel_events(a, b)
    got = plan.adjoint(fA, None, T, 40, fA, want_a=True)
    again = plan.run_keep(fA, None, T, j_r=40)
    plan.check()
    assert a.elapsed_time(b) == before
    assert torch.equal(got["grad_fA"], ref["grad_fA"]) and got["grad_a"].item() == ref["grad_a"].item()
    assert torch.equal(again["u"], kept["u"]) and torch.equal(again["recv"], kept["recv"])


def test_batch_runs(R):
    class P:
        def __init__(self, nx):
            self.nx, self.xa, self.xb, self.a, self.dt, self.n_sub, self.overlap = nx, 0.0, 1.0, 1.0, 0.8 / (nx - 1), 1, 64

    batch = R.Batch([P(n) for n in (4001, 777, 12345)], dtype=F32)
    T = 90
    fA = torch.as_tensor(inputs.rng(3).standard_normal((3, T + 1)).astype(np.float32), device="cuda")
    for graph in (True, False):
        batch.set_graph(graph)
        timed(batch, lambda: (batch.run(fA, None, T)["u"],))
