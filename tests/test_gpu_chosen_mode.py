"""A mode that was set is kept to: such a plan or batch runs with tickets (or span
by span) also where a plan as created runs on resident windows.  The results
have the same bits, so the route shows in the kernels' time only: 2000 steps of
1001 FP64 points take 0.7 ms on resident windows, 4.6 ms with tickets and more
span by span."""
import pytest

torch = pytest.importorskip("torch")

from paper_2203_10477_gb300 import inputs

pytestmark = pytest.mark.gpu

F64 = 1


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_10477_gb300 import build, rswr

    build.build()
    return rswr


@pytest.mark.parametrize("kind", ["plan", "batch"])
@pytest.mark.parametrize("mode", [0, 1])
def test_a_set_mode_is_kept_to(R, kind, mode):
    p = inputs.c1()
    T = 2000
    fA = torch.as_tensor(p.fA[:T + 1], device="cuda", dtype=torch.float64)
    times, u = [], []
    for chosen in (False, True):
        h = R.Plan.from_problem(p, dtype=F64) if kind == "plan" else R.Batch([p], dtype=F64)
        if chosen:
            h.set_mode(mode)
            assert h.info()["mode"] == mode
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        b.record()
        h.set_kernel_events(a, b)
        best = 1e9
        for _ in range(5):
            out = h.run(fA if kind == "plan" else fA.reshape(1, -1), None, T)
            h.check()
            best = min(best, a.elapsed_time(b))
        times.append(best)
        u.append(out["u"].clone())
    assert torch.equal(u[0], u[1])
    assert times[1] > 3 * times[0], f"mode {mode} set: {times[1]} ms, as created {times[0]} ms"
