"""The gradient with dL/da on resident windows (csrc/resident_adjoint.cu)."""
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


@pytest.mark.parametrize("nx", [5001, 1 << 20])  # eight and sixteen points per lane
def test_sums_over_spans_leave_fp32s_range(R, oracle_mod, nx):
    """With a cotangent of 2^112 a chain of products (eight points, one span) stays
    below FP32's largest value: at most 7.5e3 times 2^112, while the sum of a
    point's chains over all spans is 5.6e5 times 2^112, beyond it (both from the
    same sweeps in FP64; nothing returns from the grid's right end).  The resident
    sweep against the persistent one (a plan on a variant with tickets), which
    sums its spans in double: the same chains, or chains of at most 128 terms that
    meet in another order."""
    T, jr = 4000, 300
    t = np.arange(T + 1)
    fA = (1e5 * np.sin(np.pi * t / T) ** 2).astype(np.float32)
    wbar = np.full(T + 1, 2.0 ** 112, np.float32)
    got = []
    for variant in (None, 0):
        plan = R.Plan(0.0, 1.0, 1.0, nx, 0.9 / (nx - 1), 8, 64, dtype=F32)
        if variant is not None:
            plan.set_variant(variant)
        got.append(plan.adjoint(fA, None, T, jr, wbar, want_a=True))
        plan.check()
    da = [g["grad_a"].item() for g in got]
    ref = oracle_mod.adjoint(5001, T, 1.0, 0.9 / 5000, fA, np.zeros(T + 1), jr, np.ones(T + 1))
    assert all(abs(x) > 2.0 ** 128 for x in da)
    assert abs(da[0] - da[1]) * 2.0 ** -112 <= 128 * 2.0 ** -24 * ref["abs_da"], da
    assert torch.equal(got[0]["grad_fA"], got[1]["grad_fA"])


SWEEP = 0x40000000  # RSWR_INJECT_SWEEP


def gradient(R, dtype, nx, T=300, jr=200):
    td = torch.float64 if dtype == F64 else torch.float32
    fA, w = (torch.as_tensor(inputs.rng(s).standard_normal(T + 1), device="cuda").to(td) for s in (1, 2))
    plan = R.Plan(0.0, 1.0, 1.3, nx, 0.9 / (nx - 1) / 1.3, 8, 64, dtype=dtype)

    def grad():
        g = plan.adjoint(fA, None, T, jr, w, want_a=True)
        return g["grad_fA"].clone(), g["grad_a"].clone()

    return plan, grad, lambda: plan.run_keep(fA, None, T, j_r=jr)


def same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("dtype", [F32, F64])
def test_gradients_run_without_the_hook(R, dtype):
    plan, grad, keep = gradient(R, dtype, 20001)
    ref, kept = grad(), keep()
    plan.set_wait_limit(0.2)
    for tile, span in ((1, 0), (2, 3)):
        plan.inject_missing_flag(tile, span)
        got = grad()
        plan.check()
        assert same(got, ref)
        again = keep()
        plan.check()
        assert torch.equal(again["u"], kept["u"]) and torch.equal(again["recv"], kept["recv"])


@pytest.mark.parametrize("dtype,nx", [(F32, 20001), (F32, 1 << 20), (F64, 20001), (F64, 60001)])
@pytest.mark.parametrize("exchange", [0, 2])
def test_an_adjoint_exchange_that_never_comes(R, dtype, nx, exchange):
    """The neighbours' waits run out, every warp leaves the sweep, the status says so,
    and the next gradient is exact."""
    plan, grad, keep = gradient(R, dtype, nx)
    ref = grad()
    plan.set_wait_limit(0.2)
    plan.inject_missing_flag(1, SWEEP + exchange)
    for kept in (False, True):
        if kept:
            keep()
            plan.check()  # (the forward run is not affected)
        grad()
        with pytest.raises(R.RSWRError) as ei:
            plan.check()
        assert ei.value.status == 6
    plan.inject_missing_flag(-1, 0)
    got = grad()
    plan.check()
    assert same(got, ref)


@pytest.mark.parametrize("barrier", [0, 1, 4])
def test_a_grid_barrier_of_the_paper_run_that_never_opens(R, barrier):
    nx, T = 60001, 150
    fA = torch.as_tensor(inputs.rng(3).standard_normal(T + 1).astype(np.float32), device="cuda")
    plan = R.Plan(0.0, 1.0, 1.0, nx, 0.9 / (nx - 1), 30, 64, dtype=F32)
    ref = plan.run_paper(fA, None, T)
    assert len(ref["spans"]) > 3
    plan.set_wait_limit(0.2)
    plan.inject_missing_flag(1, SWEEP + barrier)
    with pytest.raises(R.RSWRError) as ei:
        plan.run_paper(fA, None, T)
    assert ei.value.status == 6
    plan.inject_missing_flag(-1, 0)
    got = plan.run_paper(fA, None, T)
    assert torch.equal(got["u"], ref["u"]) and list(got["spans"]) == list(ref["spans"])
