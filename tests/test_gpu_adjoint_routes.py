"""The three sweeps of a gradient with dL/da on the same problems: resident (plans
as created that fit on the chip), persistent with tickets (a set variant, span
or mode) and span by span (a checkpoint spacing), single plans and batches, both
precisions; the resident one also at the sizes where its cut can go wrong.

They update every adjoint point with the same operations on the same operands,
so dL/dfA agrees bit for bit (FP64: with the oracle too).  They tile the grid
differently, so the sums of pairing terms meet in another order: dL/da is
asserted to the rounding of a 128-term FP32 sum (128 * 2^-24 of the sum of |terms|,
from the FP64 oracle), in FP64 to 1e-12 of it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2203_10477_gb300 import inputs

pytestmark = pytest.mark.gpu

F32, F64 = 0, 1
A = 1.3


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_10477_gb300 import build, rswr

    build.build()
    return rswr


def waves(dtype, T, seed):
    dt_ = np.float64 if dtype == F64 else np.float32
    r = inputs.rng(seed)
    return [r.standard_normal(T + 1).astype(dt_) for _ in range(3)]


def bound(dtype, abs_da):
    return (1e-12 if dtype == F64 else 128 * 2.0 ** -24) * abs_da


def ticketed(R, plan, how, dtype):
    """Takes a plan off the resident path."""
    if how == "variant":
        own = [v for v in R.variants() if v["dtype"] == dtype and v["form"] == plan.info()["form"] and not v["resident"]]
        plan.set_variant(own[0]["variant"])
    elif how == "span":
        plan.set_span(plan.info()["span_steps"])
    else:
        plan.set_mode(R.MODE_PERSISTENT)


# nx = 8192 puts the right node on a thread's last register, 8001 on its first;
# 600001 FP32 points: sixteen points per lane, two parts to a span
@pytest.mark.parametrize("dtype,nx,T,jr", [(F32, 8001, 4001, 2500), (F32, 8192, 1000, 300), (F32, 600001, 300, 100),
                                           (F32, 600001, 296, 100), (F64, 8001, 1003, 400), (F64, 60001, 250, 100)])
@pytest.mark.parametrize("ov", [64, 20])
def test_the_three_sweeps_agree(R, oracle_mod, dtype, nx, T, jr, ov):
    dt = 0.9 / (nx - 1) / A
    fA, fB, w = waves(dtype, T, nx + T)
    ref = oracle_mod.adjoint(nx, T, A, dt, fA, fB, jr, w)
    first = None
    for how in ("resident", "variant", "span", "mode", "spacing"):
        plan = R.Plan(0.0, 1.0, A, nx, dt, 8, ov, dtype=dtype)
        if how == "spacing":
            plan.set_checkpoint_spacing(5)
        elif how != "resident":
            ticketed(R, plan, how, dtype)
        got = plan.adjoint(fA, fB, T, jr, w, want_a=True)
        plan.check()
        g, da = got["grad_fA"].clone(), got["grad_a"].item()
        first = g if first is None else first
        assert torch.equal(g, first), how
        assert abs(da - ref["da"]) <= (1e-12 if dtype == F64 else 1e-4) * ref["abs_da"], how
        if dtype == F64:
            assert np.array_equal(g.cpu().numpy(), ref["dg"]), how
        if how in ("resident", "variant"):
            # a kept forward run, and the gradient from its states
            kept = plan.run_keep(torch.as_tensor(fA, device="cuda"), torch.as_tensor(fB, device="cuda"), T, j_r=jr)
            run = plan.run(fA, fB, T, j_r=jr)
            for k in ("u", "w", "recv"):
                assert torch.equal(kept[k], run[k]), (how, k)
        if how == "resident":
            da0 = da
        assert abs(da - da0) <= bound(dtype, ref["abs_da"]), how


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("how", ["variant", "mode"])
def test_batches(R, oracle_mod, dtype, how):
    class P:
        def __init__(self, nx, a):
            self.nx, self.xa, self.xb, self.a, self.n_sub, self.overlap = nx, 0.0, 1.0, a, 2, 64
            self.dt = 0.9 / (nx - 1) / a

    probs, T = [P(2001, 1.0), P(777, 1.7), P(4096, 0.6), P(129, 1.0)], 333
    jr = [150, 300, 0, 128]
    ws = [waves(dtype, T, 10 + p) for p in range(len(probs))]
    fA, fB, w = (torch.as_tensor(np.stack([x[k] for x in ws]), device="cuda") for k in range(3))
    got = []
    for chosen in (False, True):
        b = R.Batch(probs, dtype=dtype)
        if chosen:
            ticketed(R, b, how, dtype)
        r = b.adjoint(fA, fB, T, jr, w, want_a=True)
        b.check()
        got.append((r["grad_fA"].clone(), r["grad_a"].cpu().numpy()))
    assert torch.equal(got[0][0], got[1][0])
    for p, q in enumerate(probs):
        ref = oracle_mod.adjoint(q.nx, T, q.a, q.dt, ws[p][0], ws[p][1], jr[p], ws[p][2])
        assert abs(got[0][1][p] - got[1][1][p]) <= bound(dtype, ref["abs_da"])
        if dtype == F64:
            assert np.array_equal(got[0][0][p].cpu().numpy(), ref["dg"])
            assert abs(got[0][1][p] - ref["da"]) <= bound(dtype, ref["abs_da"])


# pieces of the smallest length (two of 25 points at a halo of 16), windows just
# full and just not, several spans between exchanges (overlaps 3 to 20), receivers
# beside the nodes, on a piece's end and in the halos beside it; run lengths on and
# off a span's end
@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("ov", [3, 10, 20, 64])
@pytest.mark.parametrize("nx", [49, 50, 51, 64, 97, 224, 225, 447, 449, 1000])
def test_the_cut_of_the_resident_sweep(R, oracle_mod, dtype, ov, nx):
    if nx < ov:
        pytest.skip("a core holds at least the overlap")
    dt = 0.9 / (nx - 1) / A
    mid = nx // 2
    js = sorted({j for j in (1, 2, mid - 17, mid - 9, mid - 1, mid, mid + 1, mid + 8, mid + 16, nx - 2) if 0 < j < nx - 1})
    for T in (nx + 1, nx + 8, nx + 15, 7):
        fA, fB, w = waves(dtype, T, nx + T)
        plan, tick = (R.Plan(0.0, 1.0, A, nx, dt, 1, ov, dtype=dtype) for _ in range(2))
        ticketed(R, tick, "variant", dtype)
        for jr in js:
            got = plan.adjoint(fA, fB, T, jr, w, want_a=True)
            plan.check()
            g, da = got["grad_fA"].clone(), got["grad_a"].item()
            ref = oracle_mod.adjoint(nx, T, A, dt, fA, fB, jr, w)
            other = tick.adjoint(fA, fB, T, jr, w, want_a=True)
            tick.check()
            assert torch.equal(g, other["grad_fA"]), (T, jr)
            assert abs(da - other["grad_a"].item()) <= bound(dtype, ref["abs_da"]), (T, jr)
            if dtype == F64:
                assert np.array_equal(g.cpu().numpy(), ref["dg"]), (T, jr)
                assert abs(da - ref["da"]) <= bound(dtype, ref["abs_da"]), (T, jr)
