"""One and two probes in a resident window, at every position: a receiver on every
grid point (every register and lane of every variant's windows, the ends of all
pieces, the halos beside them), and the two fluxes of an interface that moves
over the windows.  Bit for bit against the CPU oracle."""
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


def data(dtype, nx, T):
    dt_ = np.float64 if dtype == F64 else np.float32
    r = inputs.rng(nx)
    return [r.standard_normal(n).astype(dt_) for n in (T + 1, T + 1, nx, nx)], dict(
        form=0 if dtype == F64 else 1, prec="f64" if dtype == F64 else "f32")


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("S", [5, 14])
def test_receiver_on_every_point(R, oracle_mod, dtype, S):
    nx, T = 2003, 45
    (fA, fB, q0, q1), kw = data(dtype, nx, T)
    dt = 0.9 / (nx - 1)
    ref = oracle_mod.leapfrog(nx, T, 1.0, dt, fA, fB, q0=q0, q1=q1, rec_j=list(range(nx)), **kw)
    ref = torch.as_tensor(ref["rec"], device="cuda")
    fA, fB, q0, q1 = (torch.as_tensor(x, device="cuda") for x in (fA, fB, q0, q1))
    out = (torch.empty_like(q0), torch.empty_like(q0))
    for v in [v["variant"] for v in R.variants() if v["dtype"] == dtype and v["resident"]]:
        plan = R.Plan(0.0, 1.0, 1.0, nx, dt, 1, 64, dtype=dtype)
        plan.set_span(S)
        plan.set_variant(v)
        got = torch.stack([plan.run(fA, fB, T, q0=q0, q1=q1, j_r=j, out=out)["recv"] for j in range(nx)])
        plan.check()
        bad = torch.nonzero((got != ref).any(dim=1)).flatten().tolist()
        assert not bad, (v, bad[:10])


@pytest.mark.parametrize("dtype", [F32, F64])
def test_fluxes_of_a_moving_interface(R, oracle_mod, dtype):
    T, ov = 37, 16
    todo = [v["variant"] for v in R.variants() if v["dtype"] == dtype and v["resident"]]
    for nx in list(range(1501, 1569, 2)) + [2600, 2601]:
        (fA, fB, q0, q1), kw = data(dtype, nx, T)
        dt = 0.9 / (nx - 1)
        ref = oracle_mod.rswr_mask(nx, T, 1.0, dt, fA, fB, 2, ov, q0=q0, q1=q1, **kw)
        for v in todo:
            plan = R.Plan(0.0, 1.0, 1.0, nx, dt, 2, ov, dtype=dtype)
            plan.set_variant(v)
            got = plan.run(fA, fB, T, q0=q0, q1=q1, traces=True)
            plan.check()
            for k in ("traces", "u", "w"):
                assert np.array_equal(got[k].cpu().numpy(), ref[k]), (nx, v, k)
