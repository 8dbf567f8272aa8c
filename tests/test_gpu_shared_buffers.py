"""Runs whose outputs share memory with what they read, or with each other:
states continued in place, the pair swapped, shifted by a few points, a record
or a final state over the samples.  The final state appears when the run has
read all of its inputs, so every such call gives the bits of the call with
buffers of its own."""
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


def td(dtype):
    return torch.float64 if dtype == F64 else torch.float32


def rand(n, dtype, seed):
    return torch.as_tensor(inputs.rng(seed).standard_normal(n), device="cuda").to(td(dtype))


# 1001: one cluster; 60001: several CTAs that exchange through L2.  T below, at
# and beyond the steps between two exchanges (64 at most), with and without probes
@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("nx", [1001, 60001])
@pytest.mark.parametrize("T", [1, 2, 31, 64, 200])
@pytest.mark.parametrize("probe", [False, True])
def test_states_in_place(R, dtype, nx, T, probe):
    plan = R.Plan(0.0, 1.0, 1.0, nx, 0.9 / (nx - 1), 1, 64, dtype=dtype)
    fA, fB = rand(T + 1, dtype, 1), rand(T + 1, dtype, 2)
    u0, w0 = rand(nx, dtype, 3), 0.1 * rand(nx, dtype, 4)
    kw = dict(j_r=nx // 2) if probe else {}
    ref = plan.run(fA, fB, T, q0=u0, q1=w0, **kw)
    for swapped in (False, True):
        u, w = u0.clone(), w0.clone()
        got = plan.run(fA, fB, T, q0=u, q1=w, out=(w, u) if swapped else (u, w), **kw)
        plan.check()
        assert torch.equal(got["u"], ref["u"]) and torch.equal(got["w"], ref["w"]), f"swapped {swapped}"
        if probe:
            assert torch.equal(got["recv"], ref["recv"])
    # the outputs lie 7 points after the inputs
    a, b = torch.empty(nx + 8, dtype=td(dtype), device="cuda"), torch.empty(nx + 8, dtype=td(dtype), device="cuda")
    a[:nx], b[:nx] = u0, w0
    got = plan.run(fA, fB, T, q0=a[:nx], q1=b[:nx], out=(a[7:7 + nx], b[7:7 + nx]), **kw)
    plan.check()
    assert torch.equal(got["u"], ref["u"]) and torch.equal(got["w"], ref["w"]), "shifted"


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("T", [1, 33])
def test_batch_states_in_place(R, dtype, T):
    class P:
        def __init__(self, nx):
            self.nx, self.xa, self.xb, self.a, self.dt, self.n_sub, self.overlap = nx, 0.0, 1.0, 1.0, 0.8 / (nx - 1), 1, 64

    batch = R.Batch([P(n) for n in (4001, 777, 12345, 129)], dtype=dtype)
    n = int(batch.offsets[-1])
    fA = rand(4 * (T + 1), dtype, 5).reshape(4, T + 1)
    u, w = rand(n, dtype, 6), 0.1 * rand(n, dtype, 7)
    ref = batch.run(fA, None, T, q0=u, q1=w)
    got = batch.run(fA, None, T, q0=u, q1=w, out=(u, w))
    batch.check()
    assert torch.equal(got["u"], ref["u"]) and torch.equal(got["w"], ref["w"])


@pytest.mark.parametrize("dtype", [F32, F64])
def test_final_state_over_the_samples(R, dtype):
    nx, T = 20001, 96
    fA0, fB0 = rand(T + 1, dtype, 8), rand(T + 1, dtype, 9)
    s0 = rand(T + 1, dtype, 10).reshape(1, -1)
    plan = R.Plan(0.0, 1.0, 1.0, nx, 0.9 / (nx - 1), 8, 64, dtype=dtype)
    for keep in (False, True):
        run = plan.run_keep if keep else plan.run
        ref = run(fA0, fB0, T, j_r=40)
        u, w = rand(nx, dtype, 11), rand(nx, dtype, 12)
        u[:T + 1], w[nx - T - 1:] = fA0, fB0
        got = run(u[:T + 1], w[nx - T - 1:], T, j_r=40, out=(u, w))
        plan.check()
        for k in ("u", "w", "recv"):
            assert torch.equal(got[k], ref[k]), f"keep {keep}: {k}"
    # point sources whose samples the final state replaces
    plan.set_sources([9000], s0)
    ref = plan.run(fA0, None, T)
    u, w = torch.empty(nx, dtype=td(dtype), device="cuda"), torch.empty(nx, dtype=td(dtype), device="cuda")
    u[500:500 + T + 1] = s0[0]
    plan.set_sources([9000], u[500:500 + T + 1].reshape(1, -1))
    got = plan.run(fA0, None, T, out=(u, w))
    plan.check()
    assert torch.equal(got["u"], ref["u"]) and torch.equal(got["w"], ref["w"])
    # one buffer for both components: the second one is in it afterwards
    plan.set_sources()
    ref = plan.run(fA0, fB0, T)
    got = plan.run(fA0, fB0, T, out=(u, u))
    plan.check()
    assert torch.equal(got["u"], ref["w"])


@pytest.mark.parametrize("dtype", [F32, F64])
def test_receiver_record_over_the_initial_state(R, dtype):
    import ctypes

    nx, T, jr = 20001, 70, 9000
    fA, u0, w0 = rand(T + 1, dtype, 13), rand(nx, dtype, 14), 0.1 * rand(nx, dtype, 15)
    plan = R.Plan(0.0, 1.0, 1.0, nx, 0.9 / (nx - 1), 1, 64, dtype=dtype)
    ref = plan.run(fA, None, T, q0=u0, q1=w0, j_r=jr)
    u, w, a, b = u0.clone(), w0.clone(), torch.empty_like(u0), torch.empty_like(w0)
    rec = u[jr:jr + T + 1]  # the record replaces the state around the receiver
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    R.check(R.lib().rswr_run(plan.h, p(fA), None, T, p(u), p(w), p(a), p(b), None, jr, p(rec),
                             torch.cuda.current_stream().cuda_stream))
    plan.check()
    assert torch.equal(rec, ref["recv"]) and torch.equal(a, ref["u"]) and torch.equal(b, ref["w"])


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("T", [5, 100])
def test_paper_run_with_shared_buffers(R, dtype, T):
    nx = 9001
    plan = R.Plan(0.0, 1.0, 1.0, nx, 0.9 / (nx - 1), 6, 32, dtype=dtype)
    fA, fB = rand(T + 1, dtype, 16), rand(T + 1, dtype, 17)
    u0, w0 = rand(nx, dtype, 18), 0.1 * rand(nx, dtype, 19)
    ref = plan.run_paper(fA, fB, T, q0=u0, q1=w0)
    u, w = u0.clone(), w0.clone()
    got = plan.run_paper(fA, fB, T, q0=u, q1=w, out=(u, w))
    assert torch.equal(got["u"], ref["u"]) and torch.equal(got["w"], ref["w"])
    ref = plan.run_paper(fA, fB, T)
    u[:T + 1], w[nx - T - 1:] = fA, fB
    got = plan.run_paper(u[:T + 1], w[nx - T - 1:], T, out=(u, w))
    assert torch.equal(got["u"], ref["u"]) and torch.equal(got["w"], ref["w"])
