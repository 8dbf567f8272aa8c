"""Many probes in one resident window (csrc/resident.cuh): interface waveforms of
short subdomains and a receiver among them, bit for bit against the CPU oracle.
Three and more probes to a window take a record per lane, several rounds of
them where a lane owns several points, and the table where they do not fit."""
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


def run_and_compare(R, oracle_mod, dtype, nx, N, ov, T, receivers, variant=None, span=None):
    dt_ = np.float64 if dtype == F64 else np.float32
    kw = dict(form=0 if dtype == F64 else 1, prec="f64" if dtype == F64 else "f32")
    dt = 0.9 / (nx - 1)
    r = inputs.rng(nx + N)
    fA, fB, q0, q1 = (r.standard_normal(n).astype(dt_) for n in (T + 1, T + 1, nx, nx))
    ref = oracle_mod.rswr_mask(nx, T, 1.0, dt, fA, fB, N, ov, q0=q0, q1=q1, **kw)
    js = [j for j in receivers if 0 <= j < nx]
    rec = oracle_mod.leapfrog(nx, T, 1.0, dt, fA, fB, q0=q0, q1=q1, rec_j=js, **kw)["rec"]
    plan = R.Plan(0.0, 1.0, 1.0, nx, dt, N, ov, dtype=dtype)
    if span is not None:
        plan.set_span(span)
    if variant is not None:
        plan.set_variant(variant)
    for j, want in zip(js, rec):
        got = plan.run(fA, fB, T, q0=q0, q1=q1, traces=True, j_r=j)
        plan.check()
        assert np.array_equal(got["recv"].cpu().numpy(), want), (variant, j)
    for k in ("u", "w", "traces"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), (variant, k)


# subdomains of 3 (several interfaces in a lane of most widths), 7, 16, 33 and 200 points
@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("length,ov", [(3, 3), (7, 5), (16, 16), (33, 20), (200, 64)])
def test_short_subdomains_on_every_resident_variant(R, oracle_mod, dtype, length, ov):
    nx, T = 2003, 67
    N = nx // length
    for v in [v["variant"] for v in R.variants() if v["dtype"] == dtype and v["resident"]]:
        # on the nodes, beside them, on and beside an interface's first traced point
        b = 5 * nx // N - (ov + 1) // 2
        run_and_compare(R, oracle_mod, dtype, nx, N, ov, T, [0, 1, b - 1, b, b + 1, nx - 2, nx - 1], variant=v,
                        span=min(ov // 2, 8))


@pytest.mark.parametrize("dtype,nx,length", [(F32, 1 << 20, 700), (F32, 1 << 20, 350), (F32, 700001, 128),
                                             (F64, 200003, 128)])
def test_full_chip(R, oracle_mod, dtype, nx, length):
    run_and_compare(R, oracle_mod, dtype, nx, nx // length, 64, 33, [nx // 2])


@pytest.mark.parametrize("dtype", [F32, F64])
def test_run_lengths(R, oracle_mod, dtype):
    for T in (1, 15, 16, 17, 32, 64, 65):
        run_and_compare(R, oracle_mod, dtype, 4001, 60, 64, T, [0, 2000])
