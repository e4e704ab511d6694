"""The reverse sweep of a batch's trajectories in one call
(jf_batch_feed_forward_vjp) against the same chain of jf_batch_step_vjp calls:
the launches are the same, so the results differ by the order of the atomic
additions only (FP64: 1e-13 of the largest value per step, FP32: 1e-6)."""
import pytest

from paper_2203_13760_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2203_13760_gb300 import jf  # noqa: E402

WALLS = (inputs.WALL,) * 4 + (1, 1)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("flux,integrator,nsteps", [("rusanov-nn", "rk2", 4), ("rusanov-nn", "euler", 3),
                                                    ("hllc", "rk3", 3), ("hllc", "rk2", 1), ("hllc", "rk2", 0)])
def test_sweep_equals_step_chain(dtype, flux, integrator, nsteps):
    t = torch.float32 if dtype == "f32" else torch.float64
    sides = [(9, 7, 1), (12, 5, 1), (33, 8, 1)]  # states of odd sizes: slots off 16-byte boundaries
    nn = flux == "rusanov-nn"
    theta = torch.tensor(inputs.nn_params(seed=4), dtype=t, device="cuda") if nn else None
    b = jf.Batch([jf.make_grid(n, bc=WALLS) for n in sides], dtype=dtype, flux=flux, recon="weno3-js",
                 integrator=integrator, nn=theta)
    U0 = [torch.tensor(inputs.random_smooth(n, seed=i).U, dtype=t, device="cuda") for i, n in enumerate(sides)]
    dts = [1e-3, 1.5e-3, 8e-4]
    trajs = b.feed_forward(U0, nsteps, dts)
    gen = torch.Generator(device="cuda").manual_seed(3)
    g = [torch.randn(tr.shape, generator=gen, device="cuda", dtype=t) for tr in trajs]
    dt = torch.tensor(dts, dtype=torch.float64, device="cuda")
    bar = torch.zeros(jf.NN_PARAMS, dtype=t, device="cuda") if nn else None
    want_bar = bar.clone() if nn else None
    got = b.feed_forward_vjp(trajs, g, nsteps, dt, bar)
    lam = [x[nsteps].clone() for x in g]
    for k in reversed(range(nsteps)):
        lam = b.step_vjp([tr[k].clone() for tr in trajs], dt, lam, adds=[x[k].clone() for x in g],
                         theta_bar=want_bar)
    b.sync()
    tol = 1e-13 if dtype == "f64" else 1e-6
    for x, y in list(zip(got, lam)) + ([(bar, want_bar)] if nn else []):
        assert torch.isfinite(x).all()
        assert (x - y).abs().max() <= (nsteps + 1) * tol * max(float(y.abs().max()), 1.0)
    b.close()


def test_sweep_refuses_an_open_parameter_gradient():
    b = jf.Batch([jf.make_grid((8, 8, 1))], flux="rusanov-nn", recon="weno3-js",
                 nn=torch.tensor(inputs.nn_params(), dtype=torch.float32, device="cuda"))
    tr = [torch.ones((2, 5, 1, 8, 8), device="cuda")]
    b.param_grad_begin(1)
    with pytest.raises(jf.JFError) as e:
        b.feed_forward_vjp(tr, [torch.zeros_like(tr[0])], 1, torch.ones(1, dtype=torch.float64, device="cuda"))
    assert e.value.status == jf.JF_ERR_ARG
    b.close()
