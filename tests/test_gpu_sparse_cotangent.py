"""The tiled adjoints pass over boxes and planes whose cotangent is uniform: a
cotangent that is zero but for a few cells, or constant but for them, gives what
linearity demands of it (the difference of two dense ones)."""
import pytest
import torch

from paper_2203_13760_gb300 import inputs, jf

pytestmark = pytest.mark.gpu


# boxes of 128 (1D) and 16 x 16 cells, columns of 16 x 8 (viscous 16 x 4) cells
@pytest.mark.parametrize("n", [(300, 1, 1), (70, 41, 1), (41, 19, 37)])
@pytest.mark.parametrize("viscous", [False, True])
@pytest.mark.parametrize("bc", [(0,) * 6, (1,) * 6])
@pytest.mark.parametrize("level", [0.0, 0.7])
def test_uniform_but_for_a_few_cells(n, viscous, bc, level):
    case = inputs.random_smooth(n, seed=9, bc=bc, viscous=viscous, mu=0.01 if viscous else 0.0)
    s = jf.Solver.from_case(case, dtype="f64")
    U = torch.tensor(case.U, dtype=torch.float64, device="cuda")
    dt = s.scalar(1e-3)
    gen = torch.Generator(device="cuda").manual_seed(4)
    dense = torch.randn(U.shape, dtype=torch.float64, device="cuda", generator=gen)
    nx, ny, nz = n
    spots = [(0, 0, 0), (nz - 1, ny - 1, nx - 1), (nz // 2, ny // 2, nx // 2), (min(4, nz - 1), 0, min(17, nx - 1))]
    for spot in spots:
        lam = torch.full_like(U, level)
        lam[(slice(None),) + spot] = torch.randn(5, dtype=torch.float64, device="cuda", generator=gen)
        got = s.rk3_step_vjp(U, dt, lam)
        want = s.rk3_step_vjp(U, dt, dense + lam) - s.rk3_step_vjp(U, dt, dense)
        s.sync()
        assert float((got - want).abs().max()) <= 1e-12 * float(want.abs().max() + dense.abs().max()), spot
