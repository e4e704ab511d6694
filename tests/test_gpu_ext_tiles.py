"""Tile shapes of the extended run-time-scheme kernels on 2D FP32 grids (walls,
WENO3-JS): the default depends on the grid, and every shape gives the same bits
(a cell's arithmetic does not depend on its tile), single grids and batches."""
import pytest

from paper_2203_13760_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2203_13760_gb300 import jf  # noqa: E402

WALLS = (inputs.WALL,) * 4 + (1, 1)
SCH = dict(dtype="f32", recon="weno3-js", integrator="rk2")


# one wave of 32 x 7 tiles, two of either, three against two, and a ragged grid of more
@pytest.mark.parametrize("n", [(64, 45, 1), (300, 300, 1), (384, 384, 1), (613, 347, 1)])
def test_tiles_agree(n):
    U0 = torch.tensor(inputs.random_smooth(n, seed=5).U, dtype=torch.float32, device="cuda")

    def run(v):
        s = jf.Solver(n, bc=WALLS, **SCH)
        if v is not None:
            s.set_variant(v)
        U = U0.clone()
        s.run(U, 3, s.scalar(1e-4))
        s.sync()
        names = s.variants()
        s.close()
        return U, names

    want, names = run(None)
    assert any("32x8" in d for d in names) and any("32x7" in d for d in names)
    for v in range(len(names)):
        assert torch.equal(run(v)[0], want), names[v]
    b = jf.Batch([jf.make_grid(n, bc=WALLS)] * 2, **SCH)
    V = [U0.clone(), U0.clone()]
    traj = b.feed_forward(V, 3, [1e-4, 1e-4])
    for t in traj:
        assert torch.equal(t[3].reshape(want.shape), want)
    b.close()
