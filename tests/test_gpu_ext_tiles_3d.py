"""The 3D FP32 kernels of the extended forms (walls, WENO3-JS) come in two tile
shapes, of which the grid picks one; the viscous 32 x 8 form reconstructs at the
faces, the others per cell.  Every shape and chunk against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2203_13760_gb300 import inputs, jf

pytestmark = pytest.mark.gpu
W = inputs.WALL


@pytest.mark.parametrize("recon", ["weno3-js", "weno5-js"])
@pytest.mark.parametrize("viscous", [False, True])
# rows a multiple of 8 but not of 7, and one more; one column and two; a few planes
@pytest.mark.parametrize("n", [(32, 8, 6), (45, 17, 11)])
def test_every_tile_shape(n, viscous, recon):
    case = inputs.random_smooth(n, seed=31, bc=(W, 1, W, W, 0, 0), viscous=viscous, mu=0.01 if viscous else 0.0)
    case.recon = recon
    U32 = case.U.astype(np.float32)
    dt = 1e-4
    want = oracle.rk3_step(oracle.config(**case.params()), U32.astype(np.float64), dt)
    s = jf.Solver.from_case(case, dtype="f32")
    names = s.variants()
    assert any("32x8" in d for d in names) and any("32x7" in d for d in names)
    for v in range(len(names)):
        s.set_variant(v)
        U = torch.from_numpy(U32).cuda()
        s.rk3_step(U, s.scalar(dt))
        s.sync()
        got = U.cpu().numpy()
        for g in ([0], [1, 2, 3], [4]):
            assert np.abs(got[g] - want[g]).max() <= 1e-5 * np.abs(want[g]).max(), names[v]


def test_default_tile_follows_the_rows():
    """48 rows are six tiles of 8 or seven of 7, 56 rows seven or eight."""
    def default_is(n, tile):
        s = jf.Solver((n,) * 3, bc=(W,) * 6, dtype="f32", recon="weno3-js")
        U = torch.tensor(inputs.random_smooth((n,) * 3, seed=2).U, dtype=torch.float32, device="cuda")
        dt = s.scalar(1e-4)
        want = s.rk3_step(U.clone(), dt)
        other = []
        for v, d in enumerate(s.variants()):
            if "zchunk=auto" in d:
                s.set_variant(v)
                same = torch.equal(s.rk3_step(U.clone(), dt), want)
                if f"tile={tile} " in d:
                    assert same
                else:
                    other.append(same)
        s.close()
        return other

    default_is(48, "32x8")
    default_is(56, "32x7")
