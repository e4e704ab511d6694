"""WENO3-JS in FP64 with an epsilon far below the default: the weights are
ratios of (eps + beta)^2, whose products the kernels may not take beyond the
range of FP64.  Uniform blocks make every indicator zero but at the jumps."""
import numpy as np
import pytest
import torch

import oracle
from paper_2203_13760_gb300 import inputs, jf

pytestmark = pytest.mark.gpu
W = inputs.WALL


@pytest.mark.parametrize("eps", [1e-6, 1e-40, 1e-100])
@pytest.mark.parametrize("flux", ["hllc", "rusanov-nn"])
@pytest.mark.parametrize("n", [(37, 1, 1), (40, 33, 1)])
def test_weno3_small_epsilon(n, flux, eps):
    case = inputs.random_blocks(n, seed=12, bc=(W, W, 1, 1, 1, 1))
    case.recon, case.flux, case.eps = "weno3-js", flux, eps
    theta = inputs.nn_params() if flux == "rusanov-nn" else None
    want = oracle.rhs(oracle.config(**case.params(), nn=theta), case.U)
    nn = None if theta is None else torch.tensor(theta, dtype=torch.float64, device="cuda")
    s = jf.Solver.from_case(case, dtype="f64", nn=nn)
    got = s.rhs(torch.tensor(case.U, dtype=torch.float64, device="cuda")).cpu().numpy()
    for g in ([0], [1, 2, 3], [4]):
        assert np.abs(got[g] - want[g]).max() <= 1e-12 * np.abs(want[g]).max()
