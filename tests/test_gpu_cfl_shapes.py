"""The CFL pass chooses its threads and CTAs by the number of cells: one CTA of
whole warps, CTAs of 128 to 512 threads, two per SM with several vectors a
thread, cell counts that fill no vector.  The fastest cell sits at either end."""
import numpy as np
import pytest
import torch

import oracle
from paper_2203_13760_gb300 import inputs, jf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("n", [5, 64, 255, 256, 258, 1023, 152 * 256 + 2, 152 * 1024 - 6, 152 * 1024 + 3, 400001])
def test_step_of_every_shape(n, dtype):
    t = np.float64 if dtype == "f64" else np.float32
    s = jf.Solver((n, 1, 1), dtype=dtype, viscous=True, mu=1e-9, heat=True)
    for fast in (0, n - 1):
        u = np.full(n, 0.1)
        u[fast] = -3.0
        U = inputs.conservative(1.0 + 0.1 * np.cos(np.arange(n)), u, 0.0, 0.0, 1.0, 1.4).reshape(5, 1, 1, n).astype(t)
        c = oracle.config((n, 1, 1), viscous=True, mu=1e-9, heat=True)
        want = oracle.compute_dt(c, U.astype(np.float64))
        got = s.compute_dt(torch.from_numpy(U).cuda()).item()
        # a few roundings of the working precision
        assert abs(got - want) <= 16 * np.finfo(t).eps * want, (fast, got, want)
