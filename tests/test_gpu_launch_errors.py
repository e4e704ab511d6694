"""A launch that the runtime refuses (a grid dimension beyond its limit) is
reported by its own call only: the next launches, of this library and of
PyTorch, do not find the error again."""
import pytest
import torch

from paper_2203_13760_gb300 import jf

pytestmark = pytest.mark.gpu


def test_refused_launch_leaves_no_error_behind():
    # 32 x 7 tiles: more than 65535 of them along y
    s = jf.Solver((6, 70000 * 8), bc=(0,) * 6, dtype="f32")
    U = torch.ones(s.shape, dtype=torch.float32, device="cuda")
    U[1:4] = 0
    U[4] = 2.5
    dt = s.scalar(1e-6)
    roe = jf.Solver((32, 16), bc=(0,) * 6, dtype="f32", flux="roe")  # launched the plain way
    V = U[:, :, :16, :1].expand(-1, -1, -1, 32).contiguous()
    want = V.clone()
    for call in (lambda: s.rhs(U), lambda: s.rk3_step(U, dt)):
        with pytest.raises(jf.JFError, match="invalid"):
            call()
        roe.rk3_step(V, roe.scalar(1e-6))
        assert torch.equal(V, want)
        with pytest.raises(jf.JFError, match="invalid"):
            call()
        assert torch.equal(U[0] + 1, 2 * U[0])
