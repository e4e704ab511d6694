"""Kernels of libjf are launched with programmatic dependence on the launch
before them.  They still see everything that precedes them on the stream: a
copy, a memset, another library's kernel and the join of another stream,
launched directly or replayed from a captured graph.  Every state equals, bit
for bit, the one with a synchronisation after each call; the adjoint up to the
order of its atomic additions (FP32 1e-5, FP64 1e-13 of its maximum)."""
import pytest

from paper_2203_13760_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2203_13760_gb300 import jf  # noqa: E402


def _chain(s, src, U, dt, used, lam, out, side, sync):
    """Steps and an adjoint between copies, scaled fields and a second stream's write."""
    U.copy_(src)
    sync()
    s.rk3_step(U, None, used)
    sync()
    dt.copy_(used)
    dt.mul_(0.5)
    sync()
    s.rk3_step(U, dt)
    sync()
    U.mul_(1.0)
    lam.zero_()
    sync()
    ev = torch.cuda.Event()
    ev.record()
    side.wait_event(ev)
    with torch.cuda.stream(side):
        lam.add_(1.0)
        done = torch.cuda.Event()
        done.record()
    torch.cuda.current_stream().wait_event(done)
    s.rk3_step_vjp(U, dt, lam, out)
    sync()
    s.rk3_step(U, dt)
    sync()


@pytest.mark.parametrize("case", [
    inputs.random_smooth((33, 1, 1), seed=1), inputs.random_smooth((70, 41, 1), seed=2, viscous=True, mu=0.01),
    inputs.random_smooth((40, 24, 19), seed=3, viscous=True, mu=0.01)], ids=["1d", "2d", "3d"])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_launches_follow_the_stream(case, dtype):
    t = torch.float32 if dtype == "f32" else torch.float64
    s = jf.Solver.from_case(case, dtype=dtype)
    src = torch.tensor(case.U, dtype=t, device="cuda")
    side = torch.cuda.Stream()

    def bufs():
        return (torch.zeros_like(src), torch.zeros(1, dtype=torch.float64, device="cuda"),
                torch.zeros(1, dtype=torch.float64, device="cuda"), torch.zeros_like(src), torch.zeros_like(src))

    U, dt, used, lam, out = bufs()
    _chain(s, src, U, dt, used, lam, out, side, torch.cuda.synchronize)
    want = [x.clone() for x in (U, dt, out)]
    tol = 1e-5 if dtype == "f32" else 1e-13

    def check(b):
        torch.cuda.synchronize()
        assert torch.equal(b[0], want[0]) and torch.equal(b[1], want[1])
        assert (b[4] - want[2]).abs().max() <= tol * want[2].abs().max()

    b = bufs()
    for _ in range(3):
        _chain(s, src, *b, side, lambda: None)
    check(b)

    b = bufs()
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        _chain(s, src, *b, side, lambda: None)
    for _ in range(3):
        g.replay()
    check(b)
    s.close()
