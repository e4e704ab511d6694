"""The FP64 reciprocal, square root and HLLC flux of the point-wise numerics and
the FP32 division of the per-face adjoint as the device evaluates them (PTX
approximations, refinement steps and integer tests; host code takes other
branches, so only a GPU sees them)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
RCP, SQRT = 0, 1


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    so = tmp_path_factory.mktemp("point_math") / "point_math.so"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O3", "--expt-relaxed-constexpr",
                    "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "paper_2203_13760_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "gpu_checks", "point_math.cu"), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def _unary(lib, f, x):
    dx = torch.tensor(x, dtype=torch.float64, device="cuda")
    dy = torch.empty_like(dx)
    torch.cuda.synchronize()
    assert lib.pm_unary(f, ctypes.c_void_p(dx.data_ptr()), ctypes.c_void_p(dy.data_ptr()), dx.numel()) == 0
    return dy.cpu().numpy()


def test_special_values(lib):
    """Zeros, infinities, NaN and negative arguments as in IEEE arithmetic."""
    inf, nan = np.inf, np.nan
    x = np.array([0.0, -0.0, inf, -inf, nan, 1.0, -2.0, 2.0**-1022, 2.0**1000])
    with np.errstate(all="ignore"):
        for f, want in ((RCP, 1.0 / x), (SQRT, np.sqrt(x))):
            got = _unary(lib, f, x)
            assert np.array_equal(got, want, equal_nan=True), (f, got, want)
            assert np.array_equal(np.signbit(got[want == 0]), np.signbit(want[want == 0]))


@pytest.mark.parametrize("f,order", [(RCP, 1.0), (SQRT, 1.5)])
def test_rounding(lib, f, order):
    """Error against extended precision, over random mantissas and exponents.
    The approximations keep the upper 20 bits of argument and result, so their
    relative error is e <= 2^-19; the steps leave `order` e^3 and one rounding."""
    rng = np.random.default_rng(17)
    x = np.concatenate([rng.uniform(1, 4, 200000), 1 + rng.integers(0, 1 << 20, 50000) * 2.0**-52,
                        rng.uniform(1, 2, 200000) * 2.0 ** rng.integers(-1000, 1000, 200000)])
    got = _unary(lib, f, x)
    X = x.astype(np.longdouble)
    want = 1 / X if f == RCP else np.sqrt(X)
    ulp = float(np.max(np.abs(got.astype(np.longdouble) - want) / np.spacing(got)))
    assert ulp <= 0.5 + order * 2.0**-57 / 2.0**-53 + 0.01, ulp


def _hllc(lib, W, speeds=0, host=False):
    """W (2, 5, n): left and right states; the fluxes (5, n), on the device or
    in the host's branch."""
    dW = torch.tensor(np.ascontiguousarray(W), dtype=torch.float64, device="cpu" if host else "cuda")
    F = torch.empty((5, W.shape[2]), dtype=torch.float64, device=dW.device)
    torch.cuda.synchronize()
    assert lib.pm_hllc(int(host), ctypes.c_void_p(dW.data_ptr()), ctypes.c_void_p(F.data_ptr()), W.shape[2],
                       ctypes.c_double(1.4), speeds) == 0
    return F.cpu().numpy()


@pytest.mark.parametrize("speeds", [0, 1, 2])
@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("comp", [0, 4])
def test_hllc_of_an_invalid_side(lib, speeds, side, comp):
    """A face with a negative density or pressure on one side (an overshoot of
    the reconstruction) has NaN wave speeds.  Its flux is NaN on the device
    where IEEE comparisons, which are false for NaN, make it so."""
    rng = np.random.default_rng(5)
    W = rng.uniform(0.5, 1.5, (2, 5, 256))
    W[:, 1:4] = rng.uniform(-2.0, 2.0, (2, 3, 256))
    assert np.isfinite(_hllc(lib, W, speeds)).all()
    W[side, comp] *= -1
    F, want = _hllc(lib, W, speeds), _hllc(lib, W, speeds, host=True)
    assert np.array_equal(np.isnan(F), np.isnan(want))
    assert np.allclose(F, want, rtol=1e-12, atol=1e-12, equal_nan=True)


@pytest.mark.parametrize("speeds", [0, 1, 2])
def test_contact_at_rest(lib, speeds):
    """A contact discontinuity at rest: S* = 0 = u_n exactly, so no mass and no
    energy cross the face and the momentum flux is the pressure."""
    rng = np.random.default_rng(6)
    W = np.zeros((2, 5, 256))
    W[:, 0] = rng.uniform(0.1, 10.0, (2, 256))
    W[:, 4] = rng.uniform(0.1, 10.0, 256)
    F = _hllc(lib, W, speeds)
    assert np.array_equal(F[1], W[0, 4])
    assert not F[[0, 2, 3, 4]].any()


def test_fp32_division_of_the_per_face_adjoint(lib):
    """1 / rho of the conversion's reverse pass is rounded as IEEE division
    rounds it (no contraction can touch it: the other terms are zero)."""
    rho = np.random.default_rng(8).uniform(0.1, 10.0, 20000).astype(np.float32)
    d = torch.tensor(rho, device="cuda")
    out = torch.empty_like(d)
    torch.cuda.synchronize()
    assert lib.pm_prim_vjp(ctypes.c_void_p(d.data_ptr()), ctypes.c_void_p(out.data_ptr()), d.numel()) == 0
    assert np.array_equal(out.cpu().numpy(), np.float32(1) / rho)
