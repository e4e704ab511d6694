"""The tiled adjoint kernels' own source (vjp.cuh, vjp3.cuh, vjp_cell.cuh),
compiled for the CPU (tests/host_emu/emu_vjp.cpp) under AddressSanitizer and
UBSan where the toolchain has them, so that every shared-memory and global
access stays inside its buffer.  One stage's result out = w + dt J^T w is
held to the oracle's forward-mode derivative of one Euler step by the
dot-product identity <out, v> = <w, v + dt J v>, for ragged grids of the 1D and
2D boxes and the 3D z-march (several chunk lengths), periodic, zero-gradient
and mixed boundaries, and the safe reconstruction.  Bounds as for the compiled
kernels: FP64 1e-12, FP32 3e-5 of the sum of |terms|."""
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

from paper_2203_13760_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2203_13760_gb300", "csrc")
HERE = os.path.join(ROOT, "tests", "host_emu")
SMEM_DECL = "extern __shared__ __align__(16) unsigned char smem_raw[];"

# name: (case, z chunk)
CASES = {
    "1d_blocks_open": (lambda: inputs.random_blocks((150, 1, 1), seed=3), 1),
    "1d_visc_periodic": (lambda: inputs.random_smooth((131, 1, 1), seed=4, viscous=True, mu=0.02), 1),
    "2d_blocks_open": (lambda: inputs.random_blocks((37, 21, 1), seed=13), 1),
    "2d_visc_mixed": (lambda: inputs.random_smooth((35, 19, 1), seed=14, bc=(0, 0, 1, 1, 1, 1), viscous=True, mu=0.02), 1),
    "2d_visc_periodic_small": (lambda: inputs.random_smooth((9, 5, 1), seed=15, viscous=True, mu=0.02), 1),
    "3d_visc_open": (lambda: inputs.random_smooth((35, 9, 5), seed=16, bc=(1,) * 6, viscous=True, mu=0.02), 3),
    "3d_visc_periodic": (lambda: inputs.random_smooth((17, 5, 6), seed=17, viscous=True, mu=0.02), 4),
    "3d_blocks_mixed": (lambda: inputs.random_blocks((34, 6, 5), seed=18, bc=(0, 0, 1, 1, 0, 0)), 5),
}


def _safe(make):
    def f():
        c = make()
        c.safe = True
        return c
    return f


CASES["2d_blocks_safe"] = (_safe(CASES["2d_blocks_open"][0]), 1)
CASES["3d_blocks_safe"] = (_safe(CASES["3d_blocks_mixed"][0]), 2)


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("host_emu_vjp")
    for f in ("stage.cuh", "jf_math.cuh", "vjp.cuh", "vjp3.cuh", "vjp_cell.cuh", "vjp_math.cuh"):
        with open(os.path.join(CSRC, f)) as fh:
            text = fh.read()
        if SMEM_DECL in text:
            text = text.replace(SMEM_DECL, "unsigned char* smem_raw = emu_smem();")
            text = text.replace("namespace jf {\n", "unsigned char* emu_smem();\nnamespace jf {\n", 1)
        (d / f).write_text(text)
    exe = str(d / "emu_vjp")
    cmd = ["g++", "-std=c++20", "-O1", "-g1", "-fno-omit-frame-pointer", "-I", os.path.join(HERE, "cuda_stub"), "-I",
           str(d), os.path.join(HERE, "emu_vjp.cpp"), "-o", exe, "-lpthread"]
    out = subprocess.run(cmd[:1] + ["-fsanitize=address,undefined", "-fno-sanitize-recover=undefined"] + cmd[1:],
                         capture_output=True, text=True)
    if out.returncode != 0:  # no sanitizer runtime
        out = subprocess.run(cmd, capture_output=True, text=True)
    if out.returncode != 0 and "barrier" in out.stderr:
        pytest.skip("the C++ library has no std::barrier")
    assert out.returncode == 0, out.stderr[-3000:]
    return exe


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_emulated_adjoint_dot_product(orc, program, tmp_path, name, dtype):
    make, zchunk = CASES[name]
    case = make()
    t = np.float64 if dtype == "f64" else np.float32
    U = np.ascontiguousarray(case.U, dtype=t)
    rng = np.random.default_rng(5)
    w = rng.standard_normal(U.shape).astype(t)
    p = case.params()
    safe = bool(getattr(case, "safe", False))
    c = orc.config(**dict(p, integrator="euler"), safe=safe)
    U64 = U.astype(np.float64)
    dt = 0.3 * orc.compute_dt(c, U64)
    n = [int(x) for x in p["n"]]
    lam = p["mu"] * p["gamma"] * p["R"] / ((p["gamma"] - 1.0) * p["Pr"]) if p["heat"] else 0.0
    head = struct.pack("=i9i", int(dtype == "f64"), *n, *[int(p["bc"][2 * a] == 0) for a in range(3)], zchunk,
                       int(p["viscous"]), int(safe))
    head += struct.pack("=9d", *[n[a] / (p["hi"][a] - p["lo"][a]) for a in range(3)], p["gamma"], p["R"],
                        p["mu"] if p["viscous"] else 0.0, lam, p["eps"], dt)
    src, dst = tmp_path / "in", tmp_path / "out"
    src.write_bytes(head + U.tobytes() + w.tobytes())
    r = subprocess.run([program, str(src), str(dst)], capture_output=True, text=True, timeout=900,
                       env=dict(os.environ, ASAN_OPTIONS="detect_leaks=0:abort_on_error=1"))
    assert r.returncode == 0, r.stderr[-3000:]
    out = np.frombuffer(dst.read_bytes(), dtype=t).reshape(U.shape).astype(np.float64)
    assert np.isfinite(out).all()
    tol = 1e-12 if dtype == "f64" else 3e-5
    for _ in range(3):
        v = rng.standard_normal(U.shape)
        _, Jv = orc.jvp_run(c, U64, v, 1, dt)
        a, b = out * v, w.astype(np.float64) * Jv
        assert abs(a.sum() - b.sum()) <= tol * (np.abs(a).sum() + np.abs(b).sum()), (a.sum(), b.sum())
