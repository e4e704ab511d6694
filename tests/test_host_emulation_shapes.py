"""The stage kernel's own source on the CPU, as in test_host_emulation.py, for
the families and tile shapes that file leaves out (tests/host_emu/emu_shapes.cpp):
component-split 1D tiles of FP64 at their remainders, the FP64 2D and 3D shapes,
the walled / WENO3-JS kernels per cell and per face, and the Rusanov-NN kernels
with their parameters in shared memory.  Every access stays inside buffers of
exactly the launch's size, vector accesses are aligned, and the right-hand side
matches the oracle: FP64 to 1e-12, FP32 to 1e-5."""
import ctypes
import json
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if __name__ == "__main__":
    sys.path.insert(0, ROOT)
    sys.path.insert(0, os.path.join(ROOT, "tests"))

import test_host_emulation as base  # noqa: E402
from paper_2203_13760_gb300 import inputs  # noqa: E402

W = inputs.WALL
SCHEME = {"flux": {"hllc": 0, "hll": 1, "rusanov": 2, "roe": 3, "rusanov-nn": 4},
          "recon": {"weno5-js": 0, "weno5-z": 1, "weno3-js": 2}, "speeds": {"einfeldt": 0, "davis": 1, "toro": 2}}

# (precision, kernel of emu_shapes.cpp, grid, boundaries, viscous, scheme, z chunk)
RUNS = [("f64", 0, (n, 1, 1), (1,) * 6, n > 30, {}, 1) for n in (5, 29, 30, 31, 61)]
RUNS += [
    ("f64", 1, (31, 1, 1), (W, 1, 1, 1, 1, 1), False, {"recon": "weno3-js"}, 1),
    ("f64", 1, (59, 1, 1), (W, W, 1, 1, 1, 1), False, {"flux": "hll", "recon": "weno5-z"}, 1),
    ("f64", 2, (37, 1, 1), (W, W, 1, 1, 1, 1), True, {"flux": "roe", "recon": "weno3-js"}, 1),
    ("f64", 3, (37, 1, 1), (0, 0, 1, 1, 1, 1), False, {"flux": "rusanov-nn"}, 1),
    ("f64", 4, (37, 11, 1), (0, 0, 1, 1, 1, 1), True, {}, 1),
    ("f64", 5, (33, 9, 1), (1,) * 6, False, {"flux": "rusanov"}, 1),
    ("f64", 6, (37, 11, 1), (W, W, 1, W, 1, 1), True, {"recon": "weno3-js"}, 1),
    ("f64", 6, (30, 5, 1), (W,) * 4 + (1, 1), False, {"recon": "weno3-js"}, 1),
    ("f64", 7, (37, 11, 1), (W, 1, W, W, 1, 1), False, {"speeds": "toro"}, 1),
    ("f64", 8, (33, 15, 9), (0, 0, 1, 1, 0, 0), True, {}, 4),
    ("f64", 9, (19, 9, 7), (W, W, 0, 0, W, 1), True, {}, 3),
    ("f64", 9, (33, 5, 6), (W,) * 6, False, {"recon": "weno3-js"}, 6),
    ("f64", 10, (37, 9, 1), (W, W, 1, W, 1, 1), False, {"flux": "rusanov-nn", "recon": "weno3-js"}, 1),
    ("f32", 0, (131, 1, 1), (W, 1, 1, 1, 1, 1), False, {"recon": "weno3-js"}, 1),
    ("f32", 1, (37, 11, 1), (W, W, 1, W, 1, 1), False, {"recon": "weno3-js"}, 1),
    ("f32", 2, (37, 11, 1), (W, W, 1, W, 1, 1), True, {"recon": "weno3-js"}, 1),
    ("f32", 2, (31, 17, 1), (W,) * 4 + (1, 1), False, {}, 1),
    ("f32", 3, (19, 9, 7), (W, W, 0, 0, W, 1), True, {"recon": "weno3-js"}, 3),
    ("f32", 3, (33, 8, 6), (W,) * 6, False, {"recon": "weno3-js"}, 6),
    ("f32", 4, (19, 9, 7), (W, W, 0, 0, W, 1), True, {"recon": "weno3-js"}, 4),
    ("f32", 4, (33, 8, 6), (W,) * 6, False, {}, 5),
    ("f32", 5, (37, 8, 1), (W, W, 1, W, 1, 1), False, {"flux": "rusanov-nn", "recon": "weno3-js"}, 1),
    ("f32", 6, (37, 11, 1), (W, W, 1, W, 1, 1), True, {"flux": "rusanov-nn"}, 1),
    ("f32", 7, (33, 8, 6), (W, W, 0, 0, 1, W), False, {"flux": "rusanov-nn", "recon": "weno3-js"}, 3),
]


def _case(i):
    dtype, kernel, n, bc, viscous, scheme, zchunk = RUNS[i]
    case = inputs.random_smooth(n, seed=40 + i, bc=bc, viscous=viscous, mu=0.01 if viscous else 0.0)
    for k, v in scheme.items():
        setattr(case, k, v)
    return dtype, kernel, case, zchunk


@pytest.fixture(scope="module")
def results(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("host_emu_shapes")
    src = d / "src"
    src.mkdir()
    shutil.copy(os.path.join(base.CSRC, "jf_math.cuh"), src)
    with open(os.path.join(base.CSRC, "stage.cuh")) as f:
        text = f.read()
    assert text.count(base.SMEM_DECL) == 1
    text = text.replace(base.SMEM_DECL, "unsigned char* smem_raw = emu_smem();")
    (src / "stage.cuh").write_text(text.replace("namespace jf {\n", "unsigned char* emu_smem();\nnamespace jf {\n", 1))
    san = base._sanitizer_libs()
    lib = str(d / "libemu_shapes.so")
    cmd = ["g++", "-std=c++20", "-O1", "-g1", "-fno-omit-frame-pointer", "-shared", "-fPIC",
           "-I", os.path.join(base.HERE, "cuda_stub"), "-I", str(src), os.path.join(base.HERE, "emu_shapes.cpp"),
           "-o", lib, "-lpthread"]
    if san:
        cmd[1:1] = ["-fsanitize=address,undefined", "-fno-sanitize-recover=undefined"]
    out = subprocess.run(cmd, capture_output=True, text=True)
    if out.returncode != 0 and "barrier" in out.stderr:
        pytest.skip("the C++ library has no std::barrier")
    assert out.returncode == 0, out.stderr[-3000:]
    env = dict(os.environ, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    if san:
        env.update(LD_PRELOAD=" ".join(san), ASAN_OPTIONS="detect_leaks=0:abort_on_error=1")
    width = max(1, min(4, (os.cpu_count() or 1) // 2))
    res, running, queue = {}, [], list(range(len(RUNS)))
    while queue or running:
        while queue and len(running) < width:
            i = queue.pop(0)
            running.append((i, subprocess.Popen([sys.executable, os.path.abspath(__file__), lib, str(i)],
                                                stdout=subprocess.PIPE, stderr=subprocess.PIPE, text=True, env=env)))
        i, p = running.pop(0)
        so, se = p.communicate(timeout=900)
        res[i] = json.loads(so.strip().splitlines()[-1]) if p.returncode == 0 else so[-2000:] + se[-4000:]
    return res


def _child(lib, i):
    import oracle as orc
    dtype, kernel, case, zchunk = _case(i)
    t = np.float64 if dtype == "f64" else np.float32
    theta = inputs.nn_params().astype(t) if case.flux == "rusanov-nn" else None
    p = case.params()
    n = [int(x) for x in p["n"]]
    periodic = [1 if p["bc"][2 * a] == 0 else 0 for a in range(3)]
    wall = [(p["bc"][2 * a] == W) + 2 * (p["bc"][2 * a + 1] == W) for a in range(3)]
    inv_h = [n[a] / (p["hi"][a] - p["lo"][a]) for a in range(3)]
    mu = p["mu"] if p["viscous"] else 0.0
    lam = p["mu"] * p["gamma"] * p["R"] / ((p["gamma"] - 1.0) * p["Pr"]) if p["heat"] else 0.0
    gas = [p["gamma"], p["R"], mu, lam, p["eps"]] + [float(SCHEME[k][p[k]]) for k in ("flux", "recon", "speeds")]
    U = np.ascontiguousarray(case.U, dtype=t)
    got = np.zeros_like(U)
    ip = lambda v: (ctypes.c_int * 3)(*[int(x) for x in v])  # noqa: E731
    dp = lambda v: (ctypes.c_double * len(v))(*v)  # noqa: E731
    vp = lambda a: a.ctypes.data_as(ctypes.c_void_p) if a is not None else None  # noqa: E731
    fn = getattr(ctypes.CDLL(lib), "emu_rhs_" + dtype)
    fn.restype = ctypes.c_int
    flag = fn(kernel, ip(n), ip(periodic), ip(wall), dp(inv_h), dp(gas), zchunk, vp(theta), vp(U), vp(got))
    assert flag == 0, flag
    c = orc.config(**p, nn=None if theta is None else theta.astype(np.float64))
    want = orc.rhs(c, U.astype(np.float64))
    rate = case.cfl / orc.compute_dt(c, U.astype(np.float64))
    err = 0.0
    for g in base.GROUPS:
        w, x, u = (a.reshape(5, -1)[list(g)].astype(np.float64) for a in (want, got, U))
        err = max(err, np.abs(x - w).max() / max(np.abs(w).max(), np.abs(u).max() * rate, 1e-300))
    return err


@pytest.mark.parametrize("i", range(len(RUNS)), ids=[f"{r[0]}-k{r[1]}-{r[2][0]}x{r[2][1]}x{r[2][2]}" for r in RUNS])
def test_emulated_shape_vs_oracle(results, i):
    assert isinstance(results[i], float), results[i]
    assert results[i] <= (1e-12 if RUNS[i][0] == "f64" else 1e-5)


if __name__ == "__main__":
    print(json.dumps(float(_child(sys.argv[1], int(sys.argv[2])))))
