"""The collisions that the FP64 steps and the plain and Powell FP32 steps run
(ideal_collide_f64, ideal_collide_f32 and the table-driven Powell and solid forms),
compiled for the host from the kernels' own source, against the oracle cell by cell
on D2Q5 and D3Q7 with uniform sources, and the non-physical flag.

test_cell_host.py covers the 16-bit, corrected and dissipative forms; its plain
entries call ideal_collide, which of the plain steps only the corrected one runs."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from test_cell_host import F32_TOL, FLAG_NONPHYSICAL, HERE, ROOT, _cells, _check, _deps, _inputs, _p

SRC = os.path.join(HERE, "cell_host_steps.cu")
LIB = os.path.join(HERE, "_build", "libcellhoststeps.so")
S8 = np.array([0.0, 1e-3, -2e-3, 5e-4, 1e-4, 2e-4, -1e-4, 3e-4])


@pytest.fixture(scope="module")
def H():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    if not os.path.exists(LIB) or any(os.path.getmtime(p) > os.path.getmtime(LIB) for p in _deps() + [SRC]):
        os.makedirs(os.path.dirname(LIB), exist_ok=True)
        tmp = LIB + ".%d.tmp" % os.getpid()
        cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "--expt-relaxed-constexpr",
               "-Xcompiler", "-fPIC", "-Xcompiler", "-ffp-contract=off",
               "-I", os.path.join(ROOT, "paper_2606_00641_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
               "-shared", SRC, "-o", tmp]
        res = subprocess.run(cmd, capture_output=True, text=True)
        assert res.returncode == 0, res.stdout + res.stderr
        os.replace(tmp, LIB)
    L = ctypes.CDLL(LIB)
    i, p = ctypes.c_int, ctypes.c_void_p
    for prec, r in (("f64", ctypes.c_double), ("f32", ctypes.c_float)):
        getattr(L, "hs_ideal_" + prec).argtypes = [i, r, p, p, p, p, p]
        getattr(L, "hs_powell_" + prec).argtypes = [i, r, p, p, p, r, p, p]
    L.hs_hom_f64.argtypes = [i, ctypes.c_double, p, p, p, ctypes.c_double, p, p, p, p]
    return L


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("model", ["ideal", "powell"])
def test_step_collision_matches_the_oracle(H, model, prec, dim):
    nl, tau_m = (9, 3.0) if model == "powell" else (8, None)
    gamma, cells = _cells(dim, 71 + dim, nl=nl)
    S = np.concatenate([S8, np.zeros(nl - 8)])
    dtype = np.float64 if prec == "f64" else np.float32
    tau, omega, src0, src1 = _inputs(dim, nl, dtype, S)
    fn = getattr(H, "hs_%s_%s" % (model, prec))
    flags = np.zeros(1, np.uint32)
    for c in cells:
        got = c.astype(dtype)
        extra = (1.0 / tau_m,) if tau_m else ()
        assert fn(dim, gamma - 1.0, _p(omega), _p(src0), _p(src1), *extra, _p(got), _p(flags)) == 0
        ref = oracle.powell_collide_cell(dim, gamma, tau, tau_m, c, src=S) if tau_m else \
            oracle.ideal_collide_cell(dim, gamma, tau, c, src=S)
        _check(got.astype(np.float64), ref, 1e-13 if prec == "f64" else F32_TOL)
    assert flags[0] == 0


@pytest.mark.parametrize("dim", [2, 3])
def test_solid_collision_from_the_table_matches_the_oracle(H, dim):
    # the oracle's step on a one-cell periodic grid is the collision alone
    gamma, cells = _cells(dim, 81 + dim)
    tau, omega, src0, src1 = _inputs(dim, 8, np.float64, S8)
    rng = np.random.default_rng(8)
    flags = np.zeros(1, np.uint32)
    one = (1,) * dim
    for n, c in enumerate(cells):
        d = [0.0, 1.0, 0.3, 0.75][n % 4]
        uB, BB = 0.05 * rng.normal(size=3), 0.1 * rng.normal(size=3)
        got = c.copy()
        assert H.hs_hom_f64(dim, gamma - 1.0, _p(omega), _p(src0), _p(src1), d, _p(uB), _p(BB), _p(got), _p(flags)) == 0
        solid = np.concatenate([[d], uB, BB]).reshape((7,) + one)
        _check(got, oracle.hlbm_step(c.reshape(c.shape + one), gamma, tau, solid, src=S8).reshape(c.shape), 1e-13)
    assert flags[0] == 0


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("bad", ["energy", "density", "nan"])
def test_non_physical_cell_raises_the_flag(H, bad, prec, dim):
    gamma, cells = _cells(dim, 91)
    dtype = np.float64 if prec == "f64" else np.float32
    c = cells[0].astype(dtype)
    if bad == "energy":
        c[4] *= -1
    elif bad == "density":
        c[0] *= -1
    else:
        c[0, 1] = np.nan
    tau, omega, src0, src1 = _inputs(dim, 8, dtype, np.zeros(8))
    flags = np.zeros(1, np.uint32)
    fn = getattr(H, "hs_ideal_" + prec)
    assert fn(dim, gamma - 1.0, _p(omega), _p(src0), _p(src1), _p(c), _p(flags)) == 0
    assert flags[0] & FLAG_NONPHYSICAL
    assert fn(4, gamma - 1.0, _p(omega), _p(src0), _p(src1), _p(c), _p(flags)) == -1
