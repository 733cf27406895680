"""The group-of-lanes collision and adjoint (csrc/lane_cell.cuh), compiled as host code with a group
of one lane, against the oracle's collision and the one-thread adjoint. Both sides are double with
the same formulas and other summation orders: 1e-13 of the largest value (a few hundred roundings of
2^-53). Runs on the CPU (nvcc needed)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import paper_2401_11086_gb300 as P
from oracle import lattice as OL
from oracle import smrt as OS
from _lb import lib_from_oracle

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "native", "lane_cell_host.cu")
OUT = os.path.join(ROOT, "paper_2401_11086_gb300", "_build", "lane_cell_host_test.so")
SETS = [("D3Q39", 3), ("D3Q103", 3), ("D3Q103", 4)]


@pytest.fixture(scope="module")
def host():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    os.makedirs(os.path.dirname(OUT), exist_ok=True)
    subprocess.run([nvcc, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", SRC,
                    "-o", OUT], check=True, capture_output=True)
    return ctypes.CDLL(OUT)


def _p(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


def _cells(name, N, maxwell):
    olat = OL.by_name(name)
    d = P.lb_lattice_named(name)
    idx = lib_from_oracle(olat, d)
    rng = np.random.default_rng(11)
    n = 4
    f = OS.equilibrium(1 + 0.3 * rng.random(n), 0.3 * rng.standard_normal((3, n)), 0.8 + 0.4 * rng.random(n), olat, N)
    f = f * (1 + 0.05 * rng.standard_normal(f.shape))
    nt = sum(k // 2 + 1 for k in range(2, N + 1))
    taus = 0.5 + rng.random(nt)
    A = taus * 1.3 if maxwell else np.zeros(nt)
    B = np.full(nt, 0.5) if maxwell else taus + 0.5
    wp = np.concatenate([[d.w[0]], d.w[1::2]])
    return olat, d, idx, rng, f, taus, A, B, wp


@pytest.mark.parametrize("name,N", SETS)
@pytest.mark.parametrize("b", [None, -0.5, 0.3])
def test_collision_matches_oracle(host, name, N, b):
    olat, d, idx, _, f, taus, A, B, wp = _cells(name, N, True)
    keys = [(n, m) for n in range(2, N + 1) for m in range(n // 2 + 1)]
    model = OS.Model(olat, N, tau_ref=1.0, maxwell_law=True, rho_ref=1.3,
                     tau_star=dict(zip(keys, taus)), **({} if b is None else {"es_b": b}))
    want = OS.collide(f, model)
    fn = getattr(host, f"step_{name.lower()}_n{N}")
    for c in range(f.shape[1]):
        x, out = np.ascontiguousarray(f[idx, c] - d.w), np.zeros(olat.q)
        fn(_p(x), ctypes.c_double(d.c), _p(wp), _p(A), _p(B), int(b is not None), ctypes.c_double(b or 0.0), _p(out))
        assert np.abs(out + d.w - want[idx, c]).max() < 1e-13 * np.abs(want).max()


@pytest.mark.parametrize("name,N", SETS)
@pytest.mark.parametrize("maxwell", [True, False])
def test_adjoint_matches_the_one_thread_form(host, name, N, maxwell):
    olat, d, idx, rng, f, taus, A, B, wp = _cells(name, N, maxwell)
    dA, dB = (1.3, 0.0) if maxwell else (0.0, 1.0)
    for c in range(f.shape[1]):
        x, lam = np.ascontiguousarray(f[idx, c] - d.w), rng.standard_normal(olat.q)
        got, want = [], []
        for tag, res in (("vjp", got), ("vjpt", want)):
            fb, tb = np.zeros(olat.q), np.zeros(len(taus))
            getattr(host, f"{tag}_{name.lower()}_n{N}")(
                _p(x), _p(lam), ctypes.c_double(d.c), _p(wp), _p(A), _p(B), ctypes.c_double(dA), ctypes.c_double(dB),
                _p(fb), _p(tb))
            res += [fb, tb]
        for g, w in zip(got, want):
            assert np.abs(g - w).max() < 1e-13 * np.abs(w).max()
