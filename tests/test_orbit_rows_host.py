"""The run-time orbit rows of the split-precision step (csrc/lattices.cuh), compiled as host code,
against the library's velocity vectors: every population is in exactly one row, v^gamma =
a^gamma (-1)^popcount(b & c) for every member b and slot up to the highest order, with c the
slot's transform entry, and the staged offsets are population x row length - e_x. Runs on the
CPU (nvcc needed)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import paper_2401_11086_gb300 as P

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "native", "orbit_rows_host.cu")
OUT = os.path.join(ROOT, "paper_2401_11086_gb300", "_build", "orbit_rows_host_test.so")


@pytest.fixture(scope="module")
def host():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    os.makedirs(os.path.dirname(OUT), exist_ok=True)
    subprocess.run([nvcc, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", SRC,
                    "-o", OUT], check=True)
    return ctypes.CDLL(OUT)


@pytest.mark.parametrize("name,N", [("D3Q39", 3), ("D3Q103", 3), ("D3Q103", 4)])
def test_rows_hold_every_population_once_and_factor_every_monomial(host, name, N):
    e = P.lb_lattice_named(name).e.astype(int)          # library population order
    M = (N + 1) * (N + 2) * (N + 3) // 6
    ip = lambda a: a.ctypes.data_as(ctypes.POINTER(ctypes.c_int))  # noqa: E731
    rows, mono, cls = (np.zeros(64 * n, dtype=np.int32) for n in (30, M, M))
    seg = np.zeros(1, dtype=np.int32)
    n = getattr(host, f"rows_{name.lower()}")(N, ip(rows), ip(mono), ip(cls), ip(seg))
    comp = np.zeros(3 * M, dtype=np.int32)
    host.slot_components(N, ip(comp))
    comp = comp.reshape(M, 3)
    assert seg[0] % 4 == 0 and seg[0] >= 32 + 2 * np.abs(e[:, 0]).max() + 3
    seen = [0]                                          # the rest population is in no row
    for r, mo, cl in zip(rows.reshape(-1, 30)[:n], mono.reshape(-1, M), cls.reshape(-1, M)):
        for b in range(r[1]):
            m = r[2 + 7 * b: 9 + 7 * b]
            v, (p, q) = m[:3], m[3:5]
            assert list(e[p]) == list(v) and list(e[q]) == list(-v)
            assert r[0] == sum(1 << d for d in range(3) if v[d])
            assert m[5] == p * seg[0] - v[0] and m[6] == q * seg[0] + v[0]
            seen += [int(p), int(q)]
            for g in range(M):
                assert np.prod(v ** comp[g]) == mo[g] * (-1) ** bin(b & cl[g]).count("1")
    assert sorted(seen) == list(range(len(e)))
