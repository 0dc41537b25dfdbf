"""Host logic of the folded full-grid sums (no GPU): the planned chunks and
tables against direct sums over every bin, with the oracle's phase."""
import json
import os
import shutil
import subprocess

import numpy as np
import pytest

import swig_inputs as si
from oracle import physics

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NB, DEG, SLOPES, NODES = 11, 8, 10, 64
D1 = 2 * NB
POLY = D1 + 2 * SLOPES
BND = POLY + (DEG - 1) * SLOPES
FC = BND + SLOPES
H, SM, LIM, ROWS = FC + 2, FC + 4, FC + 6, FC + 8
BNS = [(1.5, 2.5), (0.5, 1.0), (-0.05, 0.05), (-0.05, 0.05), (0.0, 5000.0), (0.0, 5000.0)]
H1_4S = [(1.1, 1.3), (0.5, 1.0), (0.0, 0.0), (0.0, 0.0), (0.0, 0.0), (0.0, 0.0)]
WIDE = [(0.87, 3.0), (0.125, 1.0), (-0.1, 0.1), (-0.1, 0.1), (0.0, 5000.0), (0.0, 5000.0)]
GRIDS = [  # f_min, f_max, df, box, most chunks
    (20.0, 2048.0, 1 / 128, BNS, 100), (20.0, 1500.0, 1 / 37, BNS, 100), (20.0, 1024.0, 0.25, H1_4S, 120),
    (20.0, 2048.0, 1 / 64, WIDE, 400), (20.0, 200.0, 1 / 16, H1_4S, 90), (30.0, 31.0, 1 / 16, BNS, 4),
]
TC, DELAY = 0.1, 0.0213


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    from paper_2607_28265_gb300 import build, swig
    if not os.path.exists(swig.LIB_PATH):
        build.build()
    lib_dir = os.path.dirname(swig.LIB_PATH)
    exe = str(tmp_path_factory.mktemp("host") / "fold_harness")
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2607_28265_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "fold_harness.cu"), "-o", exe, "-L", lib_dir, "-lswig",
                        "-Xlinker", "-rpath", "-Xlinker", lib_dir], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    return exe


def _plan(exe, f_min, f_max, df, box):
    args = ["plan", f_min, f_max, df, -TC, TC, DELAY] + [v for b in box for v in b]
    r = subprocess.run([exe] + [repr(float(a)) if not isinstance(a, str) else a for a in args], capture_output=True,
                       text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    out = json.loads(r.stdout)
    out["table"] = np.array(out["table"], dtype=np.float32).astype(np.float64).reshape(out["rows"], -1)
    out["x"] = np.array(out["x"], dtype=np.float32).astype(np.float64).sum(1).reshape(-1, 32)
    assert out["rows"] == ROWS
    return out


def _coeffs(exe, v):
    """Phase-basis coefficients of (Mc q chi1 chi2 L1 L2) by the library's set-up code."""
    r = subprocess.run([exe, "coeffs"] + [repr(float(x)) for x in v], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
    return np.array(json.loads(r.stdout))


def _draw(rng, box):
    return np.array([lo + (hi - lo) * rng.random() for lo, hi in box])


@pytest.mark.parametrize("grid", GRIDS)
def test_chunks_tile_the_grid(harness, grid):
    out = _plan(harness, *grid[:4])
    k = 0
    for k0, nb, kind, _ in out["chunks"]:
        assert k0 == k and nb >= 1
        assert nb > NODES if kind == 0 else nb <= (2 * NODES >> kind)
        k += nb
    assert k == out["n_bins"] and len(out["chunks"]) <= grid[4]
    assert np.isfinite(out["table"]).all() and np.abs(out["x"]).max() <= 1.0


@pytest.mark.parametrize("grid", GRIDS)
def test_folded_sums_equal_the_sums_over_every_bin(harness, grid):
    """kappa from the nodes, read as the device reads the table (centre value,
    Taylor terms of the scaled offset, reference slope), against the direct
    sum over every bin, for templates of the prior box and random data: the
    planned interpolation (1e-8) and Taylor errors (2e-8 cycles) bound the
    difference by 1.4e-7 of sum |D| in the worst case and by that of the root
    of sum |D|^2 for random data (bound: ten times as much)."""
    f_min, f_max, df, box, _ = grid
    out = _plan(harness, f_min, f_max, df, box)
    T, X = out["table"], out["x"]
    n = out["n_bins"]
    f = (out["k_min"] + np.arange(n)) * df
    rng = np.random.default_rng(4)
    D = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    W = []
    for q, (k0, nb, kind, sh) in enumerate(out["chunks"]):
        fc, h = T[FC, q] + T[FC + 1, q], T[H, q] + T[H + 1, q]
        x = (f[k0:k0 + nb] - fc) / h
        d = D[k0:k0 + nb] * np.exp(-2j * np.pi * sh * x)
        if kind:
            bw = 2 * NODES >> kind
            w = np.zeros(NODES, complex)
            for k in range(nb):  # node +x_l: bin bw / 2 + l, node -x_l: bin bw / 2 - 1 - l
                w[k - bw // 2 if k >= bw // 2 else 32 + bw // 2 - 1 - k] = d[k]
        else:
            V = np.polynomial.chebyshev.chebvander(x, NODES - 1)
            xn = np.concatenate([X[0], -X[0]])
            C = np.polynomial.chebyshev.chebvander(xn, NODES - 1)
            C[:, 0] *= 0.5
            w = (2.0 / NODES) * C @ (V.T @ d)
        W.append(w)
    scale = np.sqrt(np.sum(np.abs(D) ** 2))
    for _ in range(3):
        v = _draw(rng, box)
        c = _coeffs(harness, v)
        tau = rng.uniform(-TC - DELAY, TC + DELAY)
        want = np.sum(D * np.exp(-1j * physics.taylorf2_phase_intrinsic(f, *v) - 2j * np.pi * f * tau))
        got = 0.0
        for q, (k0, nb, kind, sh) in enumerate(out["chunks"]):
            fc, h = T[FC, q] + T[FC + 1, q], T[H, q] + T[H + 1, q]
            x = np.concatenate([X[kind], -X[kind]])
            A = c @ (T[:NB, q] + T[NB:D1, q])
            S = c[:SLOPES] @ (T[D1:D1 + SLOPES, q] + T[D1 + SLOPES:POLY, q]) + h * tau - (T[SM, q] + T[SM + 1, q])
            a = [c[:SLOPES] @ T[POLY + m * SLOPES:POLY + (m + 1) * SLOPES, q] for m in range(DEG - 1)]
            g, om = 1.0, abs(S)
            for m, am in enumerate(a):
                g *= 0.5 * (3.0 + 1.0 / 3.0)
                om += (m + 2) * g * abs(am)
            assert om <= T[LIM, q]  # the device would take these chunks folded
            assert np.abs(c[:SLOPES]) @ T[BND:BND + SLOPES, q] <= 1e-7
            ph = A + fc * tau + S * x + sum(am * x ** (m + 2) for m, am in enumerate(a))
            got = got + np.sum(W[q] * np.exp(-2j * np.pi * ph))
        assert abs(got - want) <= 1.4e-6 * scale, (abs(got - want) / scale)

