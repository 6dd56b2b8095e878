"""The moment bounds with 6 / 8 power and 3 / 4 trigonometric moments in the
library's float32 arithmetic (compiled for the host) against their definition
in 64 bits: the kernel polynomial's roots and Christoffel weights by numpy.

Tolerance: float32 rounding (2^-24) times the condition of the biased moment
matrix, which the bias bounds.  Trigonometric: (n + 1) / beta <= 2500 at beta
= 2e-3, so 1.5e-4.  Power: the standardised Hankel matrix at beta = 5e-5; a
unit of its smallest pivot is about beta / 6, so 2^-24 * 6 / beta < 7.2e-3 in
the worst case for one value; over all values the root mean square stays
below a thousandth of it."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LAW = np.array([1, 0, 0.5, 0, 0.375, 0, 0.3125, 0, 0.2734375])


def _power(m, z, n, w0, beta):
    b = (1 - beta) * m / m[0] + beta * LAW
    H = np.array([[b[i + j] for j in range(n + 1)] for i in range(n + 1)])
    v = lambda x: x ** np.arange(n + 1)  # noqa: E731
    weight = lambda x: 1 / (v(x) @ np.linalg.solve(H, v(x)))  # noqa: E731
    roots = np.roots(np.linalg.solve(H, v(z))[::-1]).real
    return w0 * weight(z) + sum(weight(x) for x in roots if x < z)


def _trig(tau, z, n, w0, beta):
    t = np.concatenate([[1], (1 - beta) * tau[:n]])
    G = np.linalg.inv([[t[l - k] if l >= k else np.conj(t[k - l]) for l in range(n + 1)] for k in range(n + 1)])
    v = lambda u: u ** np.arange(n + 1)  # noqa: E731
    weight = lambda u: 1 / (v(u) @ G @ np.conj(v(u))).real  # noqa: E731
    u0 = np.exp(1j * z * float(np.float32(0.9 * np.pi)))
    roots = np.roots((G @ np.conj(v(u0)))[::-1])
    return w0 * weight(u0) + sum(weight(u) for u in roots / np.abs(roots) if np.angle(u) < np.angle(u0))


def test_bounds_against_64_bits(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "bound_check"
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", "-include", "math.h",
                           "-I", os.path.join(ROOT, "paper_2501_12581_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "bound_check.cpp"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    rows = np.array([[float(x) for x in line.split()] for line in out.splitlines()])
    w0, bp, bt = (float(np.float32(x)) for x in (0.3, 5e-5, 2e-3))
    err = np.empty((len(rows), 4))
    for r, e in zip(rows, err):
        m, tau = r[5:14], r[14::2] + 1j * r[15::2]
        e[:] = np.abs(r[1:5] - [_power(m, r[0], 3, w0, bp), _power(m, r[0], 4, w0, bp),
                                _trig(tau, r[0], 3, w0, bt), _trig(tau, r[0], 4, w0, bt)])
    assert np.isfinite(err).all() and len(err) == 2400
    assert (err[:, :2] <= 7.2e-3).all() and (np.sqrt((err[:, :2] ** 2).mean(0)) <= 7.2e-6).all(), err.max(0)
    assert (err[:, 2:] <= 1.5e-4).all(), err.max(0)
