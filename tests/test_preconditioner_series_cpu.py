"""The series by which the complex128 preconditioner makes its transformation unitary.

V, a product of FP32 rotations, has V^H V = I - E; the kernels form I + F as
    F = E/2 + B - K^4/8 + E R,   R = 3/8 E + B/2 + E (5/16 E + 3/8 B),   B = K + K^2/2
(K anti-Hermitian), so that V (I + F) is unitary.  In extended precision, at the sizes that
occur (|E|_2 = 5e-6, and K as large as its row sums admit: |K^2|_inf <= 2^-17), the defect has
to be that of the terms left out, 2 (|K|^6 / 16 + |E| |K|^4 / 16) < 1.2e-16.  Without the
product of E^2 and K it is 8e-15.
"""
import numpy as np


def _norm(a):
    return np.linalg.norm(a.astype(np.complex128), 2)


def _inputs(n=48, seed=1):
    rng = np.random.default_rng(seed)
    a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    e = a + a.conj().T
    # one strong direction: row sums near the norm, the worst case of the bound
    v = np.exp(2j * np.pi * rng.random(n)) / np.sqrt(n)
    k = 1j * np.outer(v, v.conj()) + 1e-2 * (a - a.conj().T) / _norm(a)
    e, k = e.astype(np.clongdouble) * (5e-6 / _norm(e)), k.astype(np.clongdouble)
    k = k * np.sqrt(np.longdouble(2.0 ** -17) / np.abs(k @ k).sum(axis=1).max())
    return e, k


def _defect(e, f):
    one = np.eye(len(e), dtype=np.clongdouble)
    g = one + f
    return _norm(g.conj().T @ (one - e) @ g - one)


def test_defect_of_the_correction():
    e, k = _inputs()
    k2 = k @ k
    b = k + k2 / 2
    r = np.longdouble(3) / 8 * e + b / 2 + e @ (np.longdouble(5) / 16 * e + np.longdouble(3) / 8 * b)
    f = e / 2 + b - k2 @ k2 / 8 + e @ r
    assert _norm(k) > 2.5e-3
    assert _defect(e, f) <= 1.2e-16
