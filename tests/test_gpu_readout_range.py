"""Expectation values of complex64 states that are far from normalised.

The left and right environment of the middle bond are each near the end of FP32's range
(1e36 or 1e-36); their product is a number of FP64 only.  Sites of squared norm 1e12 or 1e-12
per left index; values to 1e-5 of the largest, as in the other complex64 read-out tests.
"""
import numpy as np
import pytest

from test_gpu_fp64 import T  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e12, 1.0, 1e-12])
@pytest.mark.parametrize("chi", [1, 5])
def test_unnormalised_states(T, scale, chi):  # noqa: F811
    n = 6
    rng = np.random.default_rng(3)
    d = [min(2 ** min(b, n - b), chi) for b in range(n + 1)]
    sites = [rng.standard_normal((d[q], 2, d[q + 1])) + 1j * rng.standard_normal((d[q], 2, d[q + 1])) for q in range(n)]
    sites = [a * np.sqrt(scale / (np.linalg.norm(a) ** 2 / d[q])) for q, a in enumerate(sites)]
    ops = {"I": np.eye(2), "X": np.array([[0, 1], [1, 0]]), "Y": np.array([[0, -1j], [1j, 0]]), "Z": np.diag([1, -1])}
    # supports that close at the middle bond
    paulis = ["IIZIII", "IIXIII", "IXYIII"]

    def value(p):
        e = np.ones((1, 1), complex)
        for a, c in zip(sites, p):
            e = np.einsum("xy,xpa,pq,yqb->ab", e, a.conj(), ops[c], a, optimize=True)
        return e[0, 0]

    want = np.array([value(p) for p in paulis])
    m = T.MPS(n, dtype=T.TNSIM_C64, chi_max=max(chi, 2))
    m.import_sites(sites)
    got = m.expect_pauli(paulis)
    m.close()
    assert np.max(np.abs(got - want)) <= 1e-5 * np.max(np.abs(want))
