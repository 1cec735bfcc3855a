"""Read-out kernels at the edges of their tiles and groups.

Amplitudes: strings in groups (bonds >= 48 and at least 8 strings) must equal the per-string
kernel bit for bit (the same sums in the same order), which a call with 7 strings takes.
Expectation values: against numpy transfer matrices in complex128; each value is a sum of
2n products of n rounded factors, so complex64 stays within 1e-5 and complex128 within
1e-12 of the largest value.
"""
import numpy as np
import pytest

import workloads as W
from oracle import mps as om
from test_gpu_fp64 import T  # noqa: F401

pytestmark = pytest.mark.gpu


def _state(T, n, chi, dtype, seed=3):  # noqa: F811
    rng = np.random.default_rng(seed)
    d = [min(2 ** min(b, n - b, 30), chi) for b in range(n + 1)]
    sites = [(rng.standard_normal((d[q], 2, d[q + 1])) + 1j * rng.standard_normal((d[q], 2, d[q + 1])))
             / np.sqrt(4 * d[q + 1]) for q in range(n)]
    m = T.MPS(n, dtype=dtype, chi_max=chi)
    m.import_sites(sites)
    return m, sites


@pytest.mark.parametrize("chi", [48, 49, 63, 64, 65, 130, 256, 258, 333])
@pytest.mark.parametrize("count", [8, 9, 33, 70])
def test_amplitude_groups_equal_single_strings(T, chi, count):  # noqa: F811
    n = 20
    m, sites = _state(T, n, chi, T.TNSIM_C64)
    bits = W.random_bitstrings(n, count, seed=chi)
    bits[0], bits[1] = 0, 1
    got = m.amplitudes(bits)
    one = np.concatenate([m.amplitudes(bits[i:i + 7]) for i in range(0, count, 7)])
    assert np.array_equal(got, one)
    want = om.amplitudes(om.MPS(sites), bits[:4])
    assert np.linalg.norm(got[:4] - want) <= 1e-5 * np.linalg.norm(want)
    m.close()


@pytest.mark.parametrize("chi,n", [(1, 3), (4, 7), (15, 12), (16, 12), (17, 12), (40, 14)])
@pytest.mark.parametrize("dt,tol", [("C64", 1e-5), ("C128", 1e-12)])
def test_expectations(T, chi, n, dt, tol):  # noqa: F811
    m, sites = _state(T, n, chi, getattr(T, "TNSIM_" + dt))
    rng = np.random.default_rng(chi)
    paulis = ["I" * n, "Z" + "I" * (n - 1), "I" * (n - 1) + "Y", "X" * n, "Z" * n]
    paulis += ["".join(rng.choice(list("IIXYZ"), n)) for _ in range(30)]
    got = m.expect_pauli(paulis)
    want = np.array([om.expect_pauli(om.MPS(sites), p) for p in paulis])
    assert np.max(np.abs(got - want)) <= tol * np.max(np.abs(want))
    m.close()
