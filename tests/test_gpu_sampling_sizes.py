"""Perfect sampling at the edges of its tiles: odd numbers of columns, one and two blocks of
128 columns, groups of 2 and of 8 nodes per CTA with remainders, and draws in one CTA and in
several.  complex128 bits equal the oracle's; complex64 shots leave its path only where the
uniform is within 1e-4 of the oracle's weight, in at most 2 % of the shots (the bars of
test_gpu_sampling.py)."""
import numpy as np
import pytest

from oracle import mps as om
from test_gpu_sampling import T, _check_against_oracle, _distinct_prefixes  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", ["C64", "C128"])
@pytest.mark.parametrize("n,chi,shots", [(6, 3, 7), (12, 33, 300), (16, 127, 301), (18, 150, 700), (17, 64, 2500),
                                         (10, 17, 9000)])
def test_sizes(T, n, chi, shots, dt):  # noqa: F811
    rng = np.random.default_rng(n * chi)
    d = [min(2 ** min(b, n - b), chi) for b in range(n + 1)]
    sites = [(rng.standard_normal((d[q], 2, d[q + 1])) + 1j * rng.standard_normal((d[q], 2, d[q + 1])))
             / np.sqrt(4 * d[q]) for q in range(n)]
    m = T.MPS(n, dtype=getattr(T, "TNSIM_" + dt), chi_max=chi)
    m.import_sites(sites)
    ref = om.MPS(m.export_sites())
    u = rng.random((shots, n))
    bits, nodes = T.tnsim_sample(m.h, u)
    m.close()
    want = om.perfect_sample_u(ref, u)
    if dt == "C128":
        assert np.array_equal(bits, want)
    else:
        _check_against_oracle(bits, want, ref, u, 0.02)
    assert nodes == _distinct_prefixes(bits)
