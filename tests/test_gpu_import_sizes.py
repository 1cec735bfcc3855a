"""Imported sites come back bit for bit: more sites than one launch places, the packed
transfer and the site by site one for large states, after sites that were refused."""
import numpy as np
import pytest

from test_gpu_fp64 import T  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", ["C64", "C128"])
@pytest.mark.parametrize("n,chi", [(2, 2), (128, 3), (300, 5), (24, 80)])
def test_round_trip(T, n, chi, dt):  # noqa: F811
    rng = np.random.default_rng(n)
    d = [min(2 ** min(b, n - b, 20), chi) for b in range(n + 1)]
    sites = [rng.standard_normal((d[q], 2, d[q + 1])) + 1j * rng.standard_normal((d[q], 2, d[q + 1])) for q in range(n)]
    m = T.MPS(n, dtype=getattr(T, "TNSIM_" + dt), chi_max=chi)
    want = [s.astype(np.complex64).astype(complex) if dt == "C64" else s for s in sites]
    bad = [s.copy() for s in sites]
    bad[-1][0, 1, 0] = np.nan
    with pytest.raises(Exception):
        m.import_sites(bad)
    m.import_sites(sites)
    assert list(m.bond_dims()) == d
    for got, w in zip(m.export_sites(), want):
        assert np.array_equal(got, w)
    m.close()
