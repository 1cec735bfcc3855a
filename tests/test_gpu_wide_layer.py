"""One complex128 layer of 33000 gates (a grid dimension holds 65535), each large enough for
the preconditioner: 66000 qubits at bond dimension 16, a few kinds of site in turn."""
import numpy as np
import pytest

import workloads as W
from test_gpu_fp64 import T  # noqa: F401

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


def test_layer_of_33000_preconditioned_gates(T):  # noqa: F811
    n, chi, kinds = 66000, 16, 6
    rng = np.random.default_rng(5)
    d = [min(2 ** min(b, n - b, 30), chi) for b in range(n + 1)]

    def site(l, r):
        return (rng.standard_normal((l, 2, r)) + 1j * rng.standard_normal((l, 2, r))) / np.sqrt(4 * r)

    bulk = [site(chi, chi) for _ in range(kinds)]
    sites = [bulk[q % kinds] if d[q] == d[q + 1] == chi else site(d[q], d[q + 1]) for q in range(n)]
    gates = np.stack([W.haar_su4(rng) for _ in range(kinds)])
    pairs = np.arange(0, n - 1, 2, dtype=np.int32)
    m = T.MPS(n, dtype=T.TNSIM_C128, chi_max=chi, renormalize=False)
    m.import_sites(sites)
    m.apply_layer(W.Layer(pairs, gates[(pairs // 2) % kinds], None))
    for q in (1000, 1002, 33000, 65534 // 2 * 2, 65536, 65900):
        t = (sites[q].reshape(2 * chi, chi) @ sites[q + 1].reshape(chi, 2 * chi)).reshape(chi, 2, 2, chi)
        t = np.einsum("abcd,lcdr->labr", gates[(q // 2) % kinds].reshape(2, 2, 2, 2), t).reshape(2 * chi, 2 * chi)
        want = np.linalg.svd(t, compute_uv=False)[:chi]
        assert np.max(np.abs(m.spectrum(q + 1) - want)) <= 64 * EPS * np.sqrt(chi) * want[0]
    m.close()
