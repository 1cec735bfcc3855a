"""The prefetching Jacobi kernel (complex64, 258 to 512 rows) while its warps claim ahead.

Whether a visit's end finds the next one already claimed is decided by timing, so one layer
is run many times: every decision has to leave every warp in step, and the arithmetic does
not depend on it, so the sites are equal bit for bit each time.  Gates of several sizes: few
visits left, visits without a partner and one-block gates at the ends of the chain.
"""
import numpy as np
import pytest

import workloads as W
from test_gpu_fp64 import T  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,chi,reps", [(24, 150, 12), (70, 130, 8)])
def test_repeated_layers_agree_bitwise(T, n, chi, reps):  # noqa: F811
    rng = np.random.default_rng(n)
    d = [min(2 ** min(b, n - b, 30), chi) for b in range(n + 1)]
    sites = [((rng.standard_normal((d[q], 2, d[q + 1])) + 1j * rng.standard_normal((d[q], 2, d[q + 1])))
              / np.sqrt(4 * d[q + 1])).astype(np.complex64).astype(np.complex128) for q in range(n)]
    lay = W.brickwork_su4(n, 1, seed=3).layers[0]
    m = T.MPS(n, dtype=T.TNSIM_C64, chi_max=chi)
    first = None
    for _ in range(reps):
        m.import_sites(sites)
        m.apply_layer(lay)
        out = m.export_sites()
        first = first or out
        assert all(np.array_equal(a, b) for a, b in zip(out, first))
    m.close()
