"""Complex64 rotations near the end of FP32's range, columns of exactly equal norm.

theta = [[x, y], [y, x]]: both columns have the norm x^2 + y^2 and the inner product 2 x y,
whose square is finite up to 1.8e19; the singular values are x + y and |x - y|.  To 1e-5 of
s_max, as in the other complex64 tests.
"""
import numpy as np
import pytest

import workloads as W
from test_gpu_fp64 import T  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g", [1e-10, 1.0, 1e15, 4e18, 6e18, 1e19, 1.5e19])
@pytest.mark.parametrize("cfg", [0, 1])
def test_equal_norms(T, g, cfg):  # noqa: F811
    # x = 2 y, so that the inner product 2 x y = 4 y^2 is g
    y = np.sqrt(g / 4.0)
    th = y * np.array([[2.0, 1.0], [1.0, 2.0]])
    m = T.MPS(2, dtype=T.TNSIM_C64, chi_max=2, renormalize=False)
    if cfg:
        T.tnsim_set_jacobi_config(m.h, cfg)
    m.import_sites([np.eye(2).reshape(1, 2, 2) * np.sqrt(y), (th / np.sqrt(y)).reshape(2, 2, 1)])
    m.apply_layer(W.Layer(np.array([0], np.int32), np.eye(4, dtype=complex)[None], None))
    s = m.spectrum(1)
    m.close()
    assert len(s) == 2 and np.max(np.abs(s - y * np.array([3.0, 1.0]))) <= 1e-5 * 3 * y
