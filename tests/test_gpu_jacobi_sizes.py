"""The Jacobi kernels at the edges of their layouts, complex64.

Sizes around the lanes-per-pair steps (m = 64, 128, 256, 512), the 16-column blocks (odd and
even block counts, one block) and the largest cluster (n = 256); rectangular blocks.  The
tolerances are those of the other complex64 tests: singular values within 1e-5 of s_max, the
new two-site block within 1e-5.
"""
import numpy as np
import pytest

import workloads as W
from test_gpu_fp64 import T, _update  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg", [0, 1, 2])
@pytest.mark.parametrize("c", [(2, 3, 2), (8, 8, 8), (9, 8, 8), (16, 16, 16), (17, 16, 24), (32, 32, 32), (33, 33, 32),
                               (64, 64, 64), (65, 40, 64), (40, 65, 65), (128, 128, 128), (129, 100, 128),
                               (100, 100, 129), (256, 256, 256), (140, 140, 137)])
def test_block_sizes(T, c, cfg):  # noqa: F811
    s, r, blk, blk_o, u = _update(T, *c, chi=1, cfg=cfg, dtype=T.TNSIM_C64)
    k = min(len(s), r.k)
    assert np.max(np.abs(s[:k] - r.s_kept[:k])) <= 1e-5 * r.s_kept[0]
    assert np.linalg.norm(blk - blk_o) <= 1e-5 * np.linalg.norm(blk_o)
    u = u.reshape(-1, u.shape[2])
    assert np.abs(u.conj().T @ u - np.eye(u.shape[1])).max() <= 1e-4


@pytest.mark.parametrize("n,chi", [(100, 128), (80, 130)])
def test_many_gates_and_one_agree_bitwise(T, n, chi):  # noqa: F811
    """46 gates of 256 columns do not fit on the GPU as clusters of 8 and run through the
    queue; one at a time they run as clusters.  32 gates of 260 rows have more visits than
    CTAs, so the prefetching warps claim ahead; with one gate they do not."""
    rng = np.random.default_rng(2)
    d = [min(2 ** min(b, n - b, 30), chi) for b in range(n + 1)]
    sites = [(rng.standard_normal((d[q], 2, d[q + 1])) + 1j * rng.standard_normal((d[q], 2, d[q + 1])))
             / np.sqrt(4 * d[q + 1]) for q in range(n)]
    lay = W.brickwork_su4(n, 1, seed=3).layers[0]
    out = []
    for sched in (T.TNSIM_SCHED_BATCHED, T.TNSIM_SCHED_PLAIN):
        m = T.MPS(n, dtype=T.TNSIM_C64, chi_max=chi, schedule=sched)
        m.import_sites(sites)
        m.apply_layer(lay)
        out.append(m.export_sites())
        m.close()
    # the bulk gates (the small ones at the ends take the layout of the launch's largest)
    for q in range(16, n - 16):
        assert np.array_equal(out[0][q], out[1][q])


@pytest.mark.parametrize("cl,cm,cr", [(150, 40, 20), (256, 16, 8), (140, 34, 17), (256, 2, 1)])
def test_few_long_columns(T, cl, cm, cr):  # noqa: F811
    """One to three blocks of columns of 280 to 512 rows: gates of one block run all their
    sweeps in one visit, odd block counts have visits without a partner."""
    rng = np.random.default_rng(cl + cr)
    d = [min(2 ** b, cl) for b in range(9)] + [cm] + [min(2 ** b, cr) for b in range(9)][::-1]
    d[8], q, n = cl, 8, 18
    sites = [(rng.standard_normal((d[i], 2, d[i + 1])) + 1j * rng.standard_normal((d[i], 2, d[i + 1])))
             / np.sqrt(4 * d[i + 1]) for i in range(n)]
    m = T.MPS(n, dtype=T.TNSIM_C64, chi_max=256, renormalize=False)
    m.import_sites(sites)
    m.apply_layer(W.Layer(np.array([q], np.int32), np.eye(4, dtype=complex)[None], None))
    s, out = m.spectrum(q + 1), m.export_sites()
    m.close()
    blk = sites[q].reshape(2 * cl, cm) @ sites[q + 1].reshape(cm, 2 * cr)
    ref = np.linalg.svd(blk, compute_uv=False)[:len(s)]
    assert len(s) >= min(cm, 2 * cr) and np.max(np.abs(s - ref)) <= 1e-5 * ref[0]
    got = out[q].reshape(2 * cl, -1) @ out[q + 1].reshape(-1, 2 * cr)
    assert np.linalg.norm(got - blk) <= 1e-5 * np.linalg.norm(blk)
