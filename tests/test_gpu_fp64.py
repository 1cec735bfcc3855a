"""complex128 updates through the FP32-preconditioned, refined SVD and the 8 x 8-tiled FP64 products.

Sizes around the edges of the tiles (8, 16), of the column blocks (8, 4), of the smallest
preconditioned block (10 columns) and of the largest (m + n = 1024 rows), rectangular
blocks, every contraction form, and spectra that FP32 cannot resolve.  The kept singular
values must agree with LAPACK's within 64 eps s_max sqrt(rank) (both are backward stable:
a few eps |theta|_2 each, and |theta|_F <= sqrt(rank) s_max), the new block with the best
approximation at the gap of the cut, which random blocks keep above 1e-6.
"""
import numpy as np
import pytest

import workloads as W
from oracle import grad as OG
from oracle import mps as om

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module")
def T():
    import __graft_entry__ as g
    g.build()
    import paper_2601_04422_gb300 as T
    return T


def _chain(cl, cm, cr):
    """Bond dimensions of a chain whose middle pair has bonds cl, cm, cr."""
    def ramp(c):
        d = [1]
        while d[-1] < c:
            d.append(min(c, 2 * d[-1]))
        return d
    a, b = ramp(cl), ramp(cr)
    return a + [cm] + b[::-1], len(a) - 1


def _update(T, cl, cm, cr, chi, cfg, decay=0.0, seed=1, dtype=None):
    rng = np.random.default_rng(seed)
    dims, q = _chain(cl, cm, cr)
    sites = [(rng.standard_normal((dims[i], 2, dims[i + 1])) + 1j * rng.standard_normal((dims[i], 2, dims[i + 1])))
             / np.sqrt(4 * dims[i + 1]) for i in range(len(dims) - 1)]
    sites[q + 1] = sites[q + 1] * np.exp(-decay * np.arange(cm) / max(1, cm - 1))[:, None, None]
    n = len(sites)
    cap = max(chi, max(dims))
    m = T.MPS(n, dtype=T.TNSIM_C128 if dtype is None else dtype, chi_max=cap)
    if any(d > c for d, c in zip(dims, [min(cap, 2 ** min(b, n - b)) for b in range(n + 1)])):
        pytest.skip("chain too short for these bonds")
    m.import_sites(sites)
    if cfg:
        T.tnsim_set_jacobi_config(m.h, cfg)
    g = W.haar_su4(rng)
    m.apply_layer(W.Layer(np.array([q], np.int32), g[None], None))
    ref = om.MPS(sites)
    r = om.apply_2q(ref, q, g, cap)
    s = m.spectrum(q + 1)
    out = m.export_sites()
    m.close()
    blk = out[q].reshape(2 * cl, -1) @ out[q + 1].reshape(-1, 2 * cr)
    blk_o = ref.sites[q].reshape(2 * cl, -1) @ ref.sites[q + 1].reshape(-1, 2 * cr)
    return s, r, blk, blk_o, out[q]


@pytest.mark.parametrize("cfg", [0, 1, 2])
@pytest.mark.parametrize("c", [(3, 4, 4), (4, 5, 5), (7, 8, 7), (8, 8, 8), (8, 9, 9), (9, 16, 12), (16, 17, 17), (33, 33, 20),
                               (20, 33, 33), (64, 64, 65), (100, 60, 90)])
def test_block_sizes(T, c, cfg):
    s, r, blk, blk_o, u = _update(T, *c, chi=1, cfg=cfg)
    assert len(s) == r.k
    assert np.max(np.abs(s - r.s_kept)) <= 64 * EPS * np.sqrt(r.k) * r.s_kept[0]
    assert np.linalg.norm(blk - blk_o) <= 1e-9 * np.linalg.norm(blk_o)
    u = u.reshape(-1, u.shape[2])
    assert np.abs(u.conj().T @ u - np.eye(u.shape[1])).max() <= 1e-11


@pytest.mark.parametrize("chi", [256, 257])
def test_largest_preconditioned_block(T, chi):
    """m + n = 1024 rows is the last preconditioned size, 1028 the first beyond it."""
    s, r, blk, blk_o, _ = _update(T, chi, chi, chi, chi=1, cfg=0)
    assert len(s) == r.k and np.max(np.abs(s - r.s_kept)) <= 64 * EPS * np.sqrt(r.k) * r.s_kept[0]
    assert np.linalg.norm(blk - blk_o) <= 1e-9 * np.linalg.norm(blk_o)


@pytest.mark.parametrize("decay", [12.0, 30.0])
def test_spectrum_below_fp32(T, decay):
    """Singular values over 5 and 13 decades: the small ones are beyond FP32 and are found
    by the FP64 iteration."""
    s, r, blk, blk_o, _ = _update(T, 32, 32, 32, chi=64, cfg=0, decay=decay)
    k = min(len(s), r.k)
    assert np.max(np.abs(s[:k] - r.s_kept[:k])) <= 64 * EPS * np.sqrt(r.k) * r.s_kept[0]
    assert np.linalg.norm(blk - blk_o) <= 1e-12 * np.linalg.norm(blk_o)


@pytest.mark.parametrize("kind", ["equal", "pairs", "rank", "tail"])
def test_close_and_vanishing_singular_values(T, kind):
    """Pairs of singular values too close for a refinement step's angles, at and below its
    limits, null columns, and a tail of 17 decades.  Untruncated: the block itself comes back
    to a few eps |theta|_F of each of the two SVDs, and the left site is an isometry on the
    columns above the tail (normalised columns of singular value s are orthogonal to
    eps s_max / s)."""
    rng = np.random.default_rng(7)
    c, k = 24, 48
    s = np.linspace(1.0, 0.5, k)
    if kind == "equal":
        s[:] = 1.0
    elif kind == "pairs":
        s[1::2] = s[::2] * (1 + 10.0 ** -np.linspace(1, 15, k // 2))
    elif kind == "rank":
        s[k // 3:] = 0.0
    else:
        s = 10.0 ** -np.linspace(0, 17, k)
    u = np.linalg.qr(rng.standard_normal((k, k)) + 1j * rng.standard_normal((k, k)))[0]
    v = np.linalg.qr(rng.standard_normal((k, k)) + 1j * rng.standard_normal((k, k)))[0]
    dims, q = _chain(c, k, c)
    sites = [rng.standard_normal((dims[i], 2, dims[i + 1])) + 0j for i in range(len(dims) - 1)]
    sites[q], sites[q + 1] = u.reshape(c, 2, k), (s[:, None] * v).reshape(k, 2, c)
    m = T.MPS(len(sites), dtype=T.TNSIM_C128, chi_max=64, renormalize=False)
    m.import_sites(sites)
    m.apply_layer(W.Layer(np.array([q], np.int32), np.eye(4, dtype=complex)[None], None))
    got, out = m.spectrum(q + 1), m.export_sites()
    m.close()
    blk = out[q].reshape(k, -1) @ out[q + 1].reshape(-1, k)
    assert np.linalg.norm(blk - (u * s) @ v) <= 64 * EPS * np.linalg.norm(s)
    want = np.sort(s)[::-1][:len(got)]
    assert np.max(np.abs(got - want)) <= 64 * EPS * np.linalg.norm(s)
    iso = out[q].reshape(k, -1)[:, got >= 1e-3]
    assert np.abs(iso.conj().T @ iso - np.eye(iso.shape[1])).max() <= 1e-11


def test_canonical_form_and_memory_cap(T):
    """Canonical-form gates precondition diag(Lam) theta; a state made under a device-memory
    cap has no preconditioner buffers and gives the same state."""
    circ = W.brickwork_u2_su4(12, 8, seed=4)
    out = []
    for cap in (0, 1 << 40):
        T.tnsim_set_device_memory_cap(cap)
        try:
            m = T.MPS(12, dtype=T.TNSIM_C128, chi_max=24, form=T.TNSIM_FORM_CANONICAL)
        finally:
            T.tnsim_set_device_memory_cap(0)
        m.run(circ)
        out.append(om.MPS(m.export_sites()))
        m.close()
    assert 1 - om.fidelity(*out) <= 1e-12


@pytest.mark.parametrize("dt,tol", [("C128", 1e-9), ("C64", 1e-3)])
def test_gradient_recomputes_layers_under_a_cap(T, dt, tol):
    """Without a cap the gradient keeps every layer's decomposition, with one it recomputes
    them; rows of Pauli strings of every length share the environments' launches.  At cutoff
    1e-4 the kept values stay above 1e-2 s_max, so both precisions resolve the gradient
    (complex64 within the bar of the other gradient tests)."""
    n, nl = 9, 5
    circ, ang = W.hea_circuit(n, nl, seed=3)
    layers = [(l.pairs, l.g4) for l in circ.layers]
    axes = ["YZ" if i % 2 == 0 else "" for i in range(len(layers))]
    theta = [ang[i // 2] if i % 2 == 0 else np.zeros((n, 0)) for i in range(len(layers))]
    rng = np.random.default_rng(1)
    paulis = ["I" * n, "Z" * n, "X" + "I" * (n - 1)] + ["".join(rng.choice(list("IIXYZ"), n)) for _ in range(20)]
    coeffs = rng.standard_normal(len(paulis))
    p = T.tnsim_params_default(getattr(T, "TNSIM_" + dt))
    p.chi_max, p.cutoff = 6, 1e-4
    out = []
    for cap in (0, 1 << 40):
        T.tnsim_set_device_memory_cap(cap)
        try:
            e, g = T.tnsim_grad(n, layers, axes, theta, paulis, coeffs, getattr(T, "TNSIM_" + dt), p)
        finally:
            T.tnsim_set_device_memory_cap(0)
        out.append(np.concatenate([[e]] + [x.reshape(-1) for x in g]))
    ref = OG.grad(n, layers, axes, theta, paulis, list(coeffs), 6, 1e-4)
    want = np.concatenate([[ref[0]]] + [x.reshape(-1) for x in ref[1]])
    for o in out:
        assert np.max(np.abs(o - want)) <= tol * np.max(np.abs(want))
