"""More Pauli terms than one launch can hold in a grid dimension (65535 steps).

A state of small bonds has room for every term at once: the 65536 Pauli strings of eight
qubits in one call, and gradients of sums of more than 32767 terms (two steps a term).
"""
import itertools

import numpy as np
import pytest

import workloads as W
from test_gpu_fp64 import T  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt,tol", [("C64", 1e-5), ("C128", 1e-12)])
def test_all_strings_of_eight_qubits(T, dt, tol):  # noqa: F811
    """A product state: every expectation is a product of one-qubit ones."""
    n = 8
    rng = np.random.default_rng(4)
    v = rng.standard_normal((n, 2)) + 1j * rng.standard_normal((n, 2))
    v /= np.linalg.norm(v, axis=1)[:, None]
    ops = {"I": np.eye(2), "X": np.array([[0, 1], [1, 0]]), "Y": np.array([[0, -1j], [1j, 0]]), "Z": np.diag([1, -1])}
    one = np.array([[(w.conj() @ ops[c] @ w).real for c in "IXYZ"] for w in v])
    paulis = ["".join(p) for p in itertools.product("IXYZ", repeat=n)] + ["I" * n, "Z" * n]
    want = np.ones(1)
    for q in range(n):
        want = np.outer(want, one[q]).reshape(-1)
    want = np.concatenate([want, want[[0, -1]]])
    m = T.MPS(n, dtype=getattr(T, "TNSIM_" + dt), chi_max=4)
    m.import_sites([w.reshape(1, 2, 1) for w in v])
    got = m.expect_pauli(paulis)
    m.close()
    assert np.max(np.abs(got - want)) <= tol


def test_gradient_of_many_terms(T):  # noqa: F811
    """40000 terms on few strings: the gradient of the same strings with summed coefficients
    (sums of 40000 terms in another order: 40000 eps of their magnitudes)."""
    n, nl = 5, 2
    circ, ang = W.hea_circuit(n, nl, seed=3)
    layers = [(l.pairs, l.g4) for l in circ.layers]
    axes = ["YZ" if i % 2 == 0 else "" for i in range(len(layers))]
    theta = [ang[i // 2] if i % 2 == 0 else np.zeros((n, 0)) for i in range(len(layers))]
    strings = ["ZIIII", "IXIII", "IIZZI", "IIIIY", "IIIXI"]
    rng = np.random.default_rng(2)
    pick, c = rng.integers(0, len(strings), 40000), rng.standard_normal(40000)
    p = T.tnsim_params_default(T.TNSIM_C128)
    p.chi_max = 4
    args = (n, layers, axes, theta)
    e, g = T.tnsim_grad(*args, [strings[i] for i in pick], list(c), T.TNSIM_C128, p)
    e1, g1 = T.tnsim_grad(*args, strings, [float(c[pick == i].sum()) for i in range(len(strings))], T.TNSIM_C128, p)
    tol = 40000 * np.finfo(float).eps * np.abs(c).sum()
    assert abs(e - e1) <= tol
    assert np.max(np.abs(np.concatenate([x.reshape(-1) for x in g]) - np.concatenate([x.reshape(-1) for x in g1]))) <= tol


def test_memory_of_many_long_terms(T):  # noqa: F811
    """60000 terms over 100 sites: the steps of all of them at once would be 336 MB.  A batch's
    are 64 MB, its environments here less than 8 MB, and its sums less than 24; and each term
    gets its value (a product state again)."""
    torch = pytest.importorskip("torch")
    import threading
    import time

    n, count = 100, 60000
    rng = np.random.default_rng(6)
    m = T.MPS(n, dtype=T.TNSIM_C64, chi_max=2)
    plus = np.array([1, 1]).reshape(1, 2, 1) / np.sqrt(2)
    zero = np.array([1, 0]).reshape(1, 2, 1)
    m.import_sites([plus if q % 2 else zero for q in range(n)])
    # X on |+>, Z on |0>: every value is 1 but those of a term with a Y or a Z on |+> (0)
    kinds = ["".join("X" if q % 2 else "Z" for q in range(n)), "Z" + "I" * (n - 2) + "X", "Y" + "I" * (n - 2) + "X"]
    paulis = [kinds[i] for i in rng.integers(0, 3, count)]
    want = np.array([0.0 if p[0] == "Y" else 1.0 for p in paulis])
    m.expect_pauli(paulis[:8])
    free = [torch.cuda.mem_get_info()[0]]
    stop = threading.Event()

    def watch():
        while not stop.is_set():
            free.append(torch.cuda.mem_get_info()[0])
            time.sleep(2e-4)

    t = threading.Thread(target=watch)
    t.start()
    try:
        got = m.expect_pauli(paulis)
    finally:
        stop.set()
        t.join()
    m.close()
    assert np.max(np.abs(got - want)) <= 1e-5
    assert free[0] - min(free) <= (64 + 8 + 24 + 32) << 20   # and 32 MB of slack for the allocator
