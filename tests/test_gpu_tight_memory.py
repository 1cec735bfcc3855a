"""Expectations and gradients of many terms with little device memory left.

The scratch of a batch of terms shrinks to what there is: the results are those with ample
memory, bit for bit (the same sums in the same order).
"""
import numpy as np
import pytest

import workloads as W
from test_gpu_fp64 import T  # noqa: F401

pytestmark = pytest.mark.gpu


def _with_free(mb, call):
    """call() with about mb MB of the device's memory free."""
    torch = pytest.importorskip("torch")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    blocks, left = [], free - (mb << 20)
    while left > (64 << 20):
        size = min(left, 16 << 30)
        blocks.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
        left = torch.cuda.mem_get_info()[0] - (mb << 20)
    try:
        return call()
    finally:
        del blocks
        torch.cuda.empty_cache()


def test_expectations(T):  # noqa: F811
    n, chi = 20, 64
    rng = np.random.default_rng(3)
    d = [min(2 ** min(b, n - b), chi) for b in range(n + 1)]
    m = T.MPS(n, dtype=T.TNSIM_C64, chi_max=chi)
    m.import_sites([(rng.standard_normal((d[q], 2, d[q + 1])) + 1j * rng.standard_normal((d[q], 2, d[q + 1])))
                    / np.sqrt(4 * d[q + 1]) for q in range(n)])
    paulis = ["".join("Z" if k in (i % (n - 1), i % (n - 1) + 1) else "I" for k in range(n)) for i in range(3000)]
    want = m.expect_pauli(paulis)
    got = _with_free(96, lambda: m.expect_pauli(paulis))
    m.close()
    assert np.array_equal(got, want)


def test_gradient(T):  # noqa: F811
    n, nl = 16, 2
    circ, ang = W.hea_circuit(n, nl, seed=3)
    layers = [(l.pairs, l.g4) for l in circ.layers]
    axes = ["YZ" if i % 2 == 0 else "" for i in range(len(layers))]
    theta = [ang[i // 2] if i % 2 == 0 else np.zeros((n, 0)) for i in range(len(layers))]
    paulis = ["".join("Z" if k in (i % (n - 1), i % (n - 1) + 1) else "I" for k in range(n)) for i in range(1000)]
    p = T.tnsim_params_default(T.TNSIM_C128)
    p.chi_max = 64

    def call():
        e, g = T.tnsim_grad(n, layers, axes, theta, paulis, [1.0] * len(paulis), T.TNSIM_C128, p)
        return np.concatenate([[e]] + [x.reshape(-1) for x in g])

    want = call()
    # the full environments of 1000 terms are 131 MB, the scratch of all at once 393 MB more
    got = _with_free(352, call)
    assert np.array_equal(got, want)
