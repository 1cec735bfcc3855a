"""Complex128 circuits of small bonds, against recorded results.

What these calls return is decided by single roundings: an amplitude that is exactly zero
comes back as the residue of the roundings (1e-23 .. 1e-46 here), and a cutoff through two
equal singular values keeps the one that rounding made larger.  Gates of at most 30 rows and
columns therefore keep one order of operations, and the results stay the recorded ones.
1e-9 of the norm separates them from any other order: that gives residues of another size
(or, of the 24-qubit gradient, sums that cancel to 1.15e-9).
"""
import json
import os

import numpy as np
import pytest

import workloads as W
from test_gpu_fp64 import T  # noqa: F401

pytestmark = pytest.mark.gpu
GOLDEN = json.load(open(os.path.join(os.path.dirname(__file__), "golden", "complex128_small.json")))


def _same(got, want):
    assert np.linalg.norm(np.asarray(got) - want) <= 1e-9 * np.linalg.norm(want)


@pytest.mark.parametrize("c", GOLDEN["gateset"], ids=lambda c: f"{c['n']}q_depth{c['depth']}")
def test_vanishing_amplitudes(T, c):  # noqa: F811
    m = T.MPS(c["n"], dtype=T.TNSIM_C128, chi_max=c["chi"])
    m.import_sites([np.array([1, 0], np.complex128).reshape(1, 2, 1)] * c["n"])
    m.run(W.gateset_circuit(c["n"], c["depth"], c["seed"]))
    got = m.amplitudes(W.random_bitstrings(c["n"], c["strings"], c["seed"]))
    m.close()
    _same(got, np.array(c["re"]) + 1j * np.array(c["im"]))


@pytest.mark.parametrize("c", GOLDEN["grad"], ids=lambda c: f"{c['n']}q")
def test_cutoff_through_equal_values(T, c):  # noqa: F811
    n = c["n"]
    circ, ang = W.hea_circuit(n, c["layers"], c["seed"])
    layers = [(l.pairs, l.g4) for l in circ.layers]
    axes = ["YZ" if i % 2 == 0 else "" for i in range(len(layers))]
    theta = [ang[i // 2] if i % 2 == 0 else np.zeros((n, 0)) for i in range(len(layers))]
    zz = ["".join("Z" if k in (i, i + 1) else "I" for k in range(n)) for i in range(n - 1)]
    xs = ["".join("X" if k == i else "I" for k in range(n)) for i in range(n)]
    p = T.tnsim_params_default(T.TNSIM_C128)
    p.chi_max, p.cutoff = c["chi"], c["cutoff"]
    e, g = T.tnsim_grad(n, layers, axes, theta, zz + xs, [1.0] * (n - 1) + [0.5] * n, T.TNSIM_C128, p)
    assert abs(e - c["energy"]) <= 1e-9 * abs(c["energy"])
    _same(np.concatenate([x.reshape(-1) for x in g]), np.array(c["grad"]))
