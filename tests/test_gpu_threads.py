"""Host threads with a state each, and equal and unequal sizes: launches of one kernel with
different amounts of shared memory must not refuse one another, and each thread's results
are those of the same calls alone, bit for bit.
"""
import threading

import numpy as np
import pytest

import workloads as W
from test_gpu_fp64 import T  # noqa: F401

pytestmark = pytest.mark.gpu


def _work(T, n, chi, dtype, reps, strings):  # noqa: F811
    rng = np.random.default_rng(n * chi)
    d = [min(2 ** min(b, n - b, 30), chi) for b in range(n + 1)]
    sites = [((rng.standard_normal((d[q], 2, d[q + 1])) + 1j * rng.standard_normal((d[q], 2, d[q + 1])))
              / np.sqrt(4 * d[q + 1])).astype(np.complex64).astype(np.complex128) for q in range(n)]
    layers = W.brickwork_su4(n, 2, seed=chi).layers
    bits = W.random_bitstrings(n, strings, seed=1)
    m = T.MPS(n, dtype=getattr(T, dtype), chi_max=chi)
    out = []
    for _ in range(reps):
        m.import_sites(sites)
        for lay in layers:
            m.apply_layer(lay)
        out.append((m.bond_dims(), m.spectrum(n // 2)))
        m.import_sites(sites)
        out[-1] += (m.amplitudes(bits),)
    m.close()
    return out


# (qubits, bond dimension, type, repetitions, strings): clusters of FP32 columns of one size
# and of two, FP64 columns of two, groups of bitstrings at two bond dimensions
JOBS = [[(12, 32, "TNSIM_C64", 150, 1), (12, 32, "TNSIM_C64", 150, 1)],
        [(14, 24, "TNSIM_C64", 100, 1), (14, 30, "TNSIM_C64", 100, 1), (10, 20, "TNSIM_C64", 100, 1)],
        [(12, 24, "TNSIM_C128", 40, 1), (14, 48, "TNSIM_C128", 40, 1)],
        [(14, 50, "TNSIM_C64", 40, 64), (16, 100, "TNSIM_C64", 40, 64), (14, 64, "TNSIM_C64", 40, 64)]]


@pytest.mark.parametrize("jobs", JOBS, ids=["equal", "complex64", "complex128", "amplitudes"])
def test_threads_do_not_disturb_each_other(T, jobs):  # noqa: F811
    want = [_work(T, n, chi, dt, 1, s)[0] for n, chi, dt, _, s in jobs]
    got, errors = [None] * len(jobs), []

    def run(i):
        try:
            got[i] = _work(T, *jobs[i])
        except Exception as e:   # noqa: BLE001 -- reported below
            errors.append(f"thread {i}: {e}")

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for g, w in zip(got, want):
        for r in g:
            assert all(np.array_equal(a, b) for a, b in zip(r, w))
