"""The complex128 preconditioner's buffers: optional, and not what a memory cap counts."""
import pytest

import workloads as W
from oracle import mps as om
from test_gpu_fp64 import T  # noqa: F401

pytestmark = pytest.mark.gpu


def _state(T, cap):  # noqa: F811
    T.tnsim_set_device_memory_cap(cap)
    try:
        return T.MPS(12, dtype=T.TNSIM_C128, chi_max=40)
    finally:
        T.tnsim_set_device_memory_cap(0)


def test_a_cap_set_later_admits_what_it_did(T):  # noqa: F811
    """Two equal states fit under twice the bytes of one, whether the first was made under the
    cap or before it."""
    held = T.tnsim_device_bytes_held()
    one = _state(T, 1 << 40)
    need = T.tnsim_device_bytes_held() - held
    one.close()
    a = _state(T, 0)
    assert T.tnsim_device_bytes_held() == held + need
    b = _state(T, held + 2 * need)
    with pytest.raises(T.TnsimError):
        _state(T, held + 2 * need)
    a.close()
    b.close()
    assert T.tnsim_device_bytes_held() == held


def test_batch_of_states_with_and_without_buffers(T):  # noqa: F811
    """Both kinds in one launch: each state as by itself (backward-stable SVDs of the same
    blocks: states equal to 1e-12)."""
    circs = [W.brickwork_u2_su4(12, 7, seed=s) for s in (1, 2)]
    ms = [_state(T, 0), _state(T, 1 << 40)]
    steps = [[(c.layers[t].pairs, c.layers[t].g4, c.layers[t].u1) for c in circs] for t in range(len(circs[0].layers))]
    T.tnsim_apply_layers_batched([m.h for m in ms], steps)
    for m, c in zip(ms, circs):
        ref = _state(T, 0)
        ref.run(c)
        assert 1 - om.fidelity(om.MPS(m.export_sites()), om.MPS(ref.export_sites())) <= 1e-12
        ref.close()
        m.close()
