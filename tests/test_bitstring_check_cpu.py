"""Host-side bitstring checks, and the argument errors of the device check, without a GPU."""
import ctypes

import pytest
import torch

import circuitgen as cg
import paper_1805_01450_gb300 as q


@pytest.mark.parametrize("rows,cols", [(3, 3), (8, 8), (8, 9)])   # 9, 64 and 72 qubits
def test_host_bitstrings(rows, cols):
    n = rows * cols
    p = q.Plan(cg.grid_circuit(rows, cols, 2, 1))
    top = (1 << n) - 1
    good = [0, 1, top]
    bad = [1 << n] if n % 64 else []
    p._check_host_bits(good)
    p._check_host_bits(torch.tensor(q.bitstring_words(good, p.words)))
    for b in bad + ([1 << (64 * p.words - 1)] if n % 64 else []):
        with pytest.raises(q.QvxError):
            p._check_host_bits([0, b])
        with pytest.raises(q.QvxError):
            p._check_host_bits(torch.tensor(q.bitstring_words([0, b], p.words)))
    # bits above the words a bitstring has are cut off, as in the upload
    p._check_host_bits([1 << (64 * p.words)])
    if n % 64:   # the sign bit of a word
        with pytest.raises(q.QvxError):
            p._check_host_bits([-1])


def test_ticket_errors():
    L = q.lib()
    t = ctypes.c_int64(5)
    p = q.Plan(cg.grid_circuit(3, 3, 2, 1))
    assert L.qvx_bits_check(None, None, 0, None, ctypes.byref(t)) == q.QVX_EINVAL
    assert L.qvx_bits_check(p._h, None, 1, None, ctypes.byref(t)) == q.QVX_EINVAL
    assert L.qvx_bits_check(p._h, None, 0, None, ctypes.byref(t)) == q.QVX_OK and t.value == -1
    assert L.qvx_bits_result(-1) == q.QVX_OK and L.qvx_bits_result(1 << 40) == q.QVX_EINVAL
