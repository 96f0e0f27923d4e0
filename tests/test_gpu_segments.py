"""Small steps run as segments: one launch, intermediates in shared memory (needs a GPU).

A segment runs only where its item count makes it the faster way, so the same bitstring contracted
alone and among thousands takes different kernels for the same steps: the amplitudes must agree bit
for bit, since every output is the same ordered sum.
"""
import numpy as np
import pytest

import oracle
from qxgen import circuits as C

from ._util import assert_parity, grid_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qx():
    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx as mod
    return mod


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("rows,cols,depth,n_open,n_slice", [
    (2, 2, 3, 0, 0), (2, 3, 9, 0, 1), (3, 4, 8, 0, 0), (3, 4, 8, 2, 3), (4, 4, 12, 0, 0), (4, 4, 10, 1, 4)])
def test_segments_give_the_bits_of_single_launches(qx, rows, cols, depth, n_open, n_slice, precision):
    circ, om, order, sliced, bits = grid_case(rows, cols, depth, 300 + depth, n_open, n_slice, 2500)
    n, recs = circ.n_qubits, C.gates_to_records(circ)
    c = qx.Contractor(n, recs, om, order, sliced, len(bits), precision=precision)
    many = c.contract(bits)
    launches_many = c.stats()["launches"]
    few = {k: c.contract(bits[:k]) for k in (1, 3, 70)}
    assert "chain=" in qx.qx_describe_plan(c.h)
    c.close()
    for k, got in few.items():
        assert np.array_equal(got, many[:k]), k
    assert launches_many >= 1
    assert_parity(many[:70], oracle.sv_amplitudes(n, recs, om, bits[:70]))


@pytest.mark.parametrize("no_slice_level", [0, 1])
def test_a_workspace_too_small_for_segments_still_contracts(qx, no_slice_level):
    """The layout without segments takes over where only it fits, with the same bits."""
    circ, om, order, sliced, bits = grid_case(4, 4, 12, 41, 0, 2, 1)
    n, recs = circ.n_qubits, C.gates_to_records(circ)
    c = qx.Contractor(n, recs, om, order, sliced, 1, no_slice_level=no_slice_level)
    want = c.contract(bits)
    need = qx.qx_workspace_size(c.h, 1, 1)
    c.close()
    fitted = []
    for cut in (256, 1024, 4096, 16384, need // 8):
        try:
            s = qx.Contractor(n, recs, om, order, sliced, 1, no_slice_level=no_slice_level, workspace_bytes=need - cut)
        except qx.QXError as e:
            assert e.code == qx.QX_ENOMEM
            continue
        fitted.append("seg=" in qx.qx_describe_plan(s.h) or "chain=" in qx.qx_describe_plan(s.h))
        assert np.array_equal(s.contract(bits), want)
        s.close()
    assert fitted and not fitted[0]  # the smaller layout fits a little below the segments' need


def test_a_long_run_of_large_steps_is_cut_into_segments_that_fit(qx):
    """A chain of dozens of steps on 2^12-entry tensors: each has 128 pieces of work, so a segment of all
    of them would not fit in shared memory."""
    n = 12
    circ = C.Circuit(n)
    rng = C.SplitMix64(9)
    for t in range(6):
        for q in range(n):
            circ.append((q,), C.ONE_QUBIT_SET[rng.randint(3)])
        for q in range(t % 2, n - 1, 2):
            circ.append((q, q + 1), C.FSIM_SYC)
    om = np.ones(n, np.uint8)
    om[0] = 0
    recs = C.gates_to_records(circ)
    # state-vector order: the inputs joined first, then every gate onto the state
    order, cur = [], 0
    total = n + len(circ.gates) + 1
    for t in list(range(1, n + len(circ.gates) + 1)):
        order.append((cur, t))
        cur = total + len(order) - 1
    c = qx.Contractor(n, recs, om, order, [], 2)
    bits = np.zeros((2, n), np.uint8)
    bits[1, 0] = 1
    got = c.contract(bits)
    c.close()
    assert_parity(got, oracle.sv_amplitudes(n, recs, om, bits))
