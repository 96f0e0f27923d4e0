"""The executor of a handle changed after its workspace was bound (needs a GPU): the call runs where
the bound regions hold it and is refused where they don't."""
import pytest

import oracle
from qxgen import circuits as C
from qxgen import workloads as W

from ._util import assert_parity, grid_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qx():
    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx as mod
    return mod


def _refused(qx, c, bits, code):
    with pytest.raises(qx.QXError) as e:
        c.contract(bits)
    assert e.value.code == code


def test_a_bound_member_contracts_by_itself_after_a_change_of_options(qx):
    w = W.batched_circuit(121)
    bits = w.bitstrings[:5]
    ref = oracle.sv_amplitudes(w.n_qubits, w.gates, w.open_mask, bits)
    c = qx.Contractor(w.n_qubits, w.gates, w.open_mask, w.order, w.sliced, 5, executor=qx.EXEC_GROUP_MEMBER)
    _refused(qx, c, bits, qx.QX_EINVAL)  # a member contracts through its group
    qx.qx_set_options(c.h)
    for _ in range(3):
        assert_parity(c.contract(bits), ref)
    qx.qx_set_options(c.h, executor=qx.EXEC_PERSISTENT)  # no CTA scratch in a member's workspace
    _refused(qx, c, bits, qx.QX_ESTATE)
    qx.qx_set_options(c.h, executor=qx.EXEC_GROUP_MEMBER)
    size = qx.qx_workspace_size(c.h, 5, 1)
    fixed, batch = qx.qx_workspace_parts(c.h, 5, 1)
    c.close()
    assert size >= fixed + batch
    # a workspace for the group's runs alone: a pair of the batched executor doesn't fit
    c = qx.Contractor(w.n_qubits, w.gates, w.open_mask, w.order, w.sliced, 5, executor=qx.EXEC_GROUP_MEMBER,
                      workspace_bytes=fixed + batch - 256)
    qx.qx_set_options(c.h)
    _refused(qx, c, bits, qx.QX_ENOMEM)
    c.close()


def test_the_persistent_executor_needs_a_workspace_bound_for_it(qx):
    circ, om, order, sliced, bits = grid_case(2, 3, 4, 7, 0, 0, 3)
    recs = C.gates_to_records(circ)
    ref = oracle.sv_amplitudes(circ.n_qubits, recs, om, bits)
    c = qx.Contractor(circ.n_qubits, recs, om, order, sliced, 3)
    assert_parity(c.contract(bits), ref)
    qx.qx_set_options(c.h, executor=qx.EXEC_PERSISTENT)
    _refused(qx, c, bits, qx.QX_ESTATE)
    need = qx.qx_workspace_size(c.h, 3, 1)
    ws = c.torch.empty(need, dtype=c.torch.uint8, device="cuda")
    qx.qx_bind_workspace(c.h, ws.data_ptr(), need, 3)
    assert_parity(c.contract(bits), ref)
    qx.qx_set_options(c.h)  # and back: the batched regions are part of it
    assert_parity(c.contract(bits), ref)
    c.close()


def test_a_split_workspace_stays_refused_for_the_persistent_executors(qx):
    import torch
    circ, om, order, sliced, _ = grid_case(2, 3, 4, 7, 0, 0, 3)
    for first, then in ((0, 2), (0, 3), (2, 2), (3, 3)):
        h = qx.qx_create(0, executor=first)
        qx.qx_build_network(h, circ.n_qubits, C.gates_to_records(circ), om)
        qx.qx_set_plan(h, order, sliced)
        qx.qx_set_options(h, executor=then)
        fixed = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
        batch = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
        with pytest.raises(qx.QXError) as e:
            qx.qx_bind_workspace_parts(h, fixed.data_ptr(), 1 << 20, batch.data_ptr(), 1 << 20, 3)
        assert e.value.code == qx.QX_EINVAL
        qx.qx_destroy(h)
