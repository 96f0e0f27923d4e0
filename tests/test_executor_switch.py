"""The executor of a handle may be changed after its plan was set: what the workspace is sized and laid
out for must hold for the executor that runs (host logic, no GPU)."""
import numpy as np
import pytest

from qxgen import circuits as C
from qxgen import workloads as W

from ._util import grid_case


def _handle(qx, circ, om, order, sliced, executor):
    h = qx.qx_create(-1, executor=executor)
    qx.qx_build_network(h, circ.n_qubits, C.gates_to_records(circ), om)
    qx.qx_set_plan(h, order, sliced)
    return h


@pytest.mark.parametrize("rows,cols,depth,n_slice", [(2, 3, 9, 1), (3, 4, 8, 3), (4, 4, 12, 2), (4, 5, 12, 6)])
@pytest.mark.parametrize("n_bits", [1, 17])
def test_a_members_workspace_holds_a_pair_of_the_batched_executor(rows, cols, depth, n_slice, n_bits):
    """qx_set_options may turn a bound group member into a handle that contracts by itself, one pair at a
    time: the size it was given covers the per-slice and per-pair regions of that pair."""
    from paper_2110_09894_gb300 import qx
    circ, om, order, sliced, _ = grid_case(rows, cols, depth, 7, 0, n_slice, 1)
    h = _handle(qx, circ, om, order, sliced, 3)
    size = qx.qx_workspace_size(h, n_bits, 1)
    fixed, batch = qx.qx_workspace_parts(h, n_bits, 1)
    qx.qx_destroy(h)
    assert size >= fixed + batch


def test_the_persistent_executor_can_be_chosen_after_the_plan():
    """A plan whose steps the persistent kernel runs too: its workspace then has the kernel's regions."""
    from paper_2110_09894_gb300 import qx
    circ, om, order, sliced, _ = grid_case(2, 3, 4, 7, 0, 0, 1)
    h = _handle(qx, circ, om, order, sliced, 0)
    batched = qx.qx_workspace_size(h, 3, 1)
    qx.qx_set_options(h, executor=2)
    persistent = qx.qx_workspace_size(h, 3, 1)
    qx.qx_set_options(h, executor=1)
    assert qx.qx_workspace_size(h, 3, 1) == batched
    qx.qx_destroy(h)
    assert persistent >= batched + 8 * 2 * 152  # at least one entry for each of two CTAs per SM


def test_a_plan_set_for_one_executor_keeps_its_storages_under_another():
    """Sizes that a plan's storage rules decide do not depend on the executor chosen later."""
    from paper_2110_09894_gb300 import qx
    w = W.batched_circuit(121)
    for first in (0, 3):
        h = qx.qx_create(-1, executor=first)
        qx.qx_build_network(h, w.n_qubits, w.gates, w.open_mask)
        qx.qx_set_plan(h, w.order, w.sliced)
        want = qx.qx_workspace_parts(h, 4, 9)[1], qx.qx_describe_plan(h)
        for other in (2, 1, 3, 0):
            qx.qx_set_options(h, executor=other)
            assert (qx.qx_workspace_parts(h, 4, 9)[1], qx.qx_describe_plan(h)) == want
        qx.qx_destroy(h)
