"""The same steps as one segment launch for a few items and as a launch each for many (needs a GPU): the
launch counts show that the two ways were taken, and the amplitudes agree bit for bit."""
import numpy as np
import pytest

from qxgen import circuits as C

from ._util import grid_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,depth,n_open,n_slice", [(3, 4, 8, 0, 0), (3, 4, 8, 2, 3), (4, 4, 10, 1, 2)])
def test_few_and_many_items_take_different_paths(rows, cols, depth, n_open, n_slice):
    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import cost, qx
    circ, om, order, sliced, bits = grid_case(rows, cols, depth, 300 + depth, n_open, n_slice, 4000)
    c = qx.Contractor(circ.n_qubits, C.gates_to_records(circ), om, order, sliced, len(bits))
    desc = qx.qx_describe_plan(c.h)
    count, got = {}, {}
    for k in (1, len(bits)):
        qx.qx_set_profiling(c.h, True)
        got[k] = c.contract(bits[:k])
        count[k] = c.stats()["launches"], qx.qx_profile_read(c.h)["wave"]["launches"], c.stats()["batches"]
    c.close()
    assert np.array_equal(got[1], got[len(bits)][:1])
    # one batch each, as the rule has it: what differs is segment launches against launches per step
    for k, (launches, waves, batches) in count.items():
        assert batches == 1
        listed = cost.launches(desc, (1, 1 << n_slice, k << n_slice))
        assert launches == len(listed) + 2  # the slice sum and its end
    assert count[1][1] > count[len(bits)][1] >= 1  # fewer segments pay; the prologue always does
    assert count[1][0] < count[len(bits)][0]
