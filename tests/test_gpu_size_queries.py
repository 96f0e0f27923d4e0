"""Size queries on a handle with a bound workspace leave its layout alone (needs a GPU)."""
import numpy as np
import pytest

import oracle
from qxgen import circuits as C

from ._util import assert_parity, grid_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("executor", [0, 2])
def test_calls_between_size_queries_give_the_same_bits(executor):
    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx
    circ, om, order, sliced, bits = grid_case(3, 4, 8, 11, 0, 3, 9)
    recs = C.gates_to_records(circ)
    ref = oracle.sv_amplitudes(circ.n_qubits, recs, om, bits)
    c = qx.Contractor(circ.n_qubits, recs, om, order, sliced, 9, executor=executor)
    want, few = c.contract(bits), c.contract(bits[:4])
    assert_parity(want, ref)
    assert_parity(few, ref[:4])
    for max_bits, items in ((1, 1), (9, 72), (5000, 1), (70000, 4000)):
        qx.qx_workspace_size(c.h, max_bits, items)
        assert np.array_equal(c.contract(bits), want)
        qx.qx_workspace_parts(c.h, max_bits, items)
        assert np.array_equal(c.contract(bits[:4]), few)
    c.close()
