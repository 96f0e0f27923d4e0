"""The bytes booked for segment launches are those they move: operands from outside the segment and its
result, not the tensors in between (needs a GPU)."""
import re

import pytest

from qxgen import circuits as C

from ._util import grid_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,depth", [(2, 2, 3), (2, 3, 6), (3, 3, 8)])
def test_segments_of_one_amplitude_move_operands_and_results(rows, cols, depth):
    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx
    circ, om, order, sliced, bits = grid_case(rows, cols, depth, 21, 0, 0, 1)
    c = qx.Contractor(circ.n_qubits, C.gates_to_records(circ), om, order, sliced, 1)
    lines = qx.qx_describe_plan(c.h).splitlines()
    root, result, expect = {}, [], 0
    for i, line in enumerate(lines):
        m = re.search(r" (seg|chain)=(\d+)", line)
        assert m  # every step belongs to a segment
        root[m.groups()] = i
        r = re.search(r" rank=(\d+)", line)
        if r:
            operands, size = 1 << int(r[1]), 1 << int(r[1])
        else:
            mb, kb, nb = (int(x) for x in re.search(r" m=(\d+) k=(\d+) n=(\d+)", line).groups())
            operands, size = (1 << (mb + kb)) + (1 << (kb + nb)), 1 << (mb + nb)
        result.append(size)
        expect += operands
    # a step's result is read once: inside its segment, from shared memory, unless it is the segment's own
    for i, size in enumerate(result):
        expect += size if i in root.values() else -size
    qx.qx_set_profiling(c.h, True)
    c.contract(bits)
    prof = qx.qx_profile_read(c.h)
    assert prof["wave"]["launches"] == c.stats()["launches"] - 2  # and the slice sum and its end
    assert prof["wave"]["bytes"] == 8 * expect
    c.close()
