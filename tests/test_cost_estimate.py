"""The launch-list estimate against measured calls (host logic, no GPU): microseconds of one call on one
stream on a GB300, as a serving lane makes it.  Steps that run as one launch are priced once."""
import re

import numpy as np
import pytest

from paper_2110_09894_gb300 import cost
from qxgen import circuits as C
from qxgen import workloads as W


def _listing(n, gates, open_mask, order, sliced, precision):
    from paper_2110_09894_gb300 import qx
    h = qx.qx_create(-1, precision=precision)
    qx.qx_build_network(h, n, gates, open_mask)
    qx.qx_set_plan(h, np.asarray(order, np.int64), np.asarray(sliced, np.int64))
    desc = qx.qx_describe_plan(h)
    qx.qx_destroy(h)
    return desc


def _grid(rows, cols, depth, precision=0):
    circ = C.random_grid_circuit(rows, cols, depth, 0)
    om = np.zeros(circ.n_qubits, np.uint8)
    order, sliced, _, _ = W.make_plan(circ, om, 0, 1)
    return _listing(circ.n_qubits, C.gates_to_records(circ), om, order, sliced, precision), 1


def _sliced(precision):
    w = W.sliced_checkpoint()
    return _listing(w.n_qubits, w.gates, w.open_mask, w.order, w.sliced, precision), 1 << len(w.sliced)


def _served(j, precision):
    w = W.serving_circuit(j)
    return _listing(w.n_qubits, w.gates, w.open_mask, w.order, w.sliced, precision), 1 << len(w.sliced)


@pytest.mark.parametrize("plan,n_bits,measured_us", [
    (lambda: _grid(3, 4, 8), 17, 32.7), (lambda: _grid(4, 4, 12), 1, 123.3),
    (lambda: _sliced(1), 256, 516.7), (lambda: _sliced(1), 1, 170.8), (lambda: _sliced(1), 1024, 1404.9),
    (lambda: _served(7, 1), 300, 865.8), (lambda: _served(7, 1), 1, 298.0), (lambda: _served(8, 0), 1, 285.1)])
def test_estimates_lie_near_the_measured_times(plan, n_bits, measured_us):
    desc, n_slices = plan()
    est = 1e6 * cost.launch_list_time(desc, n_slices, n_bits)
    assert measured_us / 1.5 < est < 1.5 * measured_us


@pytest.mark.parametrize("j,precision,n_bits,items,measured_ms", [
    (9, 1, 1, 1024, 0.20), (9, 1, 300, 1024, 6.52), (3, 0, 40, 185, 1.84), (6, 0, 40, 101, 6.85),
    (7, 1, 300, 658, 0.89), (6, 1, 102, 102, 3.83)])
def test_a_lanes_piece_is_priced_in_its_batches_with_kept_invariants(j, precision, n_bits, items, measured_ms):
    """Requests on an idle server after the lane's first one (host time among it)."""
    desc, n_slices = _served(j, precision)
    est = 1e3 * cost.launch_list_time(desc, n_slices, n_bits, max_items=items, kept=True)
    assert measured_ms / 1.5 < est < 1.5 * measured_ms
    assert cost.launch_list_time(desc, n_slices, n_bits, max_items=items) > est / 1e3


def test_batches_of_a_sliced_call_repeat_its_per_batch_launches():
    desc, n_slices = _sliced(1)
    whole = cost.launch_list_time(desc, n_slices, 16)
    assert cost.launch_list_time(desc, n_slices, 16, max_items=16 * n_slices) == whole
    half = cost.launch_list_time(desc, n_slices, 16, max_items=16 * n_slices // 2)
    assert whole < half < 2 * whole


def test_a_segment_is_one_launch_where_it_runs_as_one():
    desc, n_slices = _sliced(1)
    seg = {m[1] for m in re.finditer(r" seg=(\d+)", desc)}
    alone = [line for line in desc.splitlines() if " seg=" not in line and " chain=" not in line]
    few, many = (cost.launches(desc, (1, n_slices, n_slices * b)) for b in (1, 256))
    assert len(few) == 1 + len(seg) + len(alone)  # and one prologue launch
    assert len(few) < len(many) < len(desc.splitlines())
    assert sum(level == 0 for level, _ in many) == 1
