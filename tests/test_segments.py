"""Segments of the compiled plan (host logic, no GPU): running a segment at its last step, without
writing its inner results, must leave every other launch the data that running step by step gives."""
import re

import numpy as np
import pytest

from qxgen import workloads as W
from tests.test_plan_deps import _check, _overlap, _parse, _plan_lines


def _segments(lines):
    segs = {}
    for i, line in enumerate(lines):
        m = re.search(r" (seg|chain)=(\d+)", line)
        if m:
            segs.setdefault((m.group(1), int(m.group(2))), []).append(i)
    return segs


def _check_segments(lines):
    ops, segs = _parse(lines), _segments(lines)
    _check(ops)
    level = [line.split()[3] for line in lines]
    for (kind, _), members in segs.items():
        root = members[-1]
        assert len({level[i] for i in members}) == 1
        made = {i: ops[i]["w"] for i in members}
        for i in members:
            # what the segment reads from outside stays as it was when its producer left it, up to the
            # segment's launch (at the root's place; a chain's at the start: it reads no storage)
            outer = [r for r in ops[i]["r"] if not any(j < i and _overlap([r], made[j]) and not any(
                _overlap([r], ops[k]["w"]) for k in range(j + 1, i) if k not in members) for j in members)]
            if kind == "chain":
                assert not outer
            for j in range(i + 1, root):
                if j not in members:
                    assert not _overlap(outer, ops[j]["w"]), f"step {j} overwrites an operand of segment step {i}"
            if i != root:  # inner results are never read from memory by anyone else
                for j in range(i + 1, len(ops)):
                    if _overlap(made[i], ops[j]["r"]) and j not in members:
                        assert any(_overlap(made[i], ops[k]["w"]) for k in range(i + 1, j)), (i, j)
    return len(segs)


@pytest.mark.parametrize("precision", [0, 1, 3])
@pytest.mark.parametrize("name", ["sliced", "sliced_checkpoint", "large_annealed", "large_local_search"])
def test_segments_leave_the_other_launches_their_data(name, precision):
    from paper_2110_09894_gb300 import qx
    w = getattr(W, name)()
    lines = _plan_lines(qx, w.n_qubits, w.gates, w.open_mask, w.order, w.sliced, precision)
    assert _check_segments(lines) > 10


def test_chain_results_are_not_overwritten_before_use():
    """Chains run at the start: nothing that starts later may use their results' space before their
    consumers have read them."""
    from paper_2110_09894_gb300 import qx
    w = W.large_annealed()
    lines = _plan_lines(qx, w.n_qubits, w.gates, w.open_mask, w.order, w.sliced, 1)
    ops = _parse(lines)
    for (kind, _), members in _segments(lines).items():
        if kind != "chain":
            continue
        root = members[-1]
        for j in range(root):
            if j in members or re.search(r" chain=", lines[j]):
                continue
            assert not _overlap(ops[root]["w"], ops[j]["w"]), (root, j)
