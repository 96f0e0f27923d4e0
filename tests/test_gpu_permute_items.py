"""Permutes of tensors smaller than a tile take several items per tile (needs a GPU).

How many depends on the powers of two in the item count (bitstrings x slices), so requests of
different sizes go through different tiles.
"""
import numpy as np
import pytest

import oracle
from qxgen import circuits as C

from ._util import assert_parity, grid_case

pytestmark = pytest.mark.gpu


def _plan(case, ranks, n_bits):
    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx
    rows, cols, depth, n_open, n_slice = case
    circ, om, order, sliced, bits = grid_case(rows, cols, depth, 1, n_open, n_slice, n_bits)
    recs = C.gates_to_records(circ)
    c = qx.Contractor(circ.n_qubits, recs, om, order, sliced, n_bits)
    steps = [line.split() for line in qx.qx_describe_plan(c.h).splitlines()]
    assert ranks <= {f[4] for f in steps if f[2] == "permute" and f[3] != "shared"}
    return circ.n_qubits, recs, om, bits, c


@pytest.mark.parametrize("s0,s1", [(0, 7), (3, 4), (0, 16), (5, 11)])
def test_merged_items_move_the_same_entries(s0, s1):
    """A permute moves entries only, and this plan's sums run in one order at every request size: the
    amplitudes agree bit for bit."""
    import torch
    *_, bits, c = _plan((3, 5, 16, 1, 6), {"rank=9", "rank=11"}, 512)
    bits = torch.from_numpy(bits).cuda()
    got = {}
    for k in (512, 1, 3, 6):
        out = torch.empty((k, 2, 2), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        c.contract_device(bits[:k].contiguous(), out, s0, s1)
        torch.cuda.synchronize()
        got[k] = out.cpu().numpy()
    c.close()
    for k in (1, 3, 6):
        assert np.array_equal(got[k], got[512][:k]), k


@pytest.mark.parametrize("n_bits", [1, 3, 6, 512])
def test_tensors_of_128_entries_match_the_oracle(n_bits):
    n, recs, om, bits, c = _plan((3, 4, 16, 0, 4), {"rank=7", "rank=11"}, n_bits)
    got = c.contract(bits)
    c.close()
    assert_parity(got, oracle.sv_amplitudes(n, recs, om, bits))
