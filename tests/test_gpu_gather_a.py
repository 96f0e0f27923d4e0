"""Direct 3xTF32 steps that read A where it is stored (needs a GPU).

The producer warp brings a stage's 128 x 16 tile of A as 2^(11 - run) contiguous blocks, one per lane,
on the resident-B' kernel (listed a_gather=1 for long blocks) and on the general one (a_gather=2).
The plans cover runs 6 to 11 (32 blocks to one), one and two column tiles of both widths, and
invariant, per-slice and per-pair steps; an entry read from the wrong place gives a wrong amplitude.
"""
import numpy as np
import pytest

import oracle
from qxgen import circuits as C

from ._util import assert_parity, grid_case

pytestmark = pytest.mark.gpu


def _steps(listing):
    """(level, n, run) of every general in-place A step."""
    out = set()
    for line in listing.splitlines():
        if " a_gather=2" not in line:
            continue
        f = dict(x.split("=", 1) for x in line.split()[4:] if "=" in x)
        am, ak = ([int(x) for x in f[k].split(",")] for k in ("am", "ak"))
        tile = sorted(am[:7] + ak[:4])
        run = next((i for i, p in enumerate(tile) if p != i), 11)
        out.add((line.split()[3], int(f["n"]), run))
    return out


@pytest.mark.parametrize("rows,cols,depth,n_open,n_slice,want", [
    (4, 4, 12, 6, 0, {("pair", 6, 6)}),
    (4, 4, 12, 8, 2, {("pair", 7, 11)}),
    (4, 4, 16, 6, 0, {("shared", 5, 6)}),
    (4, 4, 20, 8, 2, {("slice", 6, 7), ("slice", 6, 8), ("slice", 5, 7), ("pair", 7, 10)}),
    (4, 5, 10, 0, 0, {("pair", 6, 9), ("pair", 5, 6)}),
])
@pytest.mark.parametrize("n_bits", [1, 5])
def test_steps_that_read_a_in_place_match_the_oracle(rows, cols, depth, n_open, n_slice, want, n_bits):
    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx
    circ, om, order, sliced, bits = grid_case(rows, cols, depth, 1, n_open, n_slice, n_bits)
    n, recs = circ.n_qubits, C.gates_to_records(circ)
    c = qx.Contractor(n, recs, om, order, sliced, n_bits, precision=qx.QX_PREC_3XTF32)
    assert want <= _steps(qx.qx_describe_plan(c.h))
    got = c.contract(bits)
    assert np.array_equal(got, c.contract(bits))
    qx.qx_device_status(c.h)
    c.close()
    assert_parity(got, oracle.sv_amplitudes(n, recs, om, bits), what="3xtf32")
