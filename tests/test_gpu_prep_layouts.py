"""The operand splits of the pre-split tensor-core forms from both stored layouts (needs a GPU): [K][R]
operands pass through a tile of shared memory, [R][K] ones don't.  Swapping the operands of a product
swaps their layouts, so both sides (the second is expanded) are read both ways.

Bounds, one tensor-core step each.  BF16x3: the parity bounds of complex64.  FP16: an operand is rounded
to 11 bits, at most 2^-11 of its magnitude, so a term of the sum is off by at most 2^-10 of its own; the
terms' errors are independent in sign, so over the request the error stays below 2^-10 of the norm."""
import numpy as np
import pytest

import oracle
from qxgen import circuits as C

from ._util import assert_parity, rel_l2
from .test_gpu_gemm_shapes import halves_order, two_halves

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("n_a,n_k,n_b", [(7, 5, 7), (8, 6, 7), (7, 8, 7)])
@pytest.mark.parametrize("precision", [2, 3])
def test_splits_from_both_layouts(precision, n_a, n_k, n_b, swap):
    import torch

    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx
    circ, n_first = two_halves(n_a, n_k, n_b, 11 * n_a + n_k + 100 * n_b)
    n, recs = circ.n_qubits, C.gates_to_records(circ)
    open_mask = np.zeros(n, np.uint8)
    open_mask[:n_a] = 1
    open_mask[n - n_b:] = 1
    order = halves_order(circ, n_first, open_mask)
    if swap:
        order[-1] = order[-1][::-1]
    bits = C.random_bitstrings(n, 5, 5)
    c = qx.Contractor(n, recs, open_mask, order, [], len(bits), precision=precision)
    tc = [line.split() for line in qx.qx_describe_plan(c.h).splitlines() if line.split()[2].startswith("tc_")]
    assert len(tc) == 1 and tc[0][2] == "tc_prep"
    assert ("a_kmajor=0" in tc[0]) == swap and ("b_kmajor=0" in tc[0]) == (not swap)
    got = c.contract(bits)
    c.close()
    torch.cuda.empty_cache()
    ref = oracle.sv_amplitudes(n, recs, open_mask, bits)
    if precision == 2:
        assert_parity(got, ref)
    else:
        assert rel_l2(got, ref) <= 2.0 ** -10
