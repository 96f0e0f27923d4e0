"""A complex64 product takes smaller tiles, or shorter pieces of its long side, where its usual ones are
fewer than the SMs (needs a GPU): a few products and many of the same shape run in different tiles and
must agree bit for bit, and with the state vector.
"""
import numpy as np
import pytest

import oracle
from qxgen import circuits as C

from ._util import assert_parity
from .test_gpu_gemm_shapes import halves_order, two_halves

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_a,n_k,n_b", [
    (6, 6, 6), (6, 7, 7), (7, 4, 6), (5, 7, 6), (4, 5, 5), (3, 3, 7),   # tiles
    (1, 8, 3), (6, 8, 1), (2, 7, 5), (0, 8, 5), (4, 8, 3)])             # a short side
def test_few_products_match_many(n_a, n_k, n_b):
    import torch

    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx
    circ, n_first = two_halves(n_a, n_k, n_b, 31 * n_a + n_k + 100 * n_b)
    n, recs = circ.n_qubits, C.gates_to_records(circ)
    open_mask = np.zeros(n, np.uint8)
    open_mask[:n_a] = 1
    open_mask[n - n_b:] = 1
    order = halves_order(circ, n_first, open_mask)
    bits = C.random_bitstrings(n, 160, 5)
    c = qx.Contractor(n, recs, open_mask, order, [], len(bits), gemm_min_bits=min(3, n_k))
    many = c.contract(bits)
    for k in (1, 17, 152, 153):
        assert np.array_equal(c.contract(bits[:k]), many[:k]), k
    c.close()
    torch.cuda.empty_cache()  # workspaces of up to a few GB: later tests measure the free memory
    assert_parity(many[:3], oracle.sv_amplitudes(n, recs, open_mask, bits[:3]))
