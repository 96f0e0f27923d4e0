"""The packed complex64 GEMM on all its tiles, and the kernels beside it (needs a GPU).

The networks are one product of two halves of a circuit (test_gpu_gemm_shapes) whose operands or result
are too large for a segment, so the last step is a launch of the kernel that gemm_route names for the
call's items; listing, route and profile are asserted.  Many items and a few take different kernels for
the same sums: the amplitudes must agree bit for bit, and with the state vector.
"""
import numpy as np
import pytest

import oracle
from qxgen import circuits as C

from ._util import assert_parity
from .test_gemm_route import PACKED, SKINNY, TILE, gemm_route
from .test_gpu_gemm_shapes import halves_order, two_halves

pytestmark = pytest.mark.gpu


def _run(n_a, n_k, n_b, swap, counts):
    """Amplitudes of the first counts[i] bitstrings, the last step's listing, and the sizes m, k, n."""
    from paper_2110_09894_gb300 import build
    build.build()
    import torch

    from paper_2110_09894_gb300 import qx
    circ, n_first = two_halves(n_a, n_k, n_b, 13 * n_a + n_k + 100 * n_b)
    n, recs = circ.n_qubits, C.gates_to_records(circ)
    open_mask = np.zeros(n, np.uint8)
    open_mask[:n_a] = 1
    open_mask[n - n_b:] = 1
    order = halves_order(circ, n_first, open_mask)
    if swap:  # half b as the first operand: the operands trade their layouts
        order[-1] = order[-1][::-1]
    m, n_cols = (n_b, n_a) if swap else (n_a, n_b)
    bits = C.random_bitstrings(n, max(counts), 5)
    c = qx.Contractor(n, recs, open_mask, order, [], len(bits), gemm_min_bits=min(3, n_k))
    gemms = [line.split() for line in qx.qx_describe_plan(c.h).splitlines() if line.split()[2] == "gemm"]
    assert len(gemms) == 1 and not any(x.startswith(("seg=", "chain=")) for x in gemms[0])
    assert {f"m={m}", f"k={n_k}", f"n={n_cols}"} <= set(gemms[0])
    out = []
    for k in counts:
        qx.qx_set_profiling(c.h, True)
        out.append(c.contract(bits[:k]))
        prof = qx.qx_profile_read(c.h)["gemm"]
        assert prof["launches"] >= 1 and prof["flops"] == 8.0 * k * 2.0 ** (m + n_k + n_cols)
    c.close()
    torch.cuda.empty_cache()  # workspaces of up to a few GB: later tests measure the free memory
    assert_parity(out[0][:3], oracle.sv_amplitudes(n, recs, open_mask, bits[:3]))
    for got in out[1:]:
        assert np.array_equal(got, out[0][:len(got)])
    return gemms[0], (m, n_k, n_cols)


@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("n_a,n_k,n_b,items", [
    (5, 5, 5, 513), (5, 6, 5, 512), (5, 7, 5, 521),                  # 32 x 32
    (6, 3, 5, 513), (7, 6, 5, 256), (7, 7, 5, 257), (7, 8, 5, 256),  # 64 x 32 (and 32 x 64 by `swap`)
    (5, 3, 6, 512), (5, 4, 7, 257), (5, 7, 6, 513),                  # 32 x 64
    (6, 3, 6, 153), (6, 6, 6, 152), (6, 7, 6, 153), (7, 8, 6, 77)])  # 64 x 64
def test_packed_tiles_match_the_other_kernels(n_a, n_k, n_b, items, swap):
    line, (m, k, n) = _run(n_a, n_k, n_b, swap, (items, 3, 1))
    assert gemm_route(m, n, k, items) == (PACKED, min(m, 6), min(n, 6))
    assert gemm_route(m, n, k, 3)[0] != PACKED
    # both layouts of both operands over the two orders
    assert ("a_kmajor=0" in line) == swap and ("b_kmajor=0" in line) == (not swap)


@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("n_a,n_k,n_b,counts,kinds", [
    (4, 7, 5, (400, 70, 1), (TILE, TILE, TILE)), (4, 7, 4, (400, 153, 1), (TILE, TILE, TILE)),
    (3, 5, 8, (300, 152, 1), (TILE, TILE, TILE)), (3, 8, 4, (310, 152, 1), (TILE, SKINNY, SKINNY)),
    (1, 10, 4, (64, 17, 1), (SKINNY, SKINNY, SKINNY)), (2, 9, 6, (80, 17, 1), (SKINNY, SKINNY, SKINNY)),
    (4, 8, 3, (400, 17, 1), (TILE, SKINNY, SKINNY)), (3, 9, 3, (160, 153, 1), (SKINNY, SKINNY, SKINNY))])
def test_short_sides_and_small_tiles_run_outside_segments(n_a, n_k, n_b, counts, kinds, swap):
    _, (m, k, n) = _run(n_a, n_k, n_b, swap, counts)
    assert tuple(gemm_route(m, n, k, c)[0] for c in counts) == kinds
