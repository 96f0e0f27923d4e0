"""The complex64 products' kernels at the edges of their tiles (needs a GPU).

Two gate-sized tensors cannot reach these shapes, so the networks here are one product between two
halves of a circuit: n_a qubits of one half, n_b of the other and the wires between them decide the
product's free and contracted sides.  Every shape is checked against the state vector; shapes of the
same sum in different kernels (few or many bitstrings) must agree bit for bit.
"""
import numpy as np
import pytest

import oracle
from qxgen import circuits as C
from qxgen import plan as P

from ._util import assert_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qx():
    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx as mod
    return mod


def two_halves(n_a, n_k, n_b, seed):
    """A circuit whose plan ends in one product of 2^(open of a) x 2^n_k x 2^(open of b): qubits 0 ..
    n_a + n_k - 1 evolve first (half a), then n_k of them meet n_b fresh qubits (half b).  Open qubits:
    n_a from half a, and those of half b that stay open."""
    n = n_a + n_k + n_b
    circ = C.Circuit(n)
    rng = C.SplitMix64(seed)

    def layer(qs):
        for q in qs:
            circ.append((q,), C.ONE_QUBIT_SET[rng.randint(3)])
        for parity in (0, 1):
            for i in range(parity, len(qs) - 1, 2):
                circ.append((qs[i], qs[i + 1]), C.FSIM_SYC)
    a, b = list(range(n_a + n_k)), list(range(n_a, n))
    for _ in range(3):
        layer(a)
    n_first = len(circ.gates)
    for _ in range(3):
        layer(b)
    return circ, n_first


def halves_order(circ, n_first, open_mask):
    """Contract half a's tensors, then half b's with the outputs, then the two results."""
    legs, _, _ = P.network_legs(circ.n_qubits, [g.qubits for g in circ.gates], open_mask)
    n, N = circ.n_qubits, len(legs)
    first_used = {}
    for g, gate in enumerate(circ.gates):
        for q in gate.qubits:
            first_used.setdefault(q, g)
    half = [None] * N
    for t in range(N):
        if t < n:
            half[t] = 0 if first_used.get(t, 0) < n_first else 1
        elif t < n + len(circ.gates):
            half[t] = 0 if t - n < n_first else 1
        else:
            wire = legs[t][0]
            src = next(s for s in range(N) if s != t and wire in legs[s])
            half[t] = half[src]
    order, roots = [], []
    for side in (0, 1):
        ids = [t for t in range(N) if half[t] == side]
        cur = ids[0]
        for t in ids[1:]:
            order.append((cur, t))
            cur = N + len(order) - 1
        roots.append(cur)
    order.append(tuple(roots))
    return order


@pytest.mark.parametrize("n_a,n_k,n_b", [
    (5, 3, 5), (5, 6, 5), (5, 7, 6), (6, 6, 6), (7, 7, 5), (6, 8, 6), (8, 5, 5), (5, 4, 9),   # packed tiles
    (0, 7, 3), (1, 6, 6), (2, 9, 5), (7, 7, 1), (8, 6, 2), (3, 8, 3), (4, 9, 4), (3, 4, 3)])  # short sides
def test_one_product_against_the_state_vector(qx, n_a, n_k, n_b):
    circ, n_first = two_halves(n_a, n_k, n_b, 17 * n_a + n_k + 100 * n_b)
    n, recs = circ.n_qubits, C.gates_to_records(circ)
    open_mask = np.zeros(n, np.uint8)
    open_mask[:n_a] = 1                 # half a's own qubits: the rows
    open_mask[n - n_b:] = 1             # half b's fresh qubits: the columns
    order = halves_order(circ, n_first, open_mask)
    bits = C.random_bitstrings(n, 9, 5)
    c = qx.Contractor(n, recs, open_mask, order, [], len(bits), gemm_min_bits=min(3, n_k))
    lines = qx.qx_describe_plan(c.h).splitlines()
    got = c.contract(bits)
    few = c.contract(bits[:1])
    c.close()
    last = lines[-1].split()
    if min(n_a, n_b) >= 3:
        assert last[2] == "gemm" and f"m={n_a}" in last and f"k={n_k}" in last and f"n={n_b}" in last
    assert np.array_equal(few, got[:1])
    assert_parity(got, oracle.sv_amplitudes(n, recs, open_mask, bits))
