"""The slice sum's look-ahead: slice counts around it give the compensated sum of the single slices
(needs a GPU)."""
import math

import numpy as np
import pytest

from qxgen import circuits as C

from ._util import grid_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qx():
    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx as mod
    return mod


@pytest.mark.parametrize("n_s", [1, 2, 15, 16, 17, 31, 32, 33, 48, 64])
def test_slice_sum_over_any_number_of_slices(qx, n_s):
    """Slice counts around the look-ahead of 16, for two amplitudes per bitstring and a ragged count of
    them: the sum equals the compensated sum of the single slices.  Each of those is a float32 value
    times one FP64 factor, rounded a few times, so the sums agree to 8 * 2^-53 of the terms' total."""
    circ, om, order, sliced, bits = grid_case(3, 4, 8, 55, 1, 6, 21)
    c = qx.Contractor(circ.n_qubits, C.gates_to_records(circ), om, order, sliced, len(bits))
    one = [c.contract_slices(bits, s, s + 1) for s in range(n_s)]
    got = c.contract_slices(bits, 0, n_s)
    c.close()
    for part in ("real", "imag"):
        terms = np.stack([getattr(v, part) for v in one])
        want = np.array([math.fsum(t) for t in terms.reshape(n_s, -1).T]).reshape(got.shape)
        room = 8 * 2.0 ** -53 * (np.abs(np.stack(one)).sum(0) + 1e-300)
        assert np.all(np.abs(getattr(got, part) - want) <= room)
