"""Graph replay with buffers that change from call to call, on a side stream and on the legacy default
stream (needs a GPU): every call gives the bits of an eager one, in the buffer it was given.
"""
import numpy as np
import pytest

from qxgen import circuits as C

from ._util import grid_case

pytestmark = pytest.mark.gpu


def _contractor(n_bits, precision, side=False):
    import torch

    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx
    circ, om, order, sliced, bits = grid_case(4, 4, 12, 7, 2, 2, n_bits)
    c = qx.Contractor(circ.n_qubits, C.gates_to_records(circ), om, order, sliced, n_bits, precision=precision,
                      stream=torch.cuda.Stream() if side else torch.cuda.default_stream())
    return torch, qx, c, bits


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("side", [False, True])
def test_fresh_buffers_and_sizes_match_eager_calls(precision, side):
    torch, qx, c, bits = _contractor(24, precision, side)
    qx.qx_set_graphs(c.h, False)
    calls = [(slice(0, 6), 0, 4)] * 4 + [(slice(6, 12), 0, 4)] * 3 + [(slice(3, 9), 1, 3)] * 2 + \
            [(slice(12, 18), 0, 4), (slice(0, 1), 0, 4), (slice(0, 24), 0, 4), (slice(0, 24), 0, 4)]
    want = []
    for sl, s0, s1 in calls:
        with torch.cuda.stream(c.stream):
            out = c.contract_device(torch.from_numpy(bits[sl].copy()).cuda(), None, s0, s1)
        torch.cuda.synchronize()
        want.append(out.cpu().numpy())
    qx.qx_set_graphs(c.h, True)
    keep = []
    with torch.cuda.stream(c.stream):
        for i, (sl, s0, s1) in enumerate(calls):
            d_bits = torch.from_numpy(bits[sl].copy()).cuda()
            out = torch.full((len(bits[sl]), 4, 2), 7.0, dtype=torch.float64, device="cuda") if i % 2 else None
            keep.append((d_bits, c.contract_device(d_bits, out, s0, s1)))  # enqueued only: no wait between
    torch.cuda.synchronize()
    qx.qx_device_status(c.h)
    for i, (got, ref) in enumerate(zip(keep, want)):
        assert np.array_equal(got[1].cpu().numpy(), ref), i
    # a host call goes through the same workspace buffers
    for i in (0, 4, 11):
        assert np.array_equal(c.contract(bits[calls[i][0]]), want[i][..., 0] + 1j * want[i][..., 1])
    c.close()


def test_a_replay_ends_an_open_sum_of_parts():
    """A replayed whole contraction ends an open sum of parts, as an eager one does."""
    torch, qx, c, bits = _contractor(5, 0)
    want = c.contract(bits)
    for _ in range(3):
        assert np.array_equal(c.contract(bits), want)
    d_bits = torch.from_numpy(bits).cuda()
    amps = torch.zeros((5, 4, 2), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for _ in range(3):
        qx.qx_submit_part(c.h, d_bits.data_ptr(), 5, 0, 2, True, False, amps.data_ptr())
        qx.qx_submit_part(c.h, d_bits.data_ptr(), 5, 2, 4, False, True, amps.data_ptr())
        torch.cuda.synchronize()
        got = amps.cpu().numpy()
        assert np.array_equal(got[..., 0] + 1j * got[..., 1], want)
    for _ in range(3):
        qx.qx_submit_part(c.h, d_bits.data_ptr(), 5, 0, 2, True, False, amps.data_ptr())
        assert np.array_equal(c.contract(bits), want)
        with pytest.raises(qx.QXError):
            qx.qx_submit_part(c.h, d_bits.data_ptr(), 5, 2, 4, False, True, amps.data_ptr())
    torch.cuda.synchronize()
    c.close()
