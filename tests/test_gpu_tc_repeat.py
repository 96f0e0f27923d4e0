"""The direct tensor-core kernels give the same bits on every call (needs a GPU).

Their converter and MMA warps hand stages to one another through rings whose slots alternate between
two warps.  With other launches on the same SMs (concurrent issue) one of the two can run ahead of
the other by a slot's whole use, so the order of the waits decides whether it reads finished data:
a call then gave one wrong amplitude in about a hundred.  Repeated calls must agree bit for bit.
"""
import numpy as np
import pytest

from qxgen import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("memo", [0, 1])
def test_repeated_direct_contractions_agree_bit_for_bit(memo):
    import torch

    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx
    w = W.sliced()
    c = qx.Contractor(w.n_qubits, w.gates, w.open_mask, w.order, w.sliced, len(w.bitstrings),
                      precision=qx.QX_PREC_3XTF32)
    qx.qx_set_memo(c.h, memo)
    assert "tc_direct" in qx.qx_describe_plan(c.h)
    bits = torch.from_numpy(w.bitstrings).cuda()
    out = torch.empty((len(w.bitstrings), 1, 2), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    first = None
    for i in range(250):
        c.contract_device(bits, out)
        torch.cuda.synchronize()
        got = out.cpu().numpy().copy()
        if first is None:
            first = got
        assert np.array_equal(got, first), f"call {i} differs"
    qx.qx_device_status(c.h)
    c.close()
