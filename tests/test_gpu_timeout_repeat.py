"""Expired waits, again and again (needs a GPU): with a limit of one cycle most CTAs of a contraction
give up or find that another has, at any moment of their start and on every stream.  Every call must end
by itself, its status must say that it expired, and a call with the default limit must give its bits again.
Nothing faults or hangs here (see test_gpu_timeout): a CTA leaves as a whole or runs to its end."""
import numpy as np
import pytest

from qxgen import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_streams", [1, 8])
@pytest.mark.parametrize("precision", [1, 2, 3])
def test_calls_whose_waits_expire_end(precision, n_streams):
    import torch

    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx
    w = W.sliced()
    bits = np.ascontiguousarray(w.bitstrings[:16])
    args = w.n_qubits, w.gates, w.open_mask, w.order, w.sliced, len(bits)
    whole = qx.Contractor(*args, precision=precision, stream=torch.cuda.Stream())
    want = whole.contract(bits)
    whole.close()
    c = qx.Contractor(*args, precision=precision, stream=torch.cuda.Stream(), timeout_cycles=1)
    qx.qx_set_streams(c.h, n_streams)
    d_bits = torch.from_numpy(bits).cuda()
    out = torch.zeros((len(bits), 1, 2), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for i in range(40):
        c.contract_device(d_bits, out)
        with pytest.raises(qx.QXError) as e:
            qx.qx_device_status(c.h)
        assert e.value.code == qx.QX_ETIMEOUT
    qx.qx_set_options(c.h, precision=precision)
    assert np.array_equal(c.contract(bits), want)
    c.close()
