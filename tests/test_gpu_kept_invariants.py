"""Invariant intermediates kept across calls (qx_set_memo), CUDA graphs and expired waits together
(needs a GPU).  A call that computes them launches more kernels than one that finds them kept, which is
what these tests count.  Nothing faults: a wait limit of one cycle makes the tensor-core kernels give up
and return (see test_gpu_timeout)."""
import numpy as np
import pytest

from qxgen import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qx():
    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx as mod
    return mod


def _contractor(qx, n_bits, **kw):
    import torch
    w = W.sliced()
    bits = np.ascontiguousarray(w.bitstrings[:n_bits])
    c = qx.Contractor(w.n_qubits, w.gates, w.open_mask, w.order, w.sliced, n_bits, precision=1,
                      stream=torch.cuda.Stream(), **kw)
    d_bits = torch.from_numpy(bits).cuda()
    out = torch.zeros((n_bits, 1, 2), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return torch, c, d_bits, out


@pytest.mark.parametrize("fresh", [False, True])
def test_a_reported_expiry_drops_graphs_without_the_invariant_steps(qx, fresh):
    torch, c, d_bits, out = _contractor(qx, 8, timeout_cycles=1)
    keep = []

    def call():
        with torch.cuda.stream(c.stream):
            keep.append(c.contract_device(d_bits.clone() if fresh else d_bits, None if fresh else out))
        return c.stats()["launches"]

    qx.qx_set_memo(c.h, True)
    whole = call()
    kept = [call(), call()]  # captured, replayed
    assert kept[0] == kept[1] < whole
    with pytest.raises(qx.QXError) as e:
        qx.qx_device_status(c.h)
    assert e.value.code == qx.QX_ETIMEOUT
    assert call() == whole
    torch.cuda.synchronize()
    c.close()


def test_a_captured_call_that_has_not_run_keeps_nothing(qx):
    torch, c, d_bits, out = _contractor(qx, 8)
    with torch.cuda.stream(c.stream):
        want = c.contract_device(d_bits, out).clone()
    whole = c.stats()["launches"]
    torch.cuda.synchronize()
    qx.qx_set_memo(c.h, True)
    captured = torch.zeros_like(out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=c.stream):
        c.contract_device(d_bits, captured)
    counts = []
    for _ in range(2):
        out.zero_()
        torch.cuda.synchronize()
        c.contract_device(d_bits, out)
        counts.append(c.stats()["launches"])
        torch.cuda.synchronize()
        assert torch.equal(out, want)
    assert counts[0] == whole > counts[1]
    with torch.cuda.stream(c.stream):
        graph.replay()  # holds the invariant steps itself
    torch.cuda.synchronize()
    assert torch.equal(captured, want)
    qx.qx_device_status(c.h)
    c.close()
