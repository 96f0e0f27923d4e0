"""A group member's amplitudes have the same bits whether its steps run as launches over batches (chosen
at bind, so it depends on the scratch and on the other members) or in the persistent launch (needs a GPU)."""
import numpy as np
import pytest

from qxgen import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("js", [(121,), (100,), (101,), (119,), (111, 121, 101), (118, 100, 107), (103,)])
def test_group_members_give_the_persistent_executors_bits(js):
    import torch

    from paper_2110_09894_gb300 import build
    build.build()
    from paper_2110_09894_gb300 import qx
    ws = [W.batched_circuit(j) for j in js]
    stream = torch.cuda.Stream()

    def contractors(executor):
        return [qx.Contractor(w.n_qubits, w.gates, w.open_mask, w.order, w.sliced, len(w.bitstrings),
                              executor=executor, stream=stream) for w in ws]

    want = []
    for w, p in zip(ws, contractors(qx.EXEC_PERSISTENT)):
        want.append(p.contract(w.bitstrings))
        p.close()
    members = contractors(qx.EXEC_GROUP_MEMBER)
    bits = [torch.from_numpy(w.bitstrings).cuda() for w in ws]
    torch.cuda.synchronize()
    group = qx.Group(members, bits)
    group.run()
    torch.cuda.synchronize()
    for got, ref in zip(group.amplitudes(), want):
        assert np.array_equal(got, ref)
    group.close()
