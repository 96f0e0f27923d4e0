"""Group members run as launches over batches (chosen at bind) and members in the persistent launch
give the values of the persistent executor (needs a GPU): the same FP32 slice results and the same
compensated sums; only the last FP64 product, by the circuit's scale factor, is rounded in another
kernel, so amplitudes agree to a few roundings of it.  A replay gives the bits of the eager run."""
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


def _same(got, ref):
    # re * sr - im * si: two products and a sum, at most three roundings of 2^-53 |amplitude| on each side
    return np.all(np.abs(got - ref) <= 8 * 2.0 ** -53 * np.abs(ref))


def _contractor(qx, w, **kw):
    return qx.Contractor(w.n_qubits, w.gates, w.open_mask, w.order, w.sliced, len(w.bitstrings), **kw)


@pytest.mark.parametrize("js", [(121,), (100,), (101,), (119,), (111, 121, 101), (118, 100, 107)])
def test_group_members_give_the_persistent_executors_values(qx, js):
    import torch
    ws = [W.batched_circuit(j) for j in js]
    want = []
    for w in ws:
        p = _contractor(qx, w, executor=qx.EXEC_PERSISTENT)
        want.append(p.contract(w.bitstrings))
        p.close()
    stream = torch.cuda.Stream()
    members = [_contractor(qx, w, executor=qx.EXEC_GROUP_MEMBER, stream=stream) for w in ws]
    bits = [torch.from_numpy(w.bitstrings).cuda() for w in ws]
    torch.cuda.synchronize()
    whole = qx.Group(members, bits)
    alone = qx.Group(members[:1], bits[:1])  # a second group over the same handle, its own scratch
    for run in range(2):
        whole.run()
        alone.run()
    torch.cuda.synchronize()
    for got, ref in zip(whole.amplitudes() + alone.amplitudes(), want + want[:1]):
        assert _same(got, ref)
    eager = whole.amplitudes()
    whole.capture()
    for a in whole.d_amps:
        a.zero_()
    torch.cuda.synchronize()
    whole.replay()
    torch.cuda.synchronize()
    for got, ref in zip(whole.amplitudes(), eager):
        assert np.array_equal(got, ref)
    alone.close()
    whole.close()


def test_both_ways_are_taken(qx):
    """Little work per pair stays in the persistent launch; much goes to launches."""
    import torch
    ws = [W.batched_circuit(j) for j in (121, 118)]
    stream = torch.cuda.Stream()
    members = [_contractor(qx, w, executor=qx.EXEC_GROUP_MEMBER, stream=stream) for w in ws]
    bits = [torch.from_numpy(w.bitstrings).cuda() for w in ws]
    torch.cuda.synchronize()
    g = qx.Group(members, bits)
    g.run()
    torch.cuda.synchronize()
    assert members[0].stats()["launches"] == 0 and members[1].stats()["launches"] > 0
    g.close()
