"""The streamed scan's failure path: with the drill on it issues no products and no state copies, so that every bounded wait runs out."""
import numpy as np
import pytest
import torch

from paper_2609_23900_b200 import binding
from synthetic import workload as W
from synthetic.device_case import DeviceCase
from tests.graph_nodes import Captured
from tests.harness import ctx
from tests.test_gpu_fused import _share_state

pytestmark = pytest.mark.gpu


@pytest.fixture
def drill():
    """Switches the drill of the shared context, which is left as it was found."""
    c = ctx("tensor")
    yield c.set_timeout_drill
    c.set_timeout_drill(False)
    ctx("auto")


def _trees(N, B, seed):
    return [W.tree_random(W.IntStream(W.stream_key(seed, b)), N, 9) for b in range(B)]


@pytest.mark.parametrize("N,B,L", [(30, 3, 8), (150, 3, 3)])
def test_every_unit_of_a_verify_reports_the_timeout(N, B, L, drill):
    """More units than CTAs: what a CTA had still to do when it gave up is reported too, and skipped sequences as ever."""
    c = W.make_case("stream", _trees(N, B, 5), seed=N, Hk=16, Hv=32, d=128, in_dtype="bf16", n_layers=L, Ns=N + 3, permute_slots=True)
    c.state_row[1] = -1
    dc = DeviceCase(ctx("tensor"), c, use_conv=False, qk_l2norm=True)
    assert any("scan_stream_kernel" in name for name, _ in Captured(dc.verify).kernels)
    dc.verify()
    torch.cuda.synchronize()
    ref = [dc.t("out", l).clone() for l in range(L)]
    drill(True)
    dc.verify()
    torch.cuda.synchronize()
    for l in range(L):
        assert dc.np("status", l).tolist() == [binding.SEQ_TIMEOUT, binding.SEQ_OK, binding.SEQ_TIMEOUT]
    drill(False)
    for l in range(L):
        dc.t("out", l).fill_(float("nan"))
    dc.verify()
    torch.cuda.synchronize()
    for l in range(L):
        assert dc.np("status", l).tolist() == [binding.SEQ_OK] * B
        assert torch.equal(dc.t("out", l), ref[l])


def _cycle(B=3, L=8):
    """A cycle whose tree is streamed, behind one that accepted paths of three nodes and more."""
    P = W.make_case("prev", [W.tree_chain(6) + [0, 0, 1]] * B, seed=11, Hk=16, Hv=32, d=128, in_dtype="bf16", n_layers=L,
                    accepted=[list(range(3 + b)) for b in range(B)], lmax=6)
    C = W.make_case("cur", _trees(30, B, 7), seed=12, Hk=16, Hv=32, d=128, in_dtype="bf16", n_layers=L, Ns=33, permute_slots=True)
    C.state_row, C.rows = P.state_row.copy(), P.rows
    for p, q in zip(P.layers, C.layers):
        q.state, q.hist = p.state.copy(), p.hist.copy()
    dcP, dcC = DeviceCase(ctx("tensor"), P), DeviceCase(ctx("tensor"), C)
    dcP.verify()
    layers = _share_state(dcP, dcC)
    return dcP, dcC, layers, lambda: ctx("tensor").commit_verify(dcP.desc, dcP.layers, dcP.accepted, dcP.accepted_len, dcC.desc, layers)


def test_every_unit_of_a_fused_call_reports_the_timeout(drill):
    dcP, dcC, layers, call = _cycle()
    assert any("scan_stream_fused_kernel" in name for name, _ in Captured(call).kernels)
    drill(True)
    call()
    torch.cuda.synchronize()
    for l, layer in enumerate(layers):
        assert layer.tensors["status"].tolist() == [binding.SEQ_TIMEOUT] * 3
        assert dcP.np("status", l).tolist() == [binding.SEQ_TIMEOUT] * 3         # nothing was committed


def test_a_state_that_does_not_arrive_is_not_written_back(drill):
    """The accepted path is replayed into the state in shared memory and the rows go back to memory: never rows that did not come."""
    dcP, dcC, layers, call = _cycle()
    before = [dcP.t("state", l).clone() for l in range(len(layers))]
    drill(True)
    call()
    torch.cuda.synchronize()
    for l in range(len(layers)):
        assert torch.equal(dcP.t("state", l), before[l])
    drill(False)
    call()
    torch.cuda.synchronize()
    for l, layer in enumerate(layers):
        assert layer.tensors["status"].tolist() == [binding.SEQ_OK] * 3
        assert not torch.equal(dcP.t("state", l), before[l])
