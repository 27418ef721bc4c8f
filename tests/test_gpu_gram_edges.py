"""The tensor-core scan where its items are stepped through: node counts around the 16- and 32-node tiles, more items than CTAs,
several key heads per value head or one, several node groups per sequence; every layer's outputs against the oracle."""
import numpy as np
import pytest
import torch

from synthetic import workload as W
from synthetic.device_case import DeviceCase
from tests.harness import assert_close, ctx, oracle_scan_from_device
from tests.test_gpu_fused import _share_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,Hk,Hv", [(1, 8, 8), (8, 2, 8), (15, 4, 12), (16, 8, 8), (17, 2, 6), (31, 8, 16), (32, 1, 8), (33, 3, 6), (150, 2, 4)])
def test_stepped_items(N, Hk, Hv):
    B = 5
    L = 600 // (B * Hv) + 3
    trees = [W.tree_random(W.IntStream(N + b), N, 14) if N > 1 else [-1] for b in range(B)]
    c = W.make_case("edges", trees, seed=N, Hk=Hk, Hv=Hv, d=128, in_dtype="bf16", n_layers=L, Ns=N + 3, permute_slots=True)
    c.state_row[3] = -1      # a skipped sequence in the middle of every layer's items
    dc = DeviceCase(ctx("tensor"), c)
    for l in range(L):
        dc.t("out", l).fill_(float("nan"))
    dc.verify()
    torch.cuda.synchronize()
    ctx("auto")
    for l in (0, 1, L // 2, L - 1):
        out, _, _ = oracle_scan_from_device(dc, layer=l)
        assert_close(dc.np("out", l), out, what=f"outputs of layer {l}")
        assert np.all(dc.np("out", l)[3] == 0.0)


@pytest.mark.parametrize("N,B,L,fused", [(24, 4, 9, False), (24, 4, 9, True), (60, 3, 12, False), (60, 3, 12, True), (150, 3, 9, False)])
def test_overlapped_launches_of_many_waves(N, B, L, fused):
    """Launches of several waves with and without kernel overlap: the same bits over cycles that feed each other."""
    P, C = [W.make_case("waves", [W.tree_random(W.IntStream(s + N + b), N, 12) for b in range(B)], seed=s, Hk=8, Hv=24, d=128,
                        in_dtype="bf16", n_layers=L, Ns=N + 2, permute_slots=True) for s in (5, 6)]
    assert L * B * 24 > 4 * 148
    C.state_row = P.state_row.copy()
    runs = []
    for on in (False, True):
        c = ctx("auto")
        c.set_overlap(on)
        dp, dc = DeviceCase(c, P), DeviceCase(c, C)
        other = _share_state(dp, dc)
        outs = []
        for _ in range(3):
            dp.verify()
            outs.append(dp.t("out", L - 1).clone())
            if fused:
                c.commit_verify(dp.desc, dp.layers, dp.accepted, dp.accepted_len, dc.desc, other)
            else:
                dp.commit()
                c.verify(dc.desc, other)
            outs += [other[l].tensors["out"].clone() for l in (0, L - 1)]
            c.commit(dc.desc, other, dc.accepted, dc.accepted_len)
        torch.cuda.synchronize()
        runs.append(outs + [dp.t("state", l).clone() for l in (0, L - 1)] + [dp.t("conv_hist", L - 1).clone()])
    ctx("auto").set_overlap(True)
    for a, b in zip(*runs):
        assert torch.equal(a, b)
    assert not torch.equal(runs[0][0], runs[0][3])      # the cycles advanced the state
