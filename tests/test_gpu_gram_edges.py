"""The tensor-core scan where its items are stepped through: node counts around the 16- and 32-node tiles, more items than CTAs,
several key heads per value head or one, several node groups per sequence; every layer's outputs against the oracle."""
import numpy as np
import pytest
import torch

from synthetic import workload as W
from synthetic.device_case import DeviceCase
from tests.harness import assert_close, ctx, oracle_scan_from_device

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
