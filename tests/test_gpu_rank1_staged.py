"""The rank-1 scan with all operands of a tree in shared memory, and the edge beyond which it falls back to the operand ring:
outputs and exported node states against the oracle, in every snapshot mode."""
import numpy as np
import pytest
import torch

from synthetic import workload as W
from synthetic.device_case import DeviceCase
from tests.harness import assert_close, ctx, oracle_scan_from_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("d,dtype,N", [(64, "f32", 1), (64, "bf16", 33), (64, "f32", 110), (64, "f32", 150), (128, "f32", 2), (128, "bf16", 31),
                                       (128, "bf16", 64), (128, "f32", 67), (128, "bf16", 72)])
def test_staged_scan(d, dtype, N, mode):
    trees = [W.tree_random(W.IntStream(N + 1), N, 9) if N > 2 else [-1] * N, [-1 if i % 7 == 0 else i - 1 for i in range(N)]]
    c = W.make_case("staged", trees, seed=N, Hk=1, Hv=2, d=d, in_dtype=dtype, Ns=N + 2, permute_slots=True)
    nodes = None
    if mode == 1:      # leaves and inner nodes, one of them twice, one entry unused
        nodes = np.stack([np.array([N - 1, 0, N // 2, N // 2, -1], dtype=np.int32)] * 2)
    dc = DeviceCase(ctx("rank1"), c, snapshot_mode=mode, snap_nodes=nodes)
    dc.verify()
    torch.cuda.synchronize()
    ctx("auto")
    want = {0: None, 1: nodes, 2: np.tile(np.arange(N, dtype=np.int32), (2, 1))}[mode]
    out, snap, _ = oracle_scan_from_device(dc, snap_nodes=want)
    assert_close(dc.np("out"), out, what="outputs")
    if mode:
        used = want >= 0
        assert_close(dc.np("snap_out")[used], np.asarray(snap)[used], what="node states")
