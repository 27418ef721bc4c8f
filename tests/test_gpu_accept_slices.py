"""The acceptance walk's ways of keeping a slice of the residual (float64 or float32 in shared memory, the caller's scratch) and
of reading rows (16 bytes at a time, or rows that start on any 4-byte boundary): vocabularies on each side, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import accept_oracle as A
from synthetic import workload as W
from tests.harness import ctx
from tests.test_gpu_accept import make_inputs, run_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["rejection", "greedy"])
@pytest.mark.parametrize("B,V", [(1, 511), (2, 2049), (2, 2052), (16, 11325), (10, 147460), (10, 151937), (10, 230000), (10, 230001)])
def test_slices_match_the_oracle(B, V, mode):
    parents = np.array([[-1, -1, 0, 2], [-1, 0, 0, 1]] * B, dtype=np.int32)[:B]
    slot = np.tile(np.array([1, 3, 0, 2], dtype=np.int32), (B, 1))
    inputs = make_inputs(parents, slot, 4, V, seed=V, agree=0.5)
    desc = ctx().tree_desc(parents, slot=slot, n_slots=4)
    lmax = max(max(W.tree_depths(p.tolist())) for p in parents)
    got = run_device(desc, 4, *inputs, mode, lmax)
    torch.cuda.synchronize()
    token, p, q, u, noise = inputs
    ref = A.accept(parents, slot, 4, token, p, q, u, noise, mode=A.GREEDY if mode == "greedy" else A.REJECTION, lmax=lmax)
    for g, r in zip(got, ref):
        assert g.cpu().numpy().tolist() == np.asarray(r).tolist()
