"""The acceptance walk's ways of keeping a slice of the residual (float64 or float32 in shared memory, the caller's scratch) and
of reading rows (16 bytes at a time, or rows that start on any 4-byte boundary): vocabularies on each side, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import accept_oracle as A
from synthetic import workload as W
from tests.graph_nodes import Captured
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


@pytest.mark.parametrize("B,V,halved", [(14, 11325, False), (16, 16384, False), (18, 11325, True), (15, 8000, False), (16, 8000, True)])
def test_clusters_are_halved_only_where_they_crowd_the_gpu(B, V, halved):
    """Eight CTAs a sequence or four, as measured: the walk's grid, read from a capture."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the lines are fractions of 148 SMs")
    parents = np.tile(np.array([-1, -1], dtype=np.int32), (B, 1))
    desc = ctx().tree_desc(parents)
    z = lambda *s: torch.zeros(*s, device="cuda")
    i = lambda *s: torch.zeros(*s, dtype=torch.int32, device="cuda")
    args = dict(token=i(B, 2), p_target=z(B, 3, V), q_draft=z(B, 2, V), uniforms=z(B, 2), noise=z(B, V) + 1, work=z(B, V),
                accepted=i(B, 1), length=i(B), next_token=i(B), final_node=i(B), mode="rejection")
    ctx().accept(desc, **args)                    # kernel attributes are set on the first call
    torch.cuda.synchronize()
    (_, params), = Captured(lambda: ctx().accept(desc, **args)).kernels
    assert tuple(params.grid) == (4 if halved else 8, B, 1)
