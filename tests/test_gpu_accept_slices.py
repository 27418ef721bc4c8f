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


@pytest.mark.parametrize("V", [515, 20000, 151936])
@pytest.mark.parametrize("kind", ["ties", "huge", "tiny", "near", "denormal"])
def test_race_and_update_at_the_edges_of_float32(kind, V):
    """The race divides only entries that an approximate quotient leaves in play, and the update widens normal numbers by hand:
    quotients that tie, that overflow or are denormal, that differ in the last bit, and rows with zeros and denormals."""
    rs = np.random.default_rng(V)
    B, N, Ns = 2, 2, 3
    parents, slot = np.array([[-1, -1]] * B, dtype=np.int32), np.array([[2, 0]] * B, dtype=np.int32)
    p = rs.dirichlet(np.full(V, 0.2), size=(B, Ns + 1)).astype(np.float32)
    q = rs.dirichlet(np.full(V, 0.2), size=(B, Ns)).astype(np.float32)
    noise = rs.exponential(size=(B, V)).astype(np.float32) + np.float32(1e-6)
    if kind == "ties":                    # a few distinct values: many entries share the largest quotient
        p = (2.0 ** rs.integers(-20, -16, size=p.shape)).astype(np.float32)
        noise = rs.choice(np.array([0.5, 0.75, 1.0], np.float32), size=noise.shape)
    elif kind == "huge":
        noise *= np.float32(1e-37)        # quotients up to and beyond the largest float, denormal divisors
    elif kind == "tiny":
        noise *= np.float32(1e37)         # denormal quotients
    elif kind == "near":                  # neighbours in float32 around one quotient
        p = np.float32(1e-5) * (1 + rs.integers(-3, 4, size=p.shape) * np.float32(2.0 ** -23)).astype(np.float32)
        noise = (1 + rs.integers(-3, 4, size=noise.shape) * np.float32(2.0 ** -23)).astype(np.float32)
    else:                                 # zeros and denormals among the probabilities
        p[rs.uniform(size=p.shape) < 0.3] = 0
        p[rs.uniform(size=p.shape) < 0.3] *= np.float32(1e-36)
        q[rs.uniform(size=q.shape) < 0.3] *= np.float32(1e-38)
    token = rs.integers(0, V, size=(B, Ns)).astype(np.int32)
    u = np.ones((B, Ns), np.float32)      # refuse what can be refused: updates, then the race
    desc = ctx().tree_desc(parents, slot=slot, n_slots=Ns)
    got = run_device(desc, Ns, token, p, q, u, noise, "rejection", 1)
    torch.cuda.synchronize()
    with np.errstate(all="ignore"):
        ref = A.accept(parents, slot, Ns, token, p, q, u, noise, mode=A.REJECTION, lmax=1)
    for g, r in zip(got, ref):
        assert g.cpu().numpy().tolist() == np.asarray(r).tolist()
