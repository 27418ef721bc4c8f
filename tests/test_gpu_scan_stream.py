"""The streamed scan (closed form, state in tensor memory) at its edges: groups of 32 nodes and what is left over, trees cut into
groups that share one state or are dealt out to several CTAs, skipped and padded rows, both output types, and values that are
not finite.

Bound: keys, values and queries enter exactly, the state, q~, M diag(beta) and the coefficients of q~ as two bf16 terms each, which leaves
2^-18 of a factor, and the product of two low terms is dropped, another 2^-18.  The same arithmetic in float64 on trees like these is off
by 1.1e-6 to 3.3e-6 (1 + |ref|), and the tensor core's fp32 sums add as much again (measured 4.7e-6 at most).  With a low term left out
it is off by 9e-6 to 3e-5 (coefficients of q~), 1e-4 (q~, the state) or 6e-4 to 2e-3 (M diag(beta))."""
import numpy as np
import pytest
import torch

from synthetic import workload as W
from synthetic.device_case import DeviceCase
from tests.graph_nodes import Captured
from tests.harness import assert_close, ctx, oracle_scan_from_device

pytestmark = pytest.mark.gpu
BOUND = 8e-6


def _case(N, B, Hk, Hv, L, depth, seed=0):
    trees = [W.tree_random(W.IntStream(N + b + seed), N, depth) if N > 1 else [-1] for b in range(B)]
    return W.make_case("stream", trees, seed=N + seed, Hk=Hk, Hv=Hv, d=128, in_dtype="bf16", n_layers=L, Ns=N + 3, permute_slots=True)


@pytest.mark.parametrize("N,B,Hk,Hv,L,depth", [(1, 1, 2, 4, 1, 1), (2, 2, 1, 3, 1, 2), (15, 3, 4, 4, 2, 16), (16, 1, 2, 4, 3, 4), (17, 2, 2, 4, 1, 9),
                                               (32, 1, 4, 8, 1, 16), (33, 1, 2, 4, 1, 6), (64, 1, 2, 4, 2, 5), (65, 2, 4, 8, 1, 16), (150, 1, 2, 6, 1, 12),
                                               (256, 1, 4, 8, 1, 16), (256, 5, 16, 32, 2, 11), (100, 3, 8, 24, 5, 8)])
@pytest.mark.parametrize("out_dtype", ["f32", "bf16"])
def test_outputs_match_oracle(N, B, Hk, Hv, L, depth, out_dtype):
    c = _case(N, B, Hk, Hv, L, depth)
    if B > 1:
        c.state_row[B - 1] = -1                       # a skipped sequence
    dc = DeviceCase(ctx("tensor"), c, out_dtype=out_dtype)
    for l in range(L):
        dc.t("out", l).fill_(float("nan"))
    dc.verify()
    torch.cuda.synchronize()
    ctx("auto")
    for l in range(L):
        ref, _, _ = oracle_scan_from_device(dc, layer=l)
        worst = assert_close(dc.np("out", l), ref, bf16=out_dtype == "bf16", what=f"layer {l}")
        assert out_dtype == "bf16" or worst < BOUND
        assert dc.np("status", l).tolist() == [0] * B
        for b in range(B):
            pad = sorted(set(range(c.Ns)) - set(c.slot[b].tolist()))
            assert np.all(dc.np("out", l)[b, pad] == 0.0)


@pytest.mark.parametrize("which", ["q", "k", "v"])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("N,B,L", [(30, 3, 8), (150, 2, 3), (150, 2, 4)])
@pytest.mark.parametrize("out_dtype", ["f32", "bf16"])
def test_values_that_are_not_finite_stay_on_their_paths(which, value, N, B, L, out_dtype):
    """One element of one node: its descendants' outputs are gone (a key's or value's: NaN in whole rows; a query's: its own alone), every
    other output keeps its bits."""
    c = _case(N, B, 16, 32, L, 9, seed=3)
    dc = DeviceCase(ctx("tensor"), c, out_dtype=out_dtype, use_conv=False, qk_l2norm=True)
    dc.verify()
    torch.cuda.synchronize()
    clean = dc.t("out", L - 1).clone()
    node, b = N // 3, B - 1
    dc.t(which, L - 1)[b, int(c.slot[b, node]), :, 77] = value
    dc.verify()
    torch.cuda.synchronize()
    ctx("auto")
    got = dc.t("out", L - 1)
    below = np.zeros(N, dtype=bool)
    for i in range(N):
        below[i] = i == node or (which != "q" and c.parent[b, i] >= 0 and below[c.parent[b, i]])
    gone = [int(c.slot[b, i]) for i in range(N) if below[i]]
    kept = [int(c.slot[b, i]) for i in range(N) if not below[i]]
    assert not torch.isfinite(got[b, gone]).all(dim=-1).any()
    assert which == "q" or torch.isnan(got[b, gone]).all()
    assert torch.equal(got[b, kept], clean[b, kept]) and torch.equal(got[:b], clean[:b])


@pytest.mark.parametrize("N,depth,items,streamed", [(64, 12, 72, True), (64, 12, 80, False), (64, 12, 304, False), (64, 12, 640, True), (50, 12, 148, True),
                                                    (50, 12, 224, True), (56, 16, 224, False), (56, 16, 304, True), (128, 9, 92, False), (128, 9, 100, True),
                                                    (150, 9, 88, False), (160, 12, 180, False), (160, 12, 224, True), (96, 12, 148, True), (28, 12, 224, True)])
def test_the_form_that_measured_faster_is_taken(N, depth, items, streamed):
    """Closed form over groups of 64 or streamed groups of 32, on a B200's 148 SMs; either way the oracle's outputs."""
    c = _case(N, items // 4, 2, 4, 1, depth)
    dc = DeviceCase(ctx("tensor"), c, use_conv=False, qk_l2norm=True)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        name, = [n for n, _ in Captured(dc.verify).kernels]
        assert ("scan_stream_kernel" in name) == streamed and ("scan_gram_kernel" in name) == (not streamed)
    dc.verify()
    torch.cuda.synchronize()
    ctx("auto")
    ref, _, _ = oracle_scan_from_device(dc)
    assert assert_close(dc.np("out"), ref) < (BOUND if streamed else 2 ** -15)     # (the closed form: pairs of 2^-16 on either side)
