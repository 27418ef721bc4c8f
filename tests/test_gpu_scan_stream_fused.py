"""The streamed scan with the commit folded in, in launches whose CTAs go from one state to the next: every way an accepted path can be
empty, refused or long beside ones that are in order, skipped sequences, raw gates and bias, with and without a convolution in the new
cycle.  State, history, statuses, recorded operands and outputs against the oracles of the separate steps."""
import numpy as np
import pytest
import torch

from oracle import gdn_oracle as O
from paper_2609_23900_b200 import binding
from synthetic import workload as W
from synthetic.device_case import DeviceCase
from tests.graph_nodes import Captured
from tests.harness import assert_close, ctx, device_gates
from tests.test_gpu_scan_stream import BOUND

pytestmark = pytest.mark.gpu

L, HK, HV, LMAX = 20, 2, 4, 16
SPINE = W.tree_chain(16) + [0, 0, 16]               # sixteen nodes in a row, branches at its root


def _paths():
    """(accepted path, claimed length) of each sequence."""
    whole = list(range(16))
    return [([], 0), ([0], 1), ([0, 1], 2), (whole, 16), (whole, 17), (whole, -1), ([0, 19, 2], 3), ([0, -1], 2), ([1, 2], 2),
            ([0, 1, 17], 3), (whole[:5], 5), (whole[:3], 3), ([0, 16, 18], 3), (whole, 16)]


STATUS = {4: binding.SEQ_BAD_LEN, 5: binding.SEQ_BAD_LEN, 6: binding.SEQ_BAD_NODE, 7: binding.SEQ_BAD_NODE, 8: binding.SEQ_BAD_ROOT,
          9: binding.SEQ_BAD_LINK, 11: binding.SEQ_BAD_ROW}
SKIPPED, OUT_OF_RANGE = 10, 11


def _raw(c, seed, shared=None):
    rs = np.random.default_rng(seed)
    out = []
    for l in range(L):
        own = dict(a_log=rs.uniform(-1.0, 1.0, HV).astype(np.float32), dt_bias=rs.uniform(-1.0, 1.0, HV).astype(np.float32))
        out.append(dict(alpha_in=(rs.standard_normal((c.B, c.Ns, HV)) * 2 - 2).astype(np.float32),
                        beta_in=(rs.standard_normal((c.B, c.Ns, HV)) * 1.5).astype(np.float32),
                        **(own if shared is None else {k: shared[l][k] for k in own})))
    return out


@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("conv", [True, False])
@pytest.mark.parametrize("out_dtype", ["f32", "bf16"])
def test_every_kind_of_path_in_one_launch(raw, conv, out_dtype):
    paths = _paths()
    B = len(paths)
    P = W.make_case("prev", [SPINE] * B, seed=3, Hk=HK, Hv=HV, d=128, in_dtype="bf16", n_layers=L, Ns=21, permute_slots=True, with_bias=True)
    C = W.make_case("cur", [W.tree_random(W.IntStream(W.stream_key(17, b)), 30, 12) for b in range(B)], seed=4, Hk=HK, Hv=HV, d=128,
                    in_dtype="bf16", n_layers=L, Ns=34, permute_slots=True, with_bias=True)
    P.accepted = np.full((B, LMAX), -1, dtype=np.int32)
    for b, (a, n) in enumerate(paths):
        P.accepted[b, :len(a)] = a
    P.accepted_len = np.array([n for _, n in paths], dtype=np.int32)
    P.state_row[SKIPPED] = -1
    known = P.state_row.copy()                      # the oracles know skipped sequences only
    known[OUT_OF_RANGE] = -1
    P.state_row[OUT_OF_RANGE] = P.rows + 3
    C.state_row, C.rows = P.state_row.copy(), P.rows
    for p, q in zip(P.layers, C.layers):
        q.state, q.hist = p.state.copy(), p.hist.copy()
    c = ctx("tensor")
    raw_p = _raw(P, 1) if raw else None
    dcP = DeviceCase(c, P, raw_gates=raw_p)
    dcC = DeviceCase(c, C, out_dtype=out_dtype, use_conv=conv, qk_l2norm=True, raw_gates=_raw(C, 2, raw_p) if raw else None)
    dcP.verify()
    layers = []
    for l, layer in enumerate(dcC.layers):
        t = dict(layer.tensors)
        t.update(state=dcP.t("state", l), conv_hist=dcP.t("conv_hist", l), state_row=dcP.state_row)
        if raw:
            t.update(a_log=dcP.t("a_log", l), dt_bias=dcP.t("dt_bias", l))
        t["out"].fill_(float("nan"))
        layers.append(binding.GdnLayer(Hk=HK, Hv=HV, d=128, scale=dcC.scale, qk_l2norm=True, l2_eps=dcC.l2_eps, **t))
    call = lambda: c.commit_verify(dcP.desc, dcP.layers, dcP.accepted, dcP.accepted_len, dcC.desc, layers)
    assert any("scan_stream_fused_kernel" in name for name, _ in Captured(call).kernels)
    assert L * B * HV > 3 * 2 * torch.cuda.get_device_properties(0).multi_processor_count      # several states a CTA
    call()
    torch.cuda.synchronize()
    ctx("auto")
    f = lambda t: t.to(torch.float64).cpu().numpy()
    for l in range(L):
        LP, LC, tc = P.layers[l], C.layers[l], layers[l].tensors
        st1, hist1, status, _ = O.commit(P.parent, P.slot, known, dcP.np("q", l), dcP.np("k", l), dcP.np("v", l), *device_gates(dcP, l),
                                         LP.state, P.accepted, P.accepted_len, x=LP.x, hist=LP.hist, l2norm=True, eps=dcP.l2_eps)
        status[OUT_OF_RANGE] = binding.SEQ_BAD_ROW
        assert status.tolist() == [STATUS.get(b, binding.SEQ_OK) for b in range(B)]
        assert dcP.t("status", l).tolist() == status.tolist(), l
        assert tc["status"].tolist() == [binding.SEQ_BAD_ROW if b == OUT_OF_RANGE else binding.SEQ_OK for b in range(B)], l
        state = dcP.np("state", l)
        assert_close(state, st1, what=f"state, layer {l}")
        for b in range(B):
            if 0 <= known[b] and (P.accepted_len[b] == 0 or status[b]):
                assert np.array_equal(state[known[b]], LP.state[known[b]])      # bitwise as it was
        assert np.array_equal(dcP.np("conv_hist", l), hist1), l
        if conv:
            y = O.conv(C.parent, C.slot, known, LC.x, LC.conv_w, LC.conv_b, hist1, C.Ns, out_dtype="none")
            got = np.concatenate([f(tc[n]).reshape(B, C.Ns, -1) for n in ("q", "k", "v")], axis=-1)
            assert_close(got, y, bf16=True, what=f"recorded operands, layer {l}")
        ref, _, _ = O.scan(C.parent, C.slot, known, f(tc["q"]), f(tc["k"]), f(tc["v"]), *device_gates(dcC, l), st1, l2norm=True, eps=dcC.l2_eps)
        worst = assert_close(f(tc["out"]), ref, bf16=out_dtype == "bf16", what=f"outputs, layer {l}")
        assert out_dtype == "bf16" or worst < BOUND
