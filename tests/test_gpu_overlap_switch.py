"""The overlap switch covers every call: with it off no captured kernel depends on the one before it programmatically."""
import pytest
import torch

from synthetic import workload as W
from synthetic.device_case import DeviceAttnCase, DeviceCase
from tests.graph_nodes import Captured
from tests.harness import ctx

pytestmark = pytest.mark.gpu


def calls():
    """One call of every kind, each enqueued twice in a row where it is a single kernel."""
    c = ctx("auto")
    g = W.config_paper(B=2)
    dg = DeviceCase(c, g, out_dtype="bf16")
    a = W.make_attn_case("switch", [p.tolist() for p in g.parent], [300, 45], seed=5, Hq=8, Hkv=2, Ns=g.Ns)
    da = DeviceAttnCase(c, a, n_splits=0)
    B, V, lmax = g.B, 512, 16
    i32 = lambda *s: torch.zeros(*s, dtype=torch.int32, device="cuda")
    acc, ln, nxt, fin, node, tok = i32(B, lmax), i32(B), i32(B), i32(B), i32(B), i32(B, g.Ns)
    p = torch.rand(B, g.Ns + 1, V, device="cuda")
    logits, spine, cand = torch.rand(4, V, device="cuda"), i32(4), i32(4, 3)
    twice = lambda f: lambda: (f(), f())
    return {
        "path": twice(lambda: c.path_from_node(dg.desc, node, lmax, acc, ln)),
        "accept": twice(lambda: c.accept(dg.desc, token=tok, p_target=p, accepted=acc, length=ln, next_token=nxt, final_node=fin)),
        "select": twice(lambda: c.select_spine_top3(logits, spine, cand)),
        "kv_write": twice(lambda: c.kv_write_tree(da.desc, da.packed)),
        "attention": lambda: c.tree_attention(da.desc, da.packed),
        "kv_publish": twice(lambda: c.kv_publish(da.desc, da.packed, acc, ln)),
        "verify": lambda: c.verify(dg.desc, dg.layers),
        "commit": lambda: (c.verify(dg.desc, dg.layers), c.commit(dg.desc, dg.layers, acc, ln)),
    }


@pytest.mark.parametrize("kind", ["path", "accept", "select", "kv_write", "attention", "kv_publish", "verify", "commit"])
def test_off_means_plain_stream_order(kind):
    call = calls()[kind]
    try:
        call()                                   # sizes the scratch
        torch.cuda.synchronize()
        ctx("auto").set_overlap(False)
        off = Captured(call)
        ctx("auto").set_overlap(True)
        on = Captured(call)
    finally:
        ctx("auto").set_overlap(True)
    assert len(off.kernels) == len(on.kernels) >= 2
    assert off.programmatic() == 0
    assert on.programmatic() == len(on.kernels) - 1
