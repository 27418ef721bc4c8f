"""Two contexts on one stream: what one of them writes is not read early by the other."""
import struct

import pytest
import torch

from paper_2609_23900_b200 import binding
from synthetic import workload as W
from synthetic.device_case import DeviceCase
from tests.graph_nodes import Captured
from tests.harness import ctx

pytestmark = pytest.mark.gpu

_WAIT_FIRST = 19          # place of Shape::wait_first among the 4-byte members of a commit's first argument


def setup():
    a, b = ctx("auto"), binding.Context(0)
    c = W.config2()
    dc = DeviceCase(a, c)
    desc_b = b.tree_desc(c.parent, slot=c.slot, n_slots=c.Ns)
    B, V, lmax = c.B, 4096, 16
    i32 = lambda *s: torch.zeros(*s, dtype=torch.int32, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(3)
    tok = torch.randint(0, V, (B, c.Ns), dtype=torch.int32, device="cuda", generator=g)
    p = torch.rand(B, c.Ns + 1, V, device="cuda", generator=g)
    for i in range(B):                                   # the favourite after every row is the token of some child
        for n, par in enumerate(c.parent[i].tolist()):
            row = c.Ns if par < 0 else int(c.slot[i, par])
            p[i, row, tok[i, int(c.slot[i, n])].long()] += 1.0
    out = dict(accepted=i32(B, lmax), length=i32(B), next_token=i32(B), final_node=i32(B))
    walk = {who: (lambda who=who, d=d: who.accept(d, token=tok, p_target=p, **out)) for who, d in ((a, dc.desc), (b, desc_b))}
    commit = lambda: a.commit(dc.desc, dc.layers, out["accepted"], out["length"])
    return a, b, dc, desc_b, out, walk, commit


def test_a_commit_behind_another_contexts_call_waits_first():
    a, b, dc, desc_b, out, walk, commit = setup()
    node = torch.zeros(dc.case.B, dtype=torch.int32, device="cuda")
    early = lambda call: struct.unpack_from("i", Captured(call).argument("commit_kernel", 0, 80), 4 * _WAIT_FIRST)[0] == 0
    dc.verify(); walk[a](); walk[b](); commit()          # sizes the scratch
    torch.cuda.synchronize()
    assert early(lambda: (dc.verify(), commit()))        # a small commit right behind its own verify does read ahead
    assert not early(lambda: (dc.verify(), walk[a](), commit()))
    assert not early(lambda: (dc.verify(), walk[b](), commit()))
    assert not early(lambda: (dc.verify(), b.path_from_node(desc_b, node, 16, out["accepted"], out["length"]), commit()))


def test_cycles_of_two_contexts_match_plain_stream_order():
    res = {}
    for on in (False, True):
        a, b, dc, desc_b, out, walk, commit = setup()
        for cx in (a, b):
            cx.set_overlap(on)
        outs = []
        for _ in range(8):
            out["accepted"].fill_(-1); out["length"].zero_()
            dc.verify(); walk[b](); commit()
            outs += [dc.t("out").clone(), out["length"].clone()]
        torch.cuda.synchronize()
        res[on] = outs + [dc.t("state").clone(), dc.t("conv_hist").clone()]
        assert int(out["length"].min()) > 0
    ctx("auto").set_overlap(True)
    assert all(torch.equal(x, y) for x, y in zip(res[False], res[True]))


def test_a_scan_behind_another_contexts_commit_takes_stream_order():
    a, b = ctx("auto"), binding.Context(0)
    c = W.config2()
    da, db = DeviceCase(a, c, use_conv=False, qk_l2norm=True), DeviceCase(b, c, use_conv=False, qk_l2norm=True)
    da.verify(); db.verify(); db.commit()
    torch.cuda.synchronize()
    assert Captured(lambda: (da.verify(), da.verify())).programmatic() == 1
    alone, behind = Captured(lambda: (db.verify(), db.commit())), Captured(lambda: (db.verify(), db.commit(), da.verify()))
    assert behind.programmatic() == alone.programmatic() == 1
