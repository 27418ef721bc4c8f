"""Automatic partitioning of short contexts: units that stay whole (their outputs leave the attention kernel as final results),
the edge where the longest is cut after all, sequences that are refused in between, and masks whose 64-key windows start and
end anywhere in the suffix; against the oracle."""
import numpy as np
import pytest
import torch

from paper_2609_23900_b200 import binding
from synthetic import workload as W
from synthetic.device_case import DeviceAttnCase
from tests.harness import ctx
from tests.test_gpu_attn import check_attention, oracle_caches, trees

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,N,Ns,Hq,Hkv,ctxs", [
    ("random", 9, 16, 4, 2, [0, 1, 63]),
    ("random", 20, 40, 8, 2, [100, 129, 250]),           # suffix across a tile edge
    ("star", 150, 250, 4, 2, [5, 77]),                   # windows in the middle of the suffix, three row tiles
    ("random", 12, 12, 4, 4, [1000, 20, 1023]),          # whole: eight tiles, shares of four
    ("random", 12, 12, 4, 4, [1024, 20, 1200]),          # longer than a share by more than the slack: cut
    ("chain", 64, 64, 2, 1, [127]),
])
def test_whole_units(kind, N, Ns, Hq, Hkv, ctxs):
    c = W.make_attn_case("whole", trees(kind, len(ctxs), N, 77), ctxs, seed=W.BASE_SEED + 60, Hq=Hq, Hkv=Hkv, Ns=Ns, layout="permuted")
    dc = DeviceAttnCase(ctx(), c)
    dc.write()
    dc.attend()
    torch.cuda.synchronize()
    check_attention(dc, c, *oracle_caches(c), what=str(ctxs))


def test_refused_sequence_among_whole_units():
    c = W.make_attn_case("refused", trees("random", 3, 10, 5), [40, 50, 60], seed=W.BASE_SEED + 61, Hq=4, Hkv=2, layout="permuted")
    dc = DeviceAttnCase(ctx(), c)
    dc.cache_row[1] = 99
    dc.write()
    dc.attend()
    torch.cuda.synchronize()
    assert dc.t("status").tolist() == [0, binding.SEQ_BAD_ROW, 0]
    assert np.all(dc.np("out")[1] == 0) and np.all(dc.np("lse")[1] == 0)
    good = DeviceAttnCase(ctx(), c)
    good.write()
    good.attend()
    torch.cuda.synchronize()
    for b in (0, 2):
        assert np.array_equal(dc.np("out")[b], good.np("out")[b])
