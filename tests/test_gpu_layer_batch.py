"""The layer batch that a launch hands to the driver holds the call's layers and zeros, whatever the calls before it left on the stack."""
import pytest
import torch

from synthetic import workload as W
from synthetic.device_case import DeviceCase
from tests.graph_nodes import Captured
from tests.harness import ctx

pytestmark = pytest.mark.gpu

_LAYER = 17 * 8           # LayerPtrs: seventeen pointers
_BATCH = 2                # conv_kernel(Shape, TreeDev, layers, ...)


@pytest.mark.parametrize("n,entries", [(1, 4), (4, 4), (5, 64), (64, 64)])
def test_entries_beyond_the_calls_layers_are_zero(n, entries):
    dc = DeviceCase(ctx("auto"), W.make_case("batch", [W.tree_chain(3)], seed=1, Hk=1, Hv=1, d=128, in_dtype="bf16", n_layers=64))
    dc.verify()                                                       # the largest batch has been on the stack
    torch.cuda.synchronize()
    got = Captured(lambda: dc.ctx.verify(dc.desc, dc.layers[:n])).argument("conv_kernel", _BATCH, entries * _LAYER)
    used, rest = got[:n * _LAYER], got[n * _LAYER:]
    assert int.from_bytes(used[:8], "little") == dc.t("q").data_ptr()
    assert rest == bytes(len(rest))
