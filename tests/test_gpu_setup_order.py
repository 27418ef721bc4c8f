"""A descriptor used at once on a stream that does not wait for the default stream: its tables have arrived when it is returned."""
import pytest
import torch

from synthetic import workload as W
from synthetic.device_case import DeviceCase
from tests.harness import ctx

pytestmark = pytest.mark.gpu


def test_fresh_descriptor_on_a_side_stream():
    c = ctx("auto")
    dc = DeviceCase(c, W.config4("random", B=4))
    dc.verify()
    torch.cuda.synchronize()
    want, side = dc.t("out").clone(), torch.cuda.Stream()
    for _ in range(10):
        dc.t("out").fill_(float("nan"))
        torch.cuda.synchronize()
        desc = c.tree_desc(dc.case.parent, slot=dc.case.slot, n_slots=dc.case.Ns)
        c.verify(desc, dc.layers, stream=side)
        torch.cuda.synchronize()
        assert torch.equal(dc.t("out"), want)
