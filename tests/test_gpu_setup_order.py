"""A descriptor used at once on a stream that does not wait for the default stream: its tables have arrived when it is returned,
and neither waits for what the default stream has to do."""
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
    want, side, kept = dc.t("out").clone(), torch.cuda.Stream(), []     # (freeing a descriptor waits for the device)
    for _ in range(5):
        dc.t("out").fill_(float("nan"))
        torch.cuda.synchronize()
        torch.cuda._sleep(40_000_000)            # the default stream is busy for some twenty milliseconds
        desc = c.tree_desc(dc.case.parent, slot=dc.case.slot, n_slots=dc.case.Ns)
        kept.append(desc)
        c.verify(desc, dc.layers, stream=side)
        side.synchronize()
        assert not torch.cuda.default_stream().query()
        torch.cuda.synchronize()
        assert torch.equal(dc.t("out"), want)
