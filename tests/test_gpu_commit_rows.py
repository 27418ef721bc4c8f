"""The commit's split into rows per CTA (32 rows in launches of up to one wave, whole heads beyond) and its staging of
eight accepted nodes at a time: path lengths on both sides of every edge, against the oracle."""
import numpy as np
import pytest
import torch

from synthetic import workload as W
from synthetic.device_case import DeviceCase
from tests.harness import assert_close, ctx, oracle_commit_from_device

pytestmark = pytest.mark.gpu

LENGTHS = [1, 7, 8, 9, 16, 17, 24, 0]


@pytest.mark.parametrize("d,dtype,Hv,n_layers", [(64, "f32", 2, 1), (64, "bf16", 6, 48), (128, "f32", 4, 1), (128, "bf16", 4, 1),
                                                 (128, "bf16", 12, 5), (128, "f32", 12, 5)])
def test_commit_rows_and_path_lengths(d, dtype, Hv, n_layers):
    c = W.make_case("rows", [W.tree_chain(24)] * len(LENGTHS), seed=21, Hk=2, Hv=Hv, d=d, in_dtype=dtype, n_layers=n_layers,
                    accepted=[list(range(n)) for n in LENGTHS], lmax=24, Ns=27, permute_slots=True)
    dc = DeviceCase(ctx(), c)
    dc.verify()
    dc.commit()
    torch.cuda.synchronize()
    for l in sorted({0, n_layers - 1}):
        st_ref, hist_ref, status, _ = oracle_commit_from_device(dc, layer=l)
        assert dc.np("status", l).tolist() == status.tolist() == [0] * c.B
        assert_close(dc.np("state", l), st_ref, what=f"d {d} {dtype}, layer {l}")
        assert np.array_equal(dc.np("conv_hist", l), hist_ref)
