"""Draft selection around its short list of candidate entries: rows with as many entries at the bound as the list holds, one
more, and a whole row of them; rows too short to give three threads an entry; the edge of the automatic split."""
import numpy as np
import pytest
import torch

from oracle import select_oracle as S
from tests.harness import ctx

pytestmark = pytest.mark.gpu


def check(x, dtype, split):
    t = torch.from_numpy(x).to(dtype)
    d = t.cuda()
    spine = torch.full((x.shape[0],), -7, dtype=torch.int32, device="cuda")
    cand = torch.full((x.shape[0], 3), -7, dtype=torch.int32, device="cuda")
    ctx().select_spine_top3(d, spine, cand, split=split)
    ref = S.select(t.to(torch.float64).numpy())
    assert spine.cpu().numpy().tobytes() == ref[0].tobytes()
    assert cand.cpu().numpy().tobytes() == ref[1].tobytes()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V,split", [(3, 0), (4, 1), (9, 2), (1025, 0), (32768, 0), (32769, 1), (65537, 4)])
def test_ties_at_the_bound(V, split, dtype):
    rs = np.random.default_rng(V)
    ties = [1, 2, 3, 32, 33, 255, 256, 257, 300, V]
    x = (rs.standard_normal((len(ties) + 2, V)) - 8).astype(np.float32)
    for r, n in enumerate(ties):
        x[r, rs.choice(V, size=min(n, V), replace=False)] = 1.5          # the row's maximum, n times
    x[-2] = -np.inf
    x[-1, :] = -np.inf
    x[-1, V // 2] = -3.0                                                  # a single finite entry
    check(x, dtype, split)
