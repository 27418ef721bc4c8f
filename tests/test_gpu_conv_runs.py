"""The tree convolution's split of a sequence into runs (one warp each) and parts (one CTA each): node counts on both sides of
every edge, windows that reach back into another part, channel counts that do not fill a CTA's groups, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import gdn_oracle as O
from synthetic import workload as W
from synthetic.device_case import DeviceCase
from tests.harness import assert_close, ctx

pytestmark = pytest.mark.gpu


def check(c):
    dc = DeviceCase(ctx(), c)
    for t in ("q", "k", "v"):
        dc.t(t).fill_(777.0)     # must be overwritten everywhere, padding rows with zeros
    dc.verify()
    torch.cuda.synchronize()
    L, hk = c.layers[0], c.Hk * c.d
    y = O.conv(c.parent, c.slot, c.state_row, L.x, L.conv_w, L.conv_b, L.hist, c.Ns, out_dtype="none")
    got = np.concatenate([dc.np("q").reshape(c.B, c.Ns, hk), dc.np("k").reshape(c.B, c.Ns, hk), dc.np("v").reshape(c.B, c.Ns, c.Hv * c.d)], axis=-1)
    assert_close(got, y, bf16=(c.in_dtype == "bf16"), what="conv")


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("N", [1, 4, 5, 8, 9, 17, 33, 65, 129, 256])
def test_runs_and_parts(N, dtype):
    depth = 3 if N < 5 else 12
    rand = W.tree_random(W.IntStream(N), N, depth) if N > 1 else [-1]
    chain = [i - 1 for i in range(N)]
    check(W.make_case("runs", [rand, chain], seed=N, Hk=1, Hv=1, d=64, in_dtype=dtype, Ns=N + 3, permute_slots=True, with_bias=True))


@pytest.mark.parametrize("B,N", [(8, 64), (24, 40), (32, 28), (12, 200)])
def test_longer_runs_of_large_launches(B, N):
    check(W.make_case("runs", [W.tree_random(W.IntStream(N + b), N, 9) for b in range(B)], seed=B, Hk=3, Hv=6, d=128, in_dtype="bf16"))


@pytest.mark.parametrize("B,N", [(12, 41), (14, 33)])
def test_runs_shared_out_evenly(B, N):
    """More CTAs than run at once: eleven runs as six and five, nine as five and four."""
    assert ctx().conv_rows_per_cta(ctx().tree_desc(np.array([[i - 1 for i in range(N)]] * B, dtype=np.int32)), 8, 16, 128) == 4
    check(W.make_case("runs", [W.tree_random(W.IntStream(N + b), N, 9) for b in range(B)], seed=B, Hk=8, Hv=16, d=128, in_dtype="bf16",
                      Ns=N, permute_slots=True))


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("N", [130, 256])
def test_windows_shared_across_parts(N, dtype):
    """The second part's first entry hangs off a node of the first part: the root of a star (two history rows and one staged), a spine of
    four whose last three nodes all have children there (windows that are the first entry's own, and others one and two rows older)."""
    star = [-1] + [0] * (N - 1)
    spine = [-1, 0, 1, 2] + [3] * (N - 24) + [2] * 10 + [1] * 10
    check(W.make_case("shared", [star, spine], seed=N, Hk=1, Hv=2, d=64, in_dtype=dtype, Ns=N + 2, permute_slots=True, with_bias=True))
