"""Draft selection around its short list of candidate entries: rows with as many entries at the bound as the list holds, one
more, and a whole row of them; ties that many threads or very few hold; rows too short to give three threads an entry; the edge of the automatic split."""
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


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("threads", [1, 2, 3, 40])
def test_hundreds_of_ties_in_the_hands_of_few_threads(threads, dtype):
    """One CTA a row: the units of `threads` of its 512 threads hold the maximum 296 times each, more than the list takes."""
    V, n = 151936, 128 // torch.finfo(dtype).bits
    rs = np.random.default_rng(threads)
    x = (rs.standard_normal((3, V)) - 8).astype(np.float32)
    owner = (np.arange(V) // n) % 512
    for r in range(3):
        x[r, np.isin(owner, rs.choice(512, threads, replace=False))] = 1.5
    x[1, rs.integers(V)] = 2.0                     # a single larger entry above the ties
    x[2, rs.choice(V, 2, replace=False)] = 2.0     # two of them
    check(x, dtype, 1)
    check(x, dtype, 0)


def device_us(x, split=0):
    """Time of one call, from a graph of twenty."""
    spine, cand = torch.zeros(x.shape[0], dtype=torch.int32, device="cuda"), torch.zeros(x.shape[0], 3, dtype=torch.int32, device="cuda")
    c = ctx()
    c.select_spine_top3(x, spine, cand, split=split)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(20):
            c.select_spine_top3(x, spine, cand, split=split)
    us = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(); g.replay(); b.record()
        torch.cuda.synchronize()
        us.append(1e3 * a.elapsed_time(b) / 20)
    return sorted(us)[4]


@pytest.mark.parametrize("fill", [0.5, -float("inf")])
def test_a_constant_row_takes_a_second_pass_and_no_more(fill):
    """A row of equal entries is read twice and ends in a few reductions: 2.1 times a plain row's time, measured; visiting one
    thread's entries after the other took 10 times.  The bound lies between the two."""
    plain = torch.randn(8, 151936, device="cuda").to(torch.bfloat16)
    assert device_us(torch.full_like(plain, fill)) < 5 * device_us(plain)
