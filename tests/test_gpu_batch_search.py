"""The batch kernel's search for an item's array: counts of arrays around the
256 that one look takes, arrays of one item between arrays of many; and its
chunks, at the shares of a block where their size changes."""

import random

import numpy as np
import pytest

import oracle
import paper_2306_07795_gb300 as bm
import workloads as wl
from oracle import f2
from paper_2306_07795_gb300.batch import Batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,hi", [(1, 16), (2, 16), (3, 18), (255, 13), (256, 13), (257, 13),
                                      (700, 12), (66000, 3)])
def test_every_array(count, hi):
    import torch
    r = random.Random(count)
    sizes = [r.choice((1, 3, hi)) if i % 7 else hi for i in range(count)]
    perms, plans = {}, {}
    for n in sorted(set(sizes)):
        perms[n] = wl.dense_bmmc(n, n, lambda a: f2.is_invertible(a, n))
        plans[n] = bm.Plan(n, perms[n][0], perms[n][1], 4)
    x = torch.randint(-2**31, 2**31 - 1, (sum(max(4, 1 << n) for n in sizes),), dtype=torch.int32,
                      device="cuda")
    out = torch.zeros_like(x)
    ins, outs, at = [], [], 0
    for n in sizes:
        ins.append(x[at:at + (1 << n)])
        outs.append(out[at:at + (1 << n)])
        at += max(4, 1 << n)
    b = Batch([plans[n] for n in sizes], ins, outs)
    for _ in range(2):  # the claim counters start over
        out.zero_()
        b()
    torch.cuda.synchronize()
    got, src, at = out.cpu().numpy(), x.cpu().numpy(), 0
    for n in sizes:
        want = oracle.apply(n, *perms[n], src[at:at + (1 << n)])
        assert np.array_equal(got[at:at + (1 << n)].view(np.uint32), want.view(np.uint32)), (at, n)
        at += max(4, 1 << n)


@pytest.mark.parametrize("share", [1, 5, 12, 13, 47, 48])
def test_chunks(share):
    """One chunk a block up to a share of 12 items, 4 items up to 48, then 8.  The
    last array stops one item short of the share."""
    import torch
    n = 13  # two items each
    rows, c = wl.dense_bmmc(n, 5, lambda a: f2.is_invertible(a, n))
    plan = bm.Plan(n, rows, c, 4)
    one = torch.randint(-2**31, 2**31 - 1, (1 << n,), dtype=torch.int32, device="cuda")

    def batch(count):
        x = one.repeat(count).view(count, -1)
        out = torch.zeros_like(x)
        return Batch([plan] * count, list(x), list(out)), x, out

    b, _, _ = batch(4096)
    grid, items = (b.describe()["launches"][0][k] for k in ("grid", "items"))
    assert items == 2 * 4096 and grid < items
    b, x, out = batch((grid * share - 1) // 2)
    d = b.describe()["launches"][0]
    assert d["grid"] == min(grid, d["items"]) and -(-d["items"] // d["grid"]) == share
    assert d["chunk"] == (share if share <= 12 else 4 if share < 48 else 8)
    x += torch.arange(x.shape[0], dtype=torch.int32, device="cuda")[:, None]
    for _ in range(2):
        out.zero_()
        b()
    torch.cuda.synchronize()
    at = torch.from_numpy(f2.index_table(n, rows, c).astype(np.int64)).cuda()
    want = torch.empty_like(x)
    want[:, at] = x
    assert torch.equal(out, want)
