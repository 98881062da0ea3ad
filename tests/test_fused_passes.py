"""Two-pass plans that run as one launch, and rows that share one: which plans
do, and that the launch moves every element as the two passes, or the launches
row by row, do."""

import gc
import weakref

import pytest

import oracle
from oracle import f2
import paper_2306_07795_gb300 as bm
from paper_2306_07795_gb300.autograd import _lifted_plan
import workloads as wl


def _inv(rows):
    return f2.is_invertible(rows, len(rows))


def _dense(n, seed):
    return wl.dense_bmmc(n, seed, _inv)


@pytest.mark.parametrize("e,n", [(4, 15), (4, 20), (8, 14), (8, 19), (16, 13), (16, 18)])
def test_rule(e, n):
    """Default segments: one launch, whose tables are walked with the passes';
    chosen segments: the two passes as asked; both keep the two matrices."""
    rows, c = _dense(n, n + e)
    for kw in ({}, {"cta_tile_log2": 12}, {"cta_tile_log2": 16, "tile_order": 2},
               {"flags": bm.BMMC_PLAN_TMA_LOAD}):
        p = bm.Plan(n, rows, c, e, **kw)
        assert (p.num_passes, p.num_launches) == (2, 1)
        assert p.workspace_bytes == p.nbytes
        assert p.verify() == 0
        d = p.describe()
        assert d["launches"] == 1 and len(d["passes"]) == 2 and "fused" in d
    q = bm.Plan(n, rows, c, e, seg_bits=8 - (e.bit_length() - 1))
    assert (q.num_passes, q.num_launches) == (2, 2)
    assert q.pass_matrices() == p.pass_matrices()
    assert q.verify() == 0


def test_batch_workspace():
    """Only plans of two launches have a slice of a batch's workspace."""
    rows, c = _dense(18, 2)
    one = [bm.Plan(18, rows, c, 4), bm.Plan(18, wl.bit_reverse(18), 0, 4),
           bm.Plan(18, rows, c, 8, flags=bm.BMMC_PLAN_SINGLE_PASS)]
    two = bm.Plan(18, rows, c, 4, seg_bits=6)
    assert bm.bmmc_batch_workspace_bytes([p.handle for p in one]) == 0
    assert bm.bmmc_batch_workspace_bytes([p.handle for p in one + [two]]) == two.nbytes


def test_lifted_plans_go_with_their_plan():
    """A program that makes a plan per call keeps none of their lifted forms."""
    rows, c = _dense(10, 4)
    p = bm.Plan(10, rows, c, 4)
    lifted = _lifted_plan(p, 3)
    assert lifted is _lifted_plan(p, 3) and lifted.n == 13
    refs = [weakref.ref(p), weakref.ref(lifted)]
    del p, lifted
    gc.collect()
    assert [r() for r in refs] == [None, None]


@pytest.mark.gpu
@pytest.mark.parametrize("e,n", [(4, 15), (4, 22), (8, 14), (8, 20), (16, 13), (16, 19)])
def test_direct_equals_workspace_form(e, n):
    import torch
    rows, c = _dense(n, 3 * n + e)
    x = wl.payload_torch(n, e, seed=n)
    p = bm.Plan(n, rows, c, e)
    q = bm.Plan(n, rows, c, e, seg_bits=8 - (e.bit_length() - 1))  # two launches
    a, b = torch.full_like(x, -1), torch.full_like(x, -1)
    s = torch.cuda.current_stream().cuda_stream
    bm.bmmc_execute_direct(p.handle, x.data_ptr(), a.data_ptr(), 1, s)
    q(x, out=b)
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    assert oracle.count_mismatch(n, rows, c, x.cpu().numpy(), a.cpu().numpy(), elem_bytes=e) == 0
    for h, i, o, code in ((q.handle, x, a, bm.BMMC_ERR_INVALID),
                          (p.handle, x, x, bm.BMMC_ERR_ALIAS)):
        with pytest.raises(bm.BmmcError) as ei:
            bm.bmmc_execute_direct(h, i.data_ptr(), o.data_ptr(), 1, s)
        assert ei.value.code == code
    with pytest.raises(bm.BmmcError) as ei:
        bm.bmmc_execute_ws(p.handle, x.data_ptr(), a.data_ptr(), None, s)
    assert ei.value.code == bm.BMMC_ERR_INVALID  # a workspace is still asked for here


@pytest.mark.gpu
@pytest.mark.parametrize("e,n,rows", [(4, 2, 7), (4, 5, 3), (4, 8, 65537), (4, 10, 1), (4, 13, 6),
                                      (8, 1, 5), (8, 16, 24), (16, 3, 9), (16, 14, 3)])
@pytest.mark.parametrize("flags", [0, bm.BMMC_PLAN_TMA_LOAD])
def test_rows_share_a_launch(e, n, rows, flags):
    """Every row as alone: arrays below and above 1 KiB, more rows than one
    grid holds, tensor-copy loads (a launch per row)."""
    import torch
    if flags and rows > 100:
        rows = 101
    mat, c = _dense(n, n + rows)
    p = bm.Plan(n, mat, c, e, flags=flags)
    x = torch.randint(-2**31, 2**31 - 1, (rows, p.nbytes // 4), dtype=torch.int32, device="cuda")
    y = p.run_rows(x, rows)
    at = torch.from_numpy(f2.index_table(n, mat, c).astype("int64")).cuda()
    want = torch.empty_like(x).view(rows, 1 << n, -1)
    want[:, at] = x.view(rows, 1 << n, -1)
    torch.cuda.synchronize()
    assert torch.equal(y, want.view_as(y))


@pytest.mark.gpu
def test_rows_refused():
    import torch
    x = torch.zeros(3 * 2, dtype=torch.int32, device="cuda")
    p = bm.Plan(1, [1], 1, 4)  # rows of 8 bytes do not start on 16-byte boundaries
    with pytest.raises(bm.BmmcError) as ei:
        p.run_rows(x, 3)
    assert ei.value.code == bm.BMMC_ERR_ALIGN
    with pytest.raises(bm.BmmcError) as ei:
        bm.bmmc_execute_direct(p.handle, x.data_ptr(), x.data_ptr(), 0, 0)
    assert ei.value.code == bm.BMMC_ERR_INVALID
