"""A round's pick and direction by one cluster (small work) and by the whole grid: zero rows (or
columns) appended to the vectors change no sum but take the same selection past the line
between the two, so the picks, their number and the status have to be the same."""
import pytest
import torch

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu
CODE = {torch.float32: cur.CUR_F32, torch.float64: cur.CUR_F64, torch.bfloat16: cur.CUR_BF16}


def _select(A, axis, r):
    idx = torch.full((r,), -7, dtype=torch.int32, device="cuda")
    with cur.Handle(A.shape[0], A.shape[1], r, CODE[A.dtype]) as hd:
        cur.cur_aca_select(hd.h, A, axis, r, 1, idx)
        return cur.cur_sync_status(hd.h), idx.tolist()


@pytest.mark.parametrize("axis", [1, 0])
@pytest.mark.parametrize("length,count,r,rank,dtype", [
    (4096, 515, 64, 64, torch.float32),      # the largest work of a cluster; uneven shares of the columns
    (2048, 130, 128, 128, torch.float32), (3001, 2011, 33, 33, torch.float32),
    (3, 5, 3, 3, torch.float32), (7, 3, 3, 3, torch.float64), (2049, 257, 47, 47, torch.float64),
    (1500, 301, 40, 12, torch.float64),      # the early stop, in the middle of the rounds
    (700, 1030, 65, 65, torch.bfloat16),
])
def test_cluster_and_grid_pick_the_same(length, count, r, rank, dtype, axis):
    assert length * r <= 1 << 18
    g = torch.Generator(device="cuda").manual_seed(length + count)
    V = torch.randn((length, rank), generator=g, device="cuda", dtype=torch.float64)
    V = V @ torch.randn((rank, count), generator=g, device="cuda", dtype=torch.float64) if rank < r else \
        torch.randn((length, count), generator=g, device="cuda", dtype=torch.float64)
    V = (V * (1.0 + torch.rand(count, generator=g, device="cuda", dtype=torch.float64))).to(dtype)
    long = torch.zeros(((1 << 18) // r + 1, count), dtype=dtype, device="cuda")
    long[:length] = V
    got = [_select(x.t().contiguous() if axis == 0 else x, axis, r) for x in (V, long)]
    assert got[0] == got[1]
    assert got[0][0] == (cur.CUR_WARN_RANK if rank < r else cur.CUR_OK)
    assert len({i for i in got[0][1] if i >= 0}) == min(r, rank)
    assert got[0][1][0] == int(V.double().square().sum(0).argmax())
