"""The batch's Algorithm 3 passes by the form of the rows: n columns off the 16-byte grid (word
copies) and the same matrix with zero columns up to a multiple of four (16-byte copies) sum the same
terms in the same order, and a zero column is never picked: the same indices come back. The row
counts leave last stages of one and two rows and row groups without a row."""
import ctypes

import pytest
import torch

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu


def _run(mats, r):
    offs, o = [], 0
    for a in mats:
        offs.append(o)
        o += a.numel()
    items = cur.batch_items([(a.shape[0], a.shape[1], r, 1, 1) for a in mats], offs)
    data = torch.cat([a.reshape(-1) for a in mats])
    IJ = torch.full((2 * r * len(mats),), -7, dtype=torch.int32, device="cuda")
    info = torch.zeros(len(mats) * ctypes.sizeof(cur.CurCrossInfo), dtype=torch.uint8, device="cuda")
    with cur.Handle(1, 1, 1, workspace_bytes=cur.cur_batch_workspace_size(items)) as hd:
        cur.cur_cross_batched(hd.h, data, items, cur.opts(1e-2), IJ, info)
        return cur.cur_sync_status(hd.h), IJ.tolist()


@pytest.mark.parametrize("n,r", [(131, 9), (1023, 17), (514, 33), (35, 8), (997, 64), (6, 5)])
def test_row_forms_pick_the_same(n, r):
    g = torch.Generator(device="cuda").manual_seed(n)
    odd, full = [], []
    for m in (257, 1030, 66, 2049, 513):
        a = torch.randn((m, n), generator=g, device="cuda") * (1.0 + torch.rand(n, generator=g, device="cuda"))
        z = torch.zeros((m, -(-n // 4) * 4), device="cuda")
        z[:, :n] = a
        odd.append(a)
        full.append(z)
    got = [_run(x, r) for x in (odd, full)]
    assert got[0] == got[1] and got[0][0] == cur.CUR_OK
    assert min(got[0][1]) >= 0
