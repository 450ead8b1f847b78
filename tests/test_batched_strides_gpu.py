"""The batch's Algorithm 3 passes on matrices with padded rows (ld > cols). The rows come through
shared memory by bulk copies of whole 16-byte lines, padding and all, a slot of as many rows as it
holds for every row group; where a slot holds fewer, they are loaded directly. Each thread sums the
same rows in the same order either way, so the crosses have to be those of the same matrices
packed. The padding is NaN, offsets are off the 16-byte grid, and the batch ends with its last
matrix's last entry."""
import ctypes

import pytest
import torch

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu


def _run(data, offs, lds, shapes):
    items = (cur.CurBatchItem * len(shapes))()
    for t, (m, n, r) in enumerate(shapes):
        items[t] = cur.CurBatchItem(offs[t], m, n, lds[t], r, 1, 1)
    IJ = torch.full((2 * sum(s[2] for s in shapes),), -7, dtype=torch.int32, device="cuda")
    info = torch.zeros(len(shapes) * ctypes.sizeof(cur.CurCrossInfo), dtype=torch.uint8, device="cuda")
    with cur.Handle(1, 1, 1, workspace_bytes=cur.cur_batch_workspace_size(items)) as hd:
        cur.cur_cross_batched(hd.h, data, items, cur.opts(1e-2), IJ, info)
        return cur.cur_sync_status(hd.h), IJ.tolist()


@pytest.mark.parametrize("shapes,lds", [
    ([(257, 131, 9), (1030, 64, 17), (2049, 514, 33), (513, 997, 40)], [133, 66, 515, 1001]),   # bulk copies
    ([(300, 1023, 17), (66, 35, 8), (801, 200, 21)], [5000, 4099, 4097]),                       # no row fits a slot
    ([(513, 35, 8), (130, 6, 5), (2050, 131, 9)], [100, 64, 1025]),                             # fewer rows than groups
    ([(2, 2, 1), (4, 900, 3), (4096, 64, 12)], [7, 903, 80]),
])
def test_padded_rows_give_the_packed_crosses(shapes, lds):
    g = torch.Generator(device="cuda").manual_seed(lds[0])
    mats = [torch.randn((m, n), generator=g, device="cuda") * (1.0 + torch.rand(n, generator=g, device="cuda")) for m, n, _ in shapes]
    offs, o = [], 0
    for a in mats:
        offs.append(o)
        o += a.numel()
    want = _run(torch.cat([a.reshape(-1) for a in mats]), offs, [n for _, n, _ in shapes], shapes)
    offs, o = [], 1
    for (m, n, _), ld in zip(shapes, lds):
        offs.append(o)
        o += (m - 1) * ld + n
    data = torch.full((o,), float("nan"), device="cuda")
    for a, off, ld in zip(mats, offs, lds):
        data.as_strided(a.shape, (ld, 1), off).copy_(a)
    got = _run(data, offs, lds, shapes)
    assert got == want and got[0] == cur.CUR_OK
