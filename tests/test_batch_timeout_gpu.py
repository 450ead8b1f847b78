"""A batch whose Algorithm 3 waits run out (its copies withheld by the self-test): the call records
CUR_ERR_TIMEOUT, every matrix still gets sets of distinct indices within it, the matrices that another
CTA took are as without the fault, and the handle goes on."""
import ctypes

import pytest
import torch

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu


def _setup(shapes):
    g = torch.Generator(device="cuda").manual_seed(len(shapes))
    offs, o = [], 0
    for m, n, *_ in shapes:
        offs.append(o)
        o += m * n
    data = torch.randn(o, generator=g, device="cuda")
    return data, cur.batch_items(shapes, offs)


def _run(hd, data, items, shapes):
    IJ = torch.full((2 * sum(s[2] for s in shapes),), -7, dtype=torch.int32, device="cuda")
    info = torch.zeros(len(shapes) * ctypes.sizeof(cur.CurCrossInfo), dtype=torch.uint8, device="cuda")
    cur.cur_cross_batched(hd.h, data, items, cur.opts(1e-2), IJ, info)
    st = cur.cur_sync_status(hd.h)
    sets, o = [], 0
    for m, n, r, *_ in shapes:
        v = IJ[o:o + 2 * r].tolist()
        sets.append((v[:r], v[r:]))
        o += 2 * r
    return st, sets


def _valid(sets, shapes):
    for (I, J), (m, n, r, *_) in zip(sets, shapes):
        assert len(set(I)) == r and 0 <= min(I) and max(I) < m
        assert len(set(J)) == r and 0 <= min(J) and max(J) < n


def test_a_lost_matrix_leaves_the_others_alone():
    shapes = [(300, 131, 9, 1, 1), (1030, 64, 17, 2, 1), (257, 514, 33, 1, 2), (66, 35, 8, 1, 1), (513, 997, 40, 1, 1)]
    data, items = _setup(shapes)
    with cur.Handle(1, 1, 1, workspace_bytes=cur.cur_batch_workspace_size(items)) as hd:
        st, want = _run(hd, data, items, shapes)
        assert st == cur.CUR_OK
        cur.cur_selftest_batch_timeout(hd.h, 2)
        st, got = _run(hd, data, items, shapes)
        assert st == cur.CUR_ERR_TIMEOUT
        _valid(got, shapes)
        assert [s for t, s in enumerate(got) if t != 2] == [s for t, s in enumerate(want) if t != 2]
        assert _run(hd, data, items, shapes) == (cur.CUR_OK, want)


def test_every_matrix_of_a_lost_batch_has_valid_sets():
    count = 2 * torch.cuda.get_device_properties(0).multi_processor_count + 57   # more than any launch has CTAs
    shapes = [(40 + t % 7, 30 + t % 5, 4, 1, 1) for t in range(count)]
    data, items = _setup(shapes)
    with cur.Handle(1, 1, 1, workspace_bytes=cur.cur_batch_workspace_size(items)) as hd:
        cur.cur_selftest_batch_timeout(hd.h, count)
        st, got = _run(hd, data, items, shapes)
        assert st == cur.CUR_ERR_TIMEOUT
        _valid(got, shapes)
        st, got = _run(hd, data, items, shapes)
        assert st == cur.CUR_OK
        _valid(got, shapes)
