"""The inverses of a stage by its number of problems: clusters of eight, four or two CTAs, one CTA with
columns in registers, one with the matrix in shared memory. P copies of one block, stacked, are P
problems whose sets and merges have to be the block's own set, whichever form inverted them (a
merge starts from the left set, and a copy of a chosen row never gains); the log-volume is its set's.
The block alone is the reference. Statuses of singular and of non-finite data do not depend on the
form either."""
import pytest
import torch

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu


def _rows(X, r, P):
    A = X.repeat(P, 1)
    J = torch.arange(r, dtype=torch.int32, device="cuda")
    I = torch.zeros(r, dtype=torch.int32, device="cuda")
    lv = torch.zeros(1, dtype=torch.float64, device="cuda")
    with cur.Handle(A.shape[0], r, r, cur.CUR_F64 if X.dtype == torch.float64 else cur.CUR_F32) as hd:
        cur.cur_maxvol_rows(hd.h, A, J, r, cur.opts(1e-2, nblocks=P, polish=False), I, lv)
        return cur.cur_sync_status(hd.h), I.tolist(), lv.item()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("r,counts", [
    (16, (153, 1024)), (24, (153,)), (25, (152, 153, 304)), (32, (152, 153)), (33, (2, 153)), (35, (76, 77)), (48, (76, 77)),
    (49, (36, 37)), (64, (36, 37, 76, 77, 305)), (65, (19, 20, 76)), (74, (20, 36)), (75, (36, 37)), (88, (36, 37, 76)),
    (89, (37, 76, 77)), (128, (19, 20, 36, 37, 77)),
])
def test_every_form_gives_the_block_s_own_set(r, counts, dtype):
    g = torch.Generator(device="cuda").manual_seed(r)
    X = torch.randn((r + 70, r), generator=g, device="cuda", dtype=torch.float64).to(dtype)
    st, I, lv = _rows(X, r, 1)
    assert st == cur.CUR_OK and len(set(I)) == r
    want = torch.linalg.slogdet(X[I].double())[1].item()
    assert lv == pytest.approx(want, abs=1e-9 * r)
    for P in counts:
        st, got, lvp = _rows(X, r, P)
        assert st == cur.CUR_OK
        assert got == I
        assert lvp == pytest.approx(want, abs=1e-9 * r)


@pytest.mark.parametrize("r", [32, 64, 96])
def test_statuses_do_not_depend_on_the_form(r):
    g = torch.Generator(device="cuda").manual_seed(r)
    X = torch.randn((r + 70, r), generator=g, device="cuda")
    X[:, 1] = X[:, 0]
    assert {_rows(X, r, P)[0] for P in (1, 36, 76, 160)} == {_rows(X, r, 1)[0]}
    X = torch.randn((r + 70, r), generator=g, device="cuda")
    X[5, 3] = float("nan")
    assert {_rows(X, r, P)[0] for P in (1, 36, 76, 160)} == {cur.CUR_ERR_NONFINITE}
