"""Groups of CTAs above rank 64 by their share of the SMs: FP32 groups whose keeper of M^-1 comes out of the
share, FP64 groups without one, groups as small as the rows allow, and a last group that waits for the
others. P copies of one block, stacked, have to give the block's own set, swaps aside: a merge
starts from the left set, and a copy of a chosen row never gains. The block alone (one group over
many SMs) is the reference, and its set is dominant in 64 bits."""
import pytest
import torch

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu
DELTA = 1e-2


def _rows(X, r, P):
    A = X.repeat(P, 1)
    J = torch.arange(r, dtype=torch.int32, device="cuda")
    I = torch.zeros(r, dtype=torch.int32, device="cuda")
    lv = torch.zeros(1, dtype=torch.float64, device="cuda")
    with cur.Handle(A.shape[0], r, r, cur.CUR_F64 if X.dtype == torch.float64 else cur.CUR_F32) as hd:
        cur.cur_maxvol_rows(hd.h, A, J, r, cur.opts(DELTA, nblocks=P, polish=False), I, lv)
        return cur.cur_sync_status(hd.h), I.tolist(), lv.item()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("P,rows,r", [(4, 3000, 128), (12, 1500, 128), (38, 600, 96), (2, 6000, 100), (19, 2000, 70), (80, 250, 127)])
def test_groups_give_the_block_s_own_set(P, rows, r, dtype):
    g = torch.Generator(device="cuda").manual_seed(P + r)
    X = torch.randn((rows, r), generator=g, device="cuda", dtype=torch.float64).to(dtype)
    st, I, lv = _rows(X, r, 1)
    assert st == cur.CUR_OK and len(set(I)) == r
    M = X[I].double()
    assert lv == pytest.approx(torch.linalg.slogdet(M)[1].item(), abs=1e-9 * r)
    assert (X.double() @ torch.linalg.inv(M)).abs().max().item() <= (1 + DELTA) * (1 + 1e-4)
    st, got, lvp = _rows(X, r, P)
    assert st == cur.CUR_OK and got == I
    assert lvp == pytest.approx(lv, abs=1e-9 * r)
