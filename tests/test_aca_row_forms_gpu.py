"""The row pass of Algorithm 3 (selection of rows) in its forms: row by row with the terms one by one, one
row per warp, four rows per warp; by vectors and off the 16-byte grid. Row counts on both sides of
each line of the dispatch (16, 40 and 64 rows per SM) in the three data types, with n that leaves
lanes and warps ragged ends, against pivoted Gram-Schmidt in 64 bits; and the column pass, where a
large matrix's chunks are at least 128 rows, and in FP64, the same way."""
import pytest

torch = pytest.importorskip("torch")

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu
CODE = {torch.float64: cur.CUR_F64, torch.float32: cur.CUR_F32, torch.bfloat16: cur.CUR_BF16}


def _select(A, axis, r):
    idx = torch.full((r,), -7, dtype=torch.int32, device="cuda")
    with cur.Handle(A.shape[0], A.shape[1], r, CODE[A.dtype]) as hd:
        cur.cur_aca_select(hd.h, A, axis, r, 1, idx)
        return cur.cur_sync_status(hd.h), idx.tolist()


def _greedy(V, r):
    """The columns that pivoted Gram-Schmidt picks, each projected twice, in 64 bits."""
    V = V.double()
    Q = torch.zeros((V.shape[0], 0), dtype=torch.float64, device=V.device)
    nu = V.square().sum(0)
    picks = []
    for _ in range(r):
        p = int(nu.argmax())
        picks.append(p)
        v = V[:, p]
        v = v - Q @ (Q.T @ v)
        v = v - Q @ (Q.T @ v)
        q = v / v.norm()
        Q = torch.cat([Q, q[:, None]], 1)
        nu = nu - (V.T @ q).square()
        nu[p] = -torch.inf
    return picks


def _matrix(m, n, dtype, per_row):
    g = torch.Generator(device="cuda").manual_seed(m + 7 * n)
    A = torch.randn((m, n), generator=g, device="cuda")
    A *= 1.0 + torch.rand((m, 1) if per_row else (1, n), generator=g, device="cuda")
    return A.to(dtype)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float64])
@pytest.mark.parametrize("n", [96, 131, 1000, 1027])
@pytest.mark.parametrize("per_sm,more", [(0, 33), (16, -1), (16, 0), (40, -1), (40, 0), (64, -1), (64, 0), (64, 5)])
def test_rows(per_sm, more, n, dtype):
    A = _matrix(per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more, n, dtype, True)
    assert _select(A, 0, 7) == (cur.CUR_OK, _greedy(A.T, 7))


@pytest.mark.parametrize("m,n,dtype", [
    (65536, 512, torch.float32), (65537, 384, torch.float32), (200003, 128, torch.float32), (3100, 8200, torch.float32),
    (65536, 64, torch.bfloat16), (20001, 256, torch.bfloat16), (300, 16384, torch.bfloat16), (100, 40000, torch.bfloat16),
    (1000, 1001, torch.float64), (31, 77, torch.float64), (5003, 640, torch.float64),
])
def test_columns(m, n, dtype):
    A = _matrix(m, n, dtype, False)
    assert _select(A, 1, 7) == (cur.CUR_OK, _greedy(A, 7))
