"""The passes of Algorithm 3 by the form of A: the same matrix on the 16-byte grid (large: the
asynchronous column pass; vector row loads) and one element off it (the direct passes) gives the
same picks, for sizes with ragged last tiles, chunks and stages. All forms sum to ~2^-48 and the
picks' norms differ by far more on these matrices (independent columns with spread scales)."""
import pytest
import torch

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu


def _select(A, axis, r):
    idx = torch.empty(r, dtype=torch.int32, device="cuda")
    code = {torch.float32: cur.CUR_F32, torch.float64: cur.CUR_F64, torch.bfloat16: cur.CUR_BF16}[A.dtype]
    with cur.Handle(A.shape[0], A.shape[1], r, code) as hd:
        cur.cur_aca_select(hd.h, A, axis, r, 1, idx)
        st = cur.cur_sync_status(hd.h)
    return st, idx.tolist()


@pytest.mark.parametrize("axis", [1, 0])
@pytest.mark.parametrize("m,n,ld,dtype", [
    (4099, 6202, 6204, torch.float32), (20011, 1301, 1304, torch.float32), (70, 380000, 380000, torch.float32),
    (4099, 1601, 1602, torch.float64), (6001, 4203, 4208, torch.bfloat16), (33000, 805, 808, torch.bfloat16),
    (2500, 130, 132, torch.float32), (10001, 33, 40, torch.bfloat16), (4099, 771, 776, torch.bfloat16),
])
def test_picks_do_not_depend_on_the_pass(m, n, ld, dtype, axis):
    g = torch.Generator(device="cuda").manual_seed(m + n)
    scale = lambda k: 1.0 + torch.rand(k, generator=g, device="cuda")
    vals = torch.randn((m, n), generator=g, device="cuda") * scale(n) * scale(m)[:, None]
    picks = []
    for off in (0, 1):
        buf = torch.full((m * ld + 8,), float("nan"), dtype=dtype, device="cuda")
        A = buf[off:off + m * ld].view(m, ld)[:, :n]
        A.copy_(vals)
        picks.append(_select(A, axis, 12))
    assert picks[0] == picks[1] and picks[0][0] == cur.CUR_OK
    exact = vals.to(dtype).double()
    norms = exact.square().sum(0 if axis == 1 else 1)
    assert picks[0][1][0] == int(norms.argmax())
