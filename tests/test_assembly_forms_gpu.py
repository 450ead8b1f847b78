"""The assembly's inverse on both sides of the rank that takes a cluster (44 and 45), against LAPACK:
|U M - 1| <= 4 r eps kappa_1 and rcond, as at the edges of the cluster's own plans."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,code", [(torch.float64, cur.CUR_F64), (torch.float32, cur.CUR_F32), (torch.bfloat16, cur.CUR_BF16)])
@pytest.mark.parametrize("r", [1, 3, 31, 43, 44, 45, 46])
def test_inverse_on_both_sides_of_the_line(r, dtype, code):
    rng = np.random.default_rng(100 + r)
    n = 3 * r + 5
    A = torch.from_numpy(rng.standard_normal((n, n))).to(dtype).cuda()
    I = rng.permutation(n)[:r].astype(np.int32)
    J = rng.permutation(n)[:r].astype(np.int32)
    U = torch.empty((r, r), dtype=torch.float64, device="cuda")
    rc = torch.empty(1, dtype=torch.float64, device="cuda")
    with cur.Handle(n, n, r, code) as hd:
        cur.cur_assemble(hd.h, A, torch.from_numpy(I).cuda(), torch.from_numpy(J).cuda(), r, None, U, None, rc)
        assert cur.cur_sync_status(hd.h) == cur.CUR_OK
    M = A.double().cpu().numpy()[np.ix_(I, J)]
    kappa = np.abs(M).sum(0).max() * np.abs(np.linalg.inv(M)).sum(0).max()
    assert np.abs(U.cpu().numpy() @ M - np.eye(r)).max() <= 4 * r * 2.2e-16 * kappa
    assert rc.item() == pytest.approx(1.0 / kappa, rel=1e-8)
