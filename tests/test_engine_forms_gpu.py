"""The swap engine's forms by size: M^-1 on a CTA of its own (ranks above 64), B in global memory
in 16-byte and in element accesses, FP64, and the refactorisation in place; against the
oracle's maxvol from the same start. And the FP64 inverses (columns in registers, one CTA or a
cluster) at the edges of their plans, against LAPACK.

The bars are those of the other engine tests: the oracle's set, or a volume within 0.999 of it, a
(1 + delta)-dominant set, the set's own log-volume. An inverse is held to |U M - 1| <= 4 r eps
kappa_1 (Gauss-Jordan with partial pivoting; growth is small for Gaussian matrices)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2502_11017_gb300 as cur
from paper_2502_11017_gb300 import workloads as wl
from oracle import cur_oracle as orc

pytestmark = pytest.mark.gpu
DELTA = 1e-2


@pytest.mark.parametrize("p,r,dtype,always", [
    (300, 70, np.float32, False), (260, 100, np.float32, False), (9001, 66, np.float32, False),
    (41000, 128, np.float32, False), (41000, 128, np.float32, True), (66001, 97, np.float32, False),
    (90001, 64, np.float32, False), (400, 100, np.float64, False), (12001, 127, np.float64, False),
])
def test_engine_forms_match_the_oracle(p, r, dtype, always):
    rng = np.random.default_rng(p + r)
    C = ((rng.standard_normal((p, r)) * np.exp(-3.0 * np.arange(r) / r)) @ wl.haar(r, r, rng).T).astype(dtype)
    C64 = C.astype(np.float64)
    S0 = rng.choice(p, r, replace=False).astype(np.int32)
    S = torch.empty(r, dtype=torch.int32, device="cuda")
    lv = torch.empty(1, dtype=torch.float64, device="cuda")
    sw = torch.zeros(2, dtype=torch.int32, device="cuda")
    with cur.Handle(p, r, r, cur.CUR_F64 if dtype == np.float64 else cur.CUR_F32) as hd:
        cur.cur_maxvol_global(hd.h, torch.from_numpy(C).cuda(), torch.from_numpy(S0).cuda(), r,
                              cur.opts(DELTA, refactor_always=always), S, lv, sw)
        assert cur.cur_sync_status(hd.h) == cur.CUR_OK
        refactors = cur.cur_prof_refactors(hd.h)
    assert refactors > 0 or not (always or dtype == np.float64)
    So, lvo, swo, _st = orc.maxvol(C64, S0.tolist(), DELTA)
    Sg = S.tolist()
    assert len(set(Sg)) == r
    lv_set = orc.logvol(C64[Sg, :])
    assert lv.item() == pytest.approx(lv_set, abs=1e-6 * max(1.0, abs(lv_set)))
    assert sorted(Sg) == sorted(So) or lv_set >= lvo + math.log(0.999)
    assert np.abs(C64 @ np.linalg.inv(C64[Sg, :])).max() <= (1 + DELTA) * (1 + 1e-4)


@pytest.mark.parametrize("r", [1, 2, 15, 16, 17, 32, 33, 34, 48, 49, 64, 65, 96, 97, 127, 128])
def test_inverse_at_the_edges_of_its_plans(r):
    rng = np.random.default_rng(r)
    n = 3 * r + 5
    a = rng.standard_normal((n, n))
    I = rng.permutation(n)[:r].astype(np.int32)
    J = rng.permutation(n)[:r].astype(np.int32)
    A = torch.from_numpy(a).cuda()
    U = torch.empty((r, r), dtype=torch.float64, device="cuda")
    rc = torch.empty(1, dtype=torch.float64, device="cuda")
    with cur.Handle(n, n, r, cur.CUR_F64) as hd:
        cur.cur_assemble(hd.h, A, torch.from_numpy(I).cuda(), torch.from_numpy(J).cuda(), r, None, U, None, rc)
        assert cur.cur_sync_status(hd.h) == cur.CUR_OK
    M = a[np.ix_(I, J)]
    kappa = np.abs(M).sum(0).max() * np.abs(np.linalg.inv(M)).sum(0).max()
    assert np.abs(U.cpu().numpy() @ M - np.eye(r)).max() <= 4 * r * 2.2e-16 * kappa
    assert rc.item() == pytest.approx(1.0 / kappa, rel=1e-8)


@pytest.mark.parametrize("r", [5, 40, 128])
def test_singular_inverse_becomes_the_pseudo_inverse(r):
    rng = np.random.default_rng(r)
    M = rng.standard_normal((r, r - 1)) @ rng.standard_normal((r - 1, r))
    M[:, r - 1] = M[:, 0]          # exactly singular
    A = torch.from_numpy(M).cuda()
    idx = torch.arange(r, dtype=torch.int32, device="cuda")
    U = torch.empty((r, r), dtype=torch.float64, device="cuda")
    rc = torch.empty(1, dtype=torch.float64, device="cuda")
    with cur.Handle(r, r, r, cur.CUR_F64) as hd:
        cur.cur_assemble(hd.h, A, idx, idx, r, None, U, None, rc)
        assert cur.cur_sync_status(hd.h) == cur.CUR_OK
    P = np.linalg.pinv(M, rcond=r * 2.2e-16)
    s = np.linalg.svd(M, compute_uv=False)
    assert np.abs(U.cpu().numpy() - P).max() <= 1e-10 * (s[0] / s[r - 3]) * np.abs(P).max()
    assert rc.item() < 1e-13
