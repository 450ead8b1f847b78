"""The paired-FMA residual (FP32 data with r other than 32 and 64 or off the 16-byte grid, BF16
data) against the plain CUDA-core kernel, which the allocation-free call still runs: each element
is the same FMA chain, so the Chebyshev residual is the same number; the Frobenius ratio adds the
same FP32 tile sums in FP64 in another order (at most 2^20 of them: 2^20 2^-53 < 2e-10)."""
import pytest
import torch

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu


def _case(m, n, r, pad, off, dtype):
    g = torch.Generator(device="cuda").manual_seed(m + 3 * n + r)
    buf = torch.randn(m * (n + pad) + off, generator=g, device="cuda").to(dtype)
    A = buf[off:].view(m, n + pad)[:, :n]
    C = torch.randn((m, r), generator=g, device="cuda").to(dtype)
    R = torch.randn((r, n), generator=g, device="cuda").to(dtype)
    U = torch.randn((r, r), generator=g, device="cuda", dtype=torch.float64) / r
    return A, C, U, R


def _both(A, C, U, R, r):
    out = []
    for alloc in (True, False):
        cheb = torch.zeros(1, dtype=torch.float64, device="cuda")
        fro = torch.zeros(1, dtype=torch.float64, device="cuda")
        if alloc:
            with cur.Handle(A.shape[0], A.shape[1], r, cur.CUR_F32) as hd:
                cur.cur_residual_cheb(hd.h, A, C, U, R, r, cheb, fro)
                st = cur.cur_sync_status(hd.h)
        else:
            cur.cur_residual_cheb_noalloc(A, C, U, R, r, cheb, fro)
        out.append((cheb.item(), fro.item()))
    return out, st


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("m,n,r,pad,off", [
    (1, 1, 1, 0, 0), (128, 128, 16, 0, 0), (129, 127, 17, 1, 0), (127, 129, 15, 0, 1), (300, 2050, 33, 0, 0),
    (1000, 700, 128, 2, 0), (40000, 130, 100, 0, 0), (260, 20003, 48, 0, 3), (3000, 4096, 127, 0, 0),
])
def test_same_as_the_plain_kernel(m, n, r, pad, off, dtype):
    (a, b), st = _both(*_case(m, n, r, pad, off, dtype), r)
    assert st == cur.CUR_OK
    assert a[0] == b[0]
    assert a[1] == pytest.approx(b[1], rel=1e-9)


@pytest.mark.parametrize("what", [float("nan"), float("inf")])
@pytest.mark.parametrize("where", [0, 1, 2])
def test_not_finite(where, what):
    A, C, U, R = _case(200, 200, 24, 0, 0, torch.bfloat16)
    (A, C, U)[where][3, 5] = what
    (a, b), st = _both(A, C, U, R, 24)
    assert str(a[0]) == str(b[0]) and (st == cur.CUR_ERR_NONFINITE) == (b[0] != b[0])
