"""sum E^2 and sum A^2 of the tensor-core residual over many tiles. Each thread first meets a tile of
ones and then tiles of entries so small that a tile's sum is below half an ulp of its FP32 running
sum. Every FP32 sum within a tile is exact by construction (squares of 19 bits, 8 of them to a
chain), and a thread's total has 43 bits, so sums of the tiles in FP64 are exact up to the few
additions over threads and CTAs, at most 30 roundings of 2^-53: 1e-14 is three times that. With
C = 0 and U = 0 the error is A itself."""
from fractions import Fraction

import pytest
import torch

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [32, 64])
def test_tile_sums_keep_64_bits(r):
    m, n = 256 * torch.cuda.get_device_properties(0).multi_processor_count, 8192   # a pair of row panels per SM
    small = 683 * 2.0 ** -21
    A = torch.full((m, n), small, device="cuda")
    A[:, :128] = 1.0
    C = torch.zeros((m, r), device="cuda")
    R = torch.zeros((r, n), device="cuda")
    U = torch.zeros((r, r), dtype=torch.float64, device="cuda")
    parts = torch.zeros(3, dtype=torch.float64, device="cuda")
    with cur.Handle(m, n, r, cur.CUR_F32) as hd:
        cur.cur_residual_parts(hd.h, A, C, U, R, r, parts)
        assert cur.cur_sync_status(hd.h) == cur.CUR_OK
    want = m * (128 + (n - 128) * Fraction(683, 2 ** 21) ** 2)
    top, e2, a2 = parts.tolist()
    assert top == 1.0
    for got in (e2, a2):
        assert abs(Fraction(got) - want) <= Fraction(1e-14) * want
