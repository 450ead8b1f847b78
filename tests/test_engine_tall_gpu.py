"""The swap engine on the tallest bases it takes: with B in global memory a CTA's rows leave less
shared memory for the staged rows of C the more of them there are. Sizes above what 128 staged rows
allow (3.7, 5.2 and 6.7 million rows at r = 128, 97 and 65 in FP32) and below what 32 did; one with
r off the 16-byte grid, one by way of the BF16 products, one FP64.

The bars are those of the other engine tests: the set's own log-volume, and a (1 + delta)-dominant
set, in 64 bits over all rows."""
import pytest
import torch

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu
DELTA = 1e-2


@pytest.mark.parametrize("p,r,dtype,bf16", [
    (4000003, 128, torch.float32, False), (4900000, 128, torch.float32, True), (6000001, 97, torch.float32, False),
    (7200000, 65, torch.float32, False), (1500001, 128, torch.float64, False),
])
def test_tall_bases_are_taken(p, r, dtype, bf16):
    g = torch.Generator(device="cuda").manual_seed(r)
    C = torch.randn((p, r), generator=g, device="cuda", dtype=dtype)
    S0 = torch.randperm(p, generator=g, device="cuda")[:r].to(torch.int32)
    S = torch.empty(r, dtype=torch.int32, device="cuda")
    lv = torch.empty(1, dtype=torch.float64, device="cuda")
    sw = torch.zeros(2, dtype=torch.int32, device="cuda")
    with cur.Handle(p, r, r, cur.CUR_F64 if dtype == torch.float64 else cur.CUR_F32) as hd:
        cur.cur_maxvol_global(hd.h, C, S0, r, cur.opts(DELTA, bf16=bf16), S, lv, sw)
        assert cur.cur_sync_status(hd.h) == cur.CUR_OK
    Sl = S.long()
    assert len(set(S.tolist())) == r and sw[0].item() > 0
    M = C[Sl].double()
    assert lv.item() == pytest.approx(torch.linalg.slogdet(M)[1].item(), abs=1e-6 * r)
    inv = torch.linalg.inv(M)
    top = max((C[s:s + (1 << 20)].double() @ inv).abs().max().item() for s in range(0, p, 1 << 20))
    assert top <= (1 + DELTA) * (1 + 1e-4)
