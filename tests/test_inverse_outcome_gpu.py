"""A cluster's FP64 inverse where one CTA's last message is withheld by the self-test: its wait runs
out, and every CTA of the cluster has to report that, not only the one that waited (the others'
columns alone are no inverse)."""
import pytest
import torch

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lost", [-1, 0, 1, 2])
def test_a_lost_message_is_every_cta_s_outcome(lost):
    out = torch.full((4,), -1, dtype=torch.int32, device="cuda")
    with cur.Handle(64, 64, 16, cur.CUR_F64) as hd:
        cur.cur_selftest_inverse(hd.h, lost, out)
        assert cur.cur_sync_status(hd.h) == cur.CUR_OK
    assert out.tolist() == ([0] * 4 if lost < 0 else [2] * 4)
