"""A round's pick and direction by 8, 4 and 1 lanes per row of the vectors. With G CTAs (one per SM) the
rows of a CTA are ceil(length / G): up to 32 take eight lanes, up to 64 four, more one. Zero rows
appended to the vectors change no sum but take the same selection past both lines, so each length
is run as it is, with four lanes and with one, and all have to pick what pivoted Gram-Schmidt
picks in 64 bits. Lengths on both sides of each line, shares that differ by a row, CTAs without a row,
and more than 32 and more than 64 directions (the sums over the CTAs go by blocks of them)."""
import pytest

torch = pytest.importorskip("torch")

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu
CODE = {torch.float32: cur.CUR_F32, torch.bfloat16: cur.CUR_BF16}


def _select(V, axis, r):
    A = V if axis == 1 else V.t().contiguous()
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


def _lengths(name):
    G = torch.cuda.get_device_properties(0).multi_processor_count
    return {"few": 101, "ragged": 31 * G + 7, "8 at most": 32 * G, "8 past": 32 * G + 1, "4 at most": 64 * G, "4 past": 64 * G + 1}[name], G


@pytest.mark.parametrize("axis", [1, 0])
@pytest.mark.parametrize("where,r,dtype", [
    ("few", 64, torch.float32), ("ragged", 128, torch.float32), ("8 at most", 33, torch.float32), ("8 at most", 65, torch.bfloat16),
    ("8 past", 128, torch.float32), ("8 past", 20, torch.bfloat16), ("4 at most", 66, torch.float32), ("4 past", 40, torch.float32),
])
def test_every_number_of_lanes_picks_the_same(where, r, dtype, axis):
    length, G = _lengths(where)
    g = torch.Generator(device="cuda").manual_seed(length + r)
    V = torch.randn((length, r + 150), generator=g, device="cuda") * (1.0 + torch.rand(r + 150, generator=g, device="cuda"))
    V = V.to(dtype)
    want = _greedy(V, r)
    for rows in sorted({length, max(length, 32 * G + 1), 64 * G + 129}):   # as it is, four lanes, one
        W = torch.zeros((rows, V.shape[1]), dtype=dtype, device="cuda")
        W[:length] = V
        assert _select(W, axis, r) == (cur.CUR_OK, want), rows


@pytest.mark.parametrize("axis", [1, 0])
@pytest.mark.parametrize("where", ["few", "ragged", "8 past", "4 past"])
def test_a_vector_that_vanishes_ends_every_form(where, axis):
    length, G = _lengths(where)
    g = torch.Generator(device="cuda").manual_seed(length)
    ints = lambda *s: torch.randint(-4, 5, s, generator=g, device="cuda").float()
    V = ints(length, 12) @ ints(12, 90)      # integers: rank 12 without rounding
    for rows in sorted({length, max(length, 32 * G + 1), 64 * G + 129}):
        W = torch.zeros((rows, 90), device="cuda")
        W[:length] = V
        st, idx = _select(W, axis, 40)
        assert st == cur.CUR_WARN_RANK
        assert len({i for i in idx if i >= 0}) == 12 and idx[12:] == [-1] * 28
