"""The reduction of the training step's partial gradients: one CTA's partials per 32 samples, summed
in order, sixteen loads at a time and a remainder. With a power of two of CTAs the weight 1 / N
scales exactly, so the whole gradient has to be, bit for bit, the ordered FP32 sum of the
gradients of each 32 samples alone (and the loss the ordered FP64 sum). With other counts the two
differ by rounding: an entry is a sum of 32 nb products, each with a weight of two roundings, summed by
32 and then by nb additions on either side, so within 2 (32 + nb + 8) 2^-24 of the sum of the
products' magnitudes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2502_11017_gb300 as cur

pytestmark = pytest.mark.gpu
K, H, PW = 32, 64, 3.0


def _grad(hd, X, y, p):
    g = torch.empty_like(p)
    loss = torch.empty(1, dtype=torch.float64, device="cuda")
    cur.cur_mlp_grad(hd.h, X, y, p, g, loss, pos_weight=PW, H=H)
    return g.cpu().numpy(), loss.item()


def _magnitudes(X, y, p):
    """Per entry of the gradient, the sum of its terms' magnitudes."""
    X, y, p = X.double(), y.double(), p.double()
    W1, b1, w2 = p[:K * H].view(K, H), p[K * H:K * H + H], p[K * H + H:K * H + 2 * H]
    hid = (X @ W1 + b1).clamp_min(0.0)
    ds = (torch.where(y > 0.5, PW, 1.0) * (torch.sigmoid(hid @ w2 + p[-1]) - y) / len(y)).abs()
    dh = ds[:, None] * w2.abs() * (hid > 0)
    return torch.cat([(X.abs().T @ dh).reshape(-1), dh.sum(0), hid.T @ ds, ds.sum()[None]]).cpu().numpy()


@pytest.mark.parametrize("nb", [1, 2, 8, 15, 16, 17, 31, 32, 33, 64, 100, 128])
def test_partial_gradients_are_summed_in_order(nb):
    rng = torch.Generator(device="cuda").manual_seed(nb)
    X = torch.randn((32 * nb, K), generator=rng, device="cuda")
    y = (torch.rand(32 * nb, generator=rng, device="cuda") < 0.25).float()
    p = torch.randn(cur.mlp_param_count(K, H), generator=rng, device="cuda") * 0.2
    with cur.Handle(4096, 1024, 16, cur.CUR_F32) as hd:
        got, loss = _grad(hd, X, y, p)
        parts = [_grad(hd, X[32 * b:32 * b + 32], y[32 * b:32 * b + 32], p) for b in range(nb)]
        assert cur.cur_sync_status(hd.h) == cur.CUR_OK
    s, t = np.zeros_like(got), 0.0
    for g, l in parts:
        s += g / np.float32(nb)
        t += float(np.float32(l) / np.float32(nb))
    if nb & (nb - 1) == 0:
        assert np.array_equal(got, s)
        assert loss == t
    else:
        assert (np.abs(got.astype(np.float64) - s) <= 2 * (32 + nb + 8) * 2.0 ** -24 * _magnitudes(X, y, p)).all()
        assert abs(loss - t) <= 2 * (32 + nb + 8) * 2.0 ** -24 * t
