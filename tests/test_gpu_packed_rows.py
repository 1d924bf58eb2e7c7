"""Rows that start and end inside 16-byte blocks (any leading dimension): the loss and its gradient,
also in place, and the forward log-probs, against float64 torch, with the sampled id at every
position of the partial blocks and the buffers' surroundings poisoned."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_2608_16798_gb300.rl_loss as R

    return R


def buffer(rows, V, ld, dtype):
    """[rows, V] view of exactly (rows - 1) ld + V elements, NaN guards on both sides."""
    n = (rows - 1) * ld + V
    whole = torch.full((64 + n + 64,), float("nan"), dtype=dtype, device="cuda")
    return whole, whole[64:64 + n].as_strided((rows, V), (ld, 1))


def outside(whole, rows, V, ld):
    """Every element of the buffer that belongs to no row."""
    keep = torch.ones(len(whole), dtype=torch.bool, device="cuda")
    at = 64 + torch.arange(rows, device="cuda")[:, None] * ld + torch.arange(V, device="cuda")
    keep[at.flatten()] = False
    return whole[keep]


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("ent", [0.0, 0.01])
@pytest.mark.parametrize("V,pad", [(1, 0), (2, 1), (5, 0), (7, 2), (9, 0), (1003, 0), (1003, 2), (4097, 0), (4099, 5),
                                   (20487, 0), (32003, 0), (163850, 3)])
def test_packed_rows(R, V, pad, ent, dtype):
    rng = np.random.default_rng(V + pad)
    rows, ld = 23, V + pad
    src, z = buffer(rows, V, ld, dtype)
    z.copy_(torch.from_numpy(rng.normal(0, 2, (rows, V)).astype(np.float32)))
    x = z.double()
    edge = np.r_[np.arange(8), V - 1 - np.arange(8), rng.integers(0, V, rows - 16)] % V
    ids = torch.from_numpy(np.maximum(edge, 0).astype(np.int32)).cuda()
    lp = torch.log_softmax(x, 1)
    logp = lp.gather(1, ids.long()[:, None])[:, 0]
    H = -(lp.exp() * lp).sum(1)
    mask = torch.from_numpy((rng.random(rows) < 0.8).astype(np.uint8)).cuda()
    mask[-1] = 1  # the last row, whose last block reaches past the buffer
    tt = torch.arange(rows, dtype=torch.int32, device="cuda") % 3
    adv, coef = (torch.tensor(a, device="cuda") for a in ([1.0, -0.5, 2.0], [1.0, 0.5, 0.25]))
    old = (logp - 0.05).float()
    ws = R.new_workspace(rows, V)
    P = R.make_params(entropy_coef=ent)
    # float64: c (rho A below the clip: g = -A rho) and the entropy term
    A, c = adv.double()[tt.long()], coef.double()[tt.long()]
    rho = torch.exp(logp - old.double())
    e32 = float(np.float32(ent))
    g = -A * rho
    ref = -g[:, None] * lp.exp() + e32 * lp.exp() * (lp + H[:, None])
    ref.scatter_add_(1, ids.long()[:, None], g[:, None])
    ref = ref * (c * (mask != 0))[:, None]
    l_ref = (c * (mask != 0) * (-A * rho - e32 * H)).sum()
    scale = (c * (A.abs() * rho + e32 * (1 + H)))[:, None]
    fmt = 2.0 ** -8 if dtype == torch.bfloat16 else 2.0 ** -23
    for in_place in (False, True):
        dst, grad = (src, z) if in_place else buffer(rows, V, ld, dtype)
        loss = torch.zeros(1, dtype=torch.float64, device="cuda")
        if not in_place:
            out = R.rl_token_logprobs(z, ids, ws, want_entropy=True, want_lse=True)
            lse = torch.logsumexp(x, 1)
            assert ((out[0] - logp).abs() <= 1e-5 + 2.0 ** -22 * logp.abs()).all()
            assert ((out[1] - H).abs() <= 5e-5 + 2e-5 * H.abs()).all()
            assert ((out[2] - lse).abs() <= 1e-5 + 2.0 ** -22 * lse.abs()).all()
        R.rl_policy_loss_fwd_bwd(z, ids, mask, tt, adv, coef, old, P, ws, loss, grad_out=grad)
        assert abs(loss.item() - l_ref.item()) <= 1e-4 * (c * A.abs() * rho).sum().item()
        # the tolerance of the aligned path: format rounding, 2e-5 of the value and of the row's scale
        err = (grad.double() - ref).abs()
        assert (err <= (fmt + 2e-5) * ref.abs() + 2e-5 * scale).all(), (in_place, err.max().item())
        assert torch.isnan(outside(dst, rows, V, ld)).all()
    assert R.rl_query_status(ws)[1] == 0
