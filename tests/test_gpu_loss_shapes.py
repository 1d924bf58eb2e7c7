"""Every shape and cluster width that the loss kernel's launcher picks by row length, at the longest row
of each (full slices, the held vectors all in use) and at odd lengths packed without padding, with and
without the entropy, against float64 torch."""

import numpy as np
import pytest
import torch

from loss_shapes import F32_PLAIN, PICKS, SHAPES, pick

ROWS = 4


def _cases():
    out = []
    for dtype, picks in PICKS.items():
        lo = F32_PLAIN if dtype == "f32" else 4096
        for V, shape, C in picks:
            mid = (lo + V) // 2 | 1  # odd: rows start anywhere
            for ent in (0.0, 0.01):
                out += [(dtype, V, V, ent), (dtype, mid, mid, ent), (dtype, V - 1, V + 7, ent)]
            lo = V
    for V in (2052, 30720, 43003, F32_PLAIN):  # fp32 rows on the plain kernel: one CTA, few, 16 of them
        out += [("f32", V, V + (-V) % 4, 0.01), ("f32", V - 1, V - 1, 0.0)]
    return out


CASES = _cases()


def test_the_cases_reach_every_shape():
    """Every row of the tables, and every (type, shape, entropy, rows off the boundaries) that is a kernel
    of its own (no GPU needed)."""
    picked = {(d, *pick(d, V)) for d, V, _, _ in CASES}
    assert {(d, s, C) for d, t in PICKS.items() for _, s, C in t} <= picked
    kernels = {(d, pick(d, V)[0], ent > 0, ld * (4 if d == "f32" else 2) % 16 != 0) for d, V, ld, ent in CASES}
    for d, t in PICKS.items():
        for s in {s for _, s, _ in t}:
            assert {(d, s, e, u) for e in (False, True) for u in (False, True)} <= kernels, (d, SHAPES[s])
    assert {s for t in PICKS.values() for _, s, _ in t} == set(range(len(SHAPES)))  # none that nothing picks


@pytest.fixture(scope="module")
def R():
    import paper_2608_16798_gb300.rl_loss as R

    return R


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,V,ld,ent", CASES)
def test_loss_at_every_shape(R, dtype, V, ld, ent):
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(V)
    z = torch.empty((ROWS - 1) * ld + V, dtype=dt, device="cuda").as_strided((ROWS, V), (ld, 1))
    z.copy_(torch.randn(ROWS, V, device="cuda", generator=g) * 2)
    ids = torch.tensor([V - 1, 0, V // 2, V // 3], dtype=torch.int32, device="cuda")
    mask = torch.tensor([1, 0, 1, 1], dtype=torch.uint8, device="cuda")
    tt = torch.tensor([0, 1, 1, 2], dtype=torch.int32, device="cuda")
    adv, coef = (torch.tensor(a, device="cuda") for a in ([1.0, -0.5, 2.0], [1.0, 0.5, 0.25]))
    x = z.double()
    lp = torch.log_softmax(x, 1)
    logp = lp.gather(1, ids.long()[:, None])[:, 0]
    H = -(lp.exp() * lp).sum(1)
    old = (logp - 0.05).float()
    # float64: c (rho A below the clip: g = -A rho) and the entropy term
    A, c = adv.double()[tt.long()], coef.double()[tt.long()] * mask
    rho = torch.exp(logp - old.double())
    e32 = float(np.float32(ent))
    d = -A * rho
    ref = -d[:, None] * lp.exp() + e32 * lp.exp() * (lp + H[:, None])
    ref.scatter_add_(1, ids.long()[:, None], d[:, None])
    ref = ref * c[:, None]
    l_ref = (c * (-A * rho - e32 * H)).sum().item()
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    ws = R.new_workspace(ROWS, V)
    R.rl_policy_loss_fwd_bwd(z, ids, mask, tt, adv, coef, old, R.make_params(entropy_coef=ent), ws, loss, grad_out=z)
    assert R.rl_query_status(ws)[1] == 0
    # the tolerances of the other parity tests: 1e-4 of the summed terms; format rounding, 2e-5 of the
    # value and of the row's scale
    assert abs(loss.item() - l_ref) <= 1e-4 * (c * (A.abs() * rho + e32 * H)).sum().item()
    scale = (c * (A.abs() * rho + e32 * (1 + H)))[:, None]
    fmt = 2.0 ** -8 if dtype == "bf16" else 2.0 ** -23
    err = (z.double() - ref).abs()
    assert (err <= (fmt + 2e-5) * ref.abs() + 2e-5 * scale).all(), err.max().item()
