"""Rows whose softmax is undefined (a NaN or +inf logit, every logit at -inf): their loss term and
gradient are NaN in every form of the loss kernel, whatever outputs are asked for, and the other rows
keep the bits that they have without them. The forward call gives such a row a NaN lse."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_2608_16798_gb300.rl_loss as R

    return R


ROWS, BAD = 5, 2


def logits(dtype, V, ld):
    g = torch.Generator(device="cuda").manual_seed(V + ld)
    z = torch.empty(ROWS, ld, dtype=dtype, device="cuda")[:, :V]
    z.copy_(torch.randn(ROWS, V, device="cuda", generator=g) * 2)
    return z


def loss(R, z, stats, ent):
    V = z.shape[1]
    ids = torch.tensor([0, V // 3, 1, V - 1, V // 2], dtype=torch.int32, device="cuda")
    mask, tt = torch.ones(ROWS, dtype=torch.uint8, device="cuda"), torch.zeros(ROWS, dtype=torch.int32, device="cuda")
    one = torch.ones(1, device="cuda")
    total = torch.zeros(1, dtype=torch.float64, device="cuda")
    ws = R.new_workspace(ROWS, V)
    g = R.rl_policy_loss_fwd_bwd(z, ids, mask, tt, one, one, torch.full((ROWS,), -8.0, device="cuda"),
                                 R.make_params(entropy_coef=ent), ws, total,
                                 token_stats=torch.empty(ROWS, 5, device="cuda") if stats else None)
    lse = R.rl_token_logprobs(z, ids, ws, want_lse=True)[2]
    assert R.rl_query_status(ws)[1] == 0
    return total.item(), g, lse


# bf16: warps with 4, 8 and 16 vectors a lane, one CTA and clusters; fp32: warps, the aligned kernel and
# the shifted one, wide rows on both of their shapes
@pytest.mark.parametrize("dtype,V,ld", [
    (torch.bfloat16, 1000, 1000), (torch.bfloat16, 2000, 2003), (torch.bfloat16, 4096, 4096),
    (torch.bfloat16, 12000, 12000), (torch.bfloat16, 32003, 32003), (torch.bfloat16, 151936, 151936),
    (torch.float32, 500, 500), (torch.float32, 2048, 2051), (torch.float32, 32000, 32000),
    (torch.float32, 32000, 32003), (torch.float32, 151936, 151936), (torch.float32, 200001, 200001)])
@pytest.mark.parametrize("what", ["nan", "inf", "none", "lanes", "all"])
def test_undefined_rows_make_the_loss_nan(R, dtype, V, ld, what):
    """lanes: every 32nd 16-byte block of the row, all that some threads hold; all: the whole row."""
    z = logits(dtype, V, ld)
    _, clean, lse0 = loss(R, z, False, 0.0)
    if what == "none":
        z[BAD] = float("-inf")
    elif what == "lanes":
        z[BAD, torch.arange(V, device="cuda") // (16 // z.element_size()) % 32 == 5] = float("nan")
    elif what == "all":
        z[BAD] = float("nan")
    else:
        z[BAD, V // 2] = float(what)
    others = [r for r in range(ROWS) if r != BAD]
    for stats, ent in ((False, 0.0), (True, 0.0), (False, 0.01)):
        total, g, lse = loss(R, z, stats, ent)
        assert total != total, (stats, ent)
        assert torch.equal(lse[others], lse0[others])
        assert what == "none" or lse[BAD].isnan()
        assert g[BAD].isnan().any()
        if not stats and not ent:
            assert torch.equal(g[others], clean[others])
