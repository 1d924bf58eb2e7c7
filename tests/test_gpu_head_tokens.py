"""The fused head's packed tokens and its work splits, against the float64 oracle: numbers of
trained tokens at the edges of a 64-token block, a 256-token tile and a chunk, workspaces that leave
out the packing or the split contraction, groups of packed chunks, and untrained tokens whose hidden
states are NaN."""

import numpy as np
import pytest
import torch

from parity_cases import cuda_params, to_dev
from test_gpu_fused_head import _bf16_dev, compare_head, make_head_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_2608_16798_gb300.rl_loss as R

    return R


def least_bytes(T, V):
    """Status word, loss terms, partials of 4,096-entry blocks, coefficients, tile maxima and one
    chunk's logits gradient: a workspace with neither packed tokens nor parts of dH."""
    al = lambda x: (x + 255) // 256 * 256  # noqa: E731
    Tc, n_nt = min(T, 4096), -(-V // 256)
    return 256 + al(T * 8) + al(2 * -(-n_nt // 16) * Tc * 16) + al(Tc * 32) + al(Tc * n_nt * 4) + al(Tc * -(-V // 8) * 16)


def run(R, c, ws_bytes=None, dh=torch.float32, d_w=None):
    T, D, V = c["T"], c["D"], c["V"]
    ws = torch.zeros(ws_bytes or R.rl_workspace_size(T, V, D), dtype=torch.uint8, device="cuda")
    ws[256:] = 255  # NaNs wherever something is read before it is written
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    dW = torch.zeros((V, D), dtype=torch.float32, device="cuda") if d_w is None else d_w
    st = torch.full((T * 5,), float("nan"), dtype=torch.float32, device="cuda")
    dH = torch.full((T, D), float("nan"), dtype=dh, device="cuda")
    R.rl_fused_head_loss_fwd_bwd(c["h_dev"] if "h_dev" in c else _bf16_dev(c["h"]), _bf16_dev(c["w"]), to_dev(c["ids"]),
                                 to_dev(c["mask"]), to_dev(c["tt"].astype(np.int32)), to_dev(c["adv32"]),
                                 to_dev(c["coef32"]), to_dev(c["old"]), cuda_params(R, c["P"]), ws, loss, dW, d_hidden=dH,
                                 ref_logp=None if c["ref"] is None else to_dev(c["ref"]),
                                 rollout_logp=None if c["roll"] is None else to_dev(c["roll"]), token_stats=st)
    word = R.rl_query_status(ws)[1]
    return dict(loss=loss.item(), dH=dH.float().cpu().numpy().astype(np.float64),
                dW=dW.cpu().numpy().astype(np.float64), stats=st.view(-1, 5).cpu().numpy(), word=word)


def case(T, D, V, n, seed, **kw):
    """A case with exactly n trained tokens, spread over the batch."""
    c = make_head_case(T, D, V, seed=seed, agg=2, **kw)
    c["mask"] = np.zeros(T, np.uint8)
    c["mask"][np.random.default_rng(seed).permutation(T)[:n]] = 1
    return c


@pytest.mark.parametrize("T,D,V,n", [(300, 128, 777, 0), (300, 128, 777, 1), (300, 128, 777, 64), (300, 192, 2100, 65),
                                     (300, 128, 777, 300), (1100, 576, 5000, 257), (4500, 64, 300, 4097),
                                     (4500, 64, 300, 4500), (9000, 64, 300, 4096)])
@pytest.mark.parametrize("dh", [torch.float32, torch.bfloat16])
def test_trained_token_counts(R, T, D, V, n, dh):
    c = case(T, D, V, n, seed=T + n)
    out = run(R, c, dh=dh)
    if n:
        compare_head(c, out, dh_bf16=dh is torch.bfloat16)
    else:
        assert out["loss"] == 0 and not out["dH"].any() and not out["dW"].any() and not out["stats"].any()


@pytest.mark.parametrize("T,D,V,n", [(500, 128, 9000, 300), (4200, 64, 520, 4150)])
def test_workspaces_without_packing(R, T, D, V, n):
    """The least workspace that is accepted takes every token through the products; one byte less is
    refused; room for several packed chunks (4,150 trained tokens are two) puts them in one group."""
    c = case(T, D, V, n, seed=T, ent=True)
    a = run(R, c, least_bytes(T, V))
    compare_head(c, a)
    with pytest.raises(R.RLError):
        run(R, c, least_bytes(T, V) - 256)
    b = run(R, c, 3 * R.rl_workspace_size(T, V, D))
    compare_head(c, b)
    assert np.allclose(a["stats"], b["stats"], rtol=1e-4, atol=1e-5)


# around the largest call that one launch selects in (8,192), and one whose first thousands of tokens
# are untrained; 70,000: more CTAs than a warp has lanes
@pytest.mark.parametrize("T,first", [(8192, 0), (8193, 0), (9217, 5000), (70000, 0)])
def test_selection_of_long_calls(R, T, first):
    c = make_head_case(T, 64, 130, seed=T, agg=2)
    c["mask"][:first] = 0
    compare_head(c, run(R, c))


# trained tokens that make 1, 2, 3 and 4 chunks of the 4 that 16,384 tokens can need
@pytest.mark.parametrize("n,need", [(4000, 1), (8100, 2), (12200, 3), (16384, 4)])
@pytest.mark.parametrize("asked", [1, 2, 3, 4])
def test_groups_are_as_large_as_asked(R, n, need, asked):
    """The size asked for a group of several chunks gives groups of that many, right also with a second
    group after a full first one. d W shows how many groups there were: each adds to it once, so on top
    of other values it is one rounded addition of the call's own d W exactly when one group holds all."""
    T, D, V = 16384, 64, 300
    c = case(T, D, V, n, seed=n)
    size = R.rl_fused_head_workspace_size(T, V, D, asked * 4096)
    a = run(R, c, size)
    compare_head(c, a)
    base = torch.from_numpy(np.random.default_rng(1).normal(0, 64 * np.abs(a["dW"]).max(), (V, D)).astype(np.float32))
    b = run(R, c, size, d_w=base.cuda())
    once = (base + torch.from_numpy(a["dW"].astype(np.float32))).numpy().astype(np.float64)
    assert np.array_equal(b["dW"], once) == (need <= asked)


def test_untrained_tokens_do_not_enter(R):
    """NaN hidden states of masked tokens, a bad id and a bad owner (flagged): no trace in d W."""
    c = case(700, 128, 1500, 400, seed=3)
    off = np.flatnonzero(c["mask"] == 0)
    on = np.flatnonzero(c["mask"])[:2]
    c["ids"][on[0]], c["tt"][on[1]] = 1500, 99
    h = _bf16_dev(c["h"])
    h[torch.from_numpy(off).cuda()] = float("nan")
    out = run(R, dict(c, h_dev=h))
    assert out["word"] == R.RL_DEV_BAD_TOKEN | R.RL_DEV_BAD_TRAJ
    c["mask"][on], c["ids"][on[0]], c["tt"][on[1]] = 0, 0, 0
    ref = run(R, c)
    compare_head(c, ref)
    for k in ("dH", "dW", "stats", "loss"):
        assert np.array_equal(out[k], ref[k]), k
