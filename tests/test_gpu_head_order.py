"""A token's statistics through the fused head do not depend on the call that it is part of: the same
bits in calls of other sizes (whose work items are other vocabulary blocks), in the smallest
workspaces, and in the forward-only call."""

import numpy as np
import pytest
import torch

from parity_cases import to_dev
from test_gpu_fused_head import _bf16_dev, compare_head, make_head_case
from test_gpu_head_tokens import least_bytes, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_2608_16798_gb300.rl_loss as R

    return R


def part(c, n):
    """The first n tokens of the case."""
    return dict(c, T=n, **{k: None if c[k] is None else c[k][:n] for k in ("h", "ids", "mask", "tt", "old", "ref", "roll")})


def forward(R, c, ws_bytes):
    ws = torch.zeros(ws_bytes, dtype=torch.uint8, device="cuda")
    ws[256:] = 255
    out = R.rl_fused_head_token_logprobs(_bf16_dev(c["h"]), _bf16_dev(c["w"]), to_dev(c["ids"]), ws, want_entropy=True,
                                         want_lse=True)
    assert R.rl_query_status(ws)[1] == 0
    return [x.cpu().numpy() for x in out]


# vocabularies of one block of 4,096 and of several with a ragged last one; the sizes have work items of
# 2 to 16 tiles of 256 entries
@pytest.mark.parametrize("V", [700, 4096, 33000])
def test_statistics_do_not_depend_on_the_call(R, V):
    T, D = 4500, 64
    c = make_head_case(T, D, V, seed=V, masked=0.4, ent=True)
    whole = run(R, c)
    fwd = forward(R, c, R.rl_workspace_size(T, V, D))
    on = (c["mask"] != 0) & (c["coef32"][c["tt"]] != 0)
    assert np.array_equal(whole["stats"][on, 0], fwd[0][on]) and np.array_equal(whole["stats"][on, 3], fwd[1][on])
    for n in (1, 100, 300, 1000, 2048, 4096):
        p = part(c, n)
        a = run(R, p)
        assert np.array_equal(a["stats"], whole["stats"][:n]), n
        if n in (300, 2048):  # without packing and finer work items
            assert np.array_equal(run(R, p, least_bytes(n, V))["stats"], a["stats"]), n
        least = 256 + 32 * -(-V // 4096) * n + 256
        for size in (R.rl_workspace_size(n, V, D), least // 256 * 256):
            for x, y in zip(forward(R, p, size), fwd):
                assert np.array_equal(x, y[:n]), (n, size)


def test_short_call_parity(R):
    """A few tokens and nine blocks of 16 tiles: every step of the merge against the oracle."""
    c = make_head_case(200, 64, 33000, seed=7, ent=True)
    compare_head(c, run(R, c))
