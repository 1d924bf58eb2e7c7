"""The fused head's rescale, which also merges a row's partials, and its loss sum: one CTA per row or
several (short calls of wide vocabularies), vocabularies that end inside a vector, a tile or a part,
with and without the entropy, against the float64 oracle; the loss total is added to, and every run
gives the same bits."""

import numpy as np
import pytest
import torch

from test_gpu_fused_head import compare_head
from test_gpu_head_tokens import case, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_2608_16798_gb300.rl_loss as R

    return R


# (T, V): V / 4,096 parts where 1,216 / T allows them: 1; 1 (8,191 is one vector short of 2); 2; 3 of
# 9; 11; 2 for T = 608, 1 for 609; a handful of tokens
@pytest.mark.parametrize("T,V", [(40, 4095), (40, 8191), (40, 8192), (400, 36867), (100, 45058), (608, 8200),
                                 (609, 8200), (5, 20001)])
@pytest.mark.parametrize("ent", [False, True])
def test_rows_shared_by_ctas(R, T, V, ent):
    c = case(T, 64, V, max(1, T * 2 // 3), seed=T + V, ent=ent)
    on = np.flatnonzero(c["mask"])
    c["ids"][on[0]], c["ids"][on[-1]] = V - 1, V // 2  # the row's last element; one near a part's edge
    a, b = run(R, c), run(R, c)
    compare_head(c, a)
    for k in ("dH", "dW", "stats", "loss"):
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("n", [4400, 3000])
def test_loss_total_is_added_to(R, n):
    """Three calls on one workspace and one total; with 3,000 trained tokens the last chunk is empty."""
    from parity_cases import cuda_params, to_dev
    from test_gpu_fused_head import _bf16_dev

    c = case(4500, 64, 300, n, seed=5)
    one = run(R, c)["loss"]
    ws = R.new_workspace(4500, 300, 64)
    loss = torch.full((1,), 1.0, dtype=torch.float64, device="cuda")
    dW = torch.zeros((300, 64), dtype=torch.float32, device="cuda")
    for _ in range(3):
        R.rl_fused_head_loss_fwd_bwd(_bf16_dev(c["h"]), _bf16_dev(c["w"]), to_dev(c["ids"]), to_dev(c["mask"]),
                                     to_dev(c["tt"].astype(np.int32)), to_dev(c["adv32"]), to_dev(c["coef32"]),
                                     to_dev(c["old"]), cuda_params(R, c["P"]), ws, loss, dW,
                                     d_hidden=torch.empty((4500, 64), dtype=torch.float32, device="cuda"),
                                     ref_logp=None if c["ref"] is None else to_dev(c["ref"]),
                                     rollout_logp=None if c["roll"] is None else to_dev(c["roll"]))
    # three additions in double precision, each rounded to 2^-53 of a total of at most 1 + 3 |one|
    assert abs(loss.item() - (1.0 + 3 * one)) <= 4 * 2.0**-53 * (1 + 3 * abs(one))
