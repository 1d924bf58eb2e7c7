"""Edges of the grid and segment splits of the small per-batch kernels: sizes where a split changes
(one cluster or several, a warp or a CTA per trajectory, vector or scalar loads), values that take
a kernel's rare path, and views whose alignment rules the wide loads out."""

import numpy as np
import pytest
import torch

import oracle.grpo_objective as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_2608_16798_gb300.rl_loss as R

    return R


def dev(x, lead=0):
    """x on the device; with `lead`, as a view that starts that many elements into its allocation."""
    t = torch.from_numpy(np.ascontiguousarray(x))
    out = torch.empty(t.numel() + lead, dtype=t.dtype, device="cuda")
    out[lead:] = t.reshape(-1).cuda()
    return out[lead:].view(t.shape)


@pytest.mark.parametrize("rows,ws_lead", [(1, 0), (8192, 0), (8193, 0), (40961, 0), (200001, 0), (8193, 4)])
def test_stats_summary_clusters(R, rows, ws_lead):
    """One cluster up to 8,192 rows, then up to five; flags other than 0 and 1, subnormals, zeros
    and an infinity are summed as the numbers they are. A workspace off the 8-byte boundary runs on
    one cluster. Double sums of at most 2e5 values: 1e-12 of the sum of magnitudes."""
    rng = np.random.default_rng(rows)
    st = rng.normal(0, 1, (rows, 5)).astype(np.float32)
    st[:, 2] = rng.integers(0, 2, rows)
    st[rng.integers(0, rows, 3), 2] = 0.5
    st[rng.integers(0, rows, 3), 4] = 1e-40
    st[rng.integers(0, rows, 3), 3] = 0.0
    mask = (rng.random(rows) < 0.7).astype(np.uint8)
    tt = rng.integers(0, 9, rows).astype(np.int32)
    coef = np.where(np.arange(9) == 4, 0.0, 0.1).astype(np.float32)
    on = (mask != 0) & (coef[tt] != 0)
    v = st[on].astype(np.float64)
    ref = np.array([on.sum(), v[:, 2].sum(), v[:, 3].sum(), v[:, 4].sum(), v[:, 1].sum()])
    mag = np.array([on.sum(), v[:, 2].sum(), np.abs(v[:, 3]).sum(), np.abs(v[:, 4]).sum(), np.abs(v[:, 1]).sum()])
    ws = torch.zeros(256 + ws_lead, dtype=torch.uint8, device="cuda")[ws_lead:]
    args = (dev(st), dev(mask), dev(tt), dev(coef), ws)
    a, b = (R.rl_token_stats_summary(*args).cpu().numpy() for _ in range(2))
    assert np.array_equal(a, b)
    assert np.all(np.abs(a - ref) <= 1e-12 * mag + 1e-30)
    st[np.flatnonzero(on)[:1], 4] = np.inf
    c = R.rl_token_stats_summary(dev(st), *args[1:]).cpu().numpy()
    assert (c[3] == np.inf if on.any() else c[3] == 0) and np.array_equal(c[[0, 1, 2, 4]], a[[0, 1, 2, 4]])
    assert R.rl_query_status(ws)[1] == 0
