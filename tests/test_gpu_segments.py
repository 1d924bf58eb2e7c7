"""Edges of the grid and segment splits of the small per-batch kernels: sizes where a split changes
(one cluster or several, a warp or a CTA per trajectory, vector or scalar loads), values that take
a kernel's rare path, and views whose alignment rules the wide loads out."""

import numpy as np
import pytest
import torch

import oracle.grpo_objective as O
import oracle.ppo_objective as PO
from parity_cases import check_gae, gae_error_scale

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


@pytest.mark.parametrize("skip", [0, 1])
@pytest.mark.parametrize("n_traj", [14, 1217, 5000])
def test_gae_warp_and_cta_trajectories(R, n_traj, skip):
    """Lengths at the edges of a lane's, a warp's and a CTA's chunk (4, 128, 1,024 tokens) and of
    the warp form (512), one and several trajectories per CTA, spans that leave tokens uncovered."""
    rng = np.random.default_rng(n_traj + skip)
    edges = np.array([0, 1, 3, 4, 5, 127, 128, 129, 511, 512, 513, 1024, 1025, 2300])
    lens = rng.integers(0, 20, n_traj)
    lens[rng.permutation(n_traj)[:14]] = edges
    offs = np.zeros(n_traj + 1, np.int64)
    np.cumsum(lens, out=offs[1:])
    offs += 3
    T = int(offs[-1]) + 5
    mask = (rng.random(T) < 0.6).astype(np.uint8)
    V = rng.normal(0.3, 0.25, T).astype(np.float32)
    rt = np.where(rng.random(T) < 0.1, rng.normal(0, 0.1, T), 0).astype(np.float32)
    Ri = (rng.random(n_traj) < 0.5).astype(np.float32)
    ws = R.new_workspace(0, 0)
    adv, ret = (torch.full((T,), 7.0, device="cuda") for _ in range(2))
    R.rl_masked_gae(dev(offs), dev(mask), dev(V), ws, 0.99, 0.97, bool(skip), token_rewards=dev(rt),
                    traj_rewards=dev(Ri), adv_out=adv, returns_out=ret)
    mask, V, rt = mask[:T - 5], V[:T - 5], rt[:T - 5]
    rew = PO.final_token_rewards(offs, mask, Ri) + rt.astype(np.float64)
    fn = PO.masked_gae_skip if skip else PO.masked_gae
    g, lam = float(np.float32(0.99)), float(np.float32(0.97))
    a_ref, r_ref = fn(offs, mask, V, rew, g, lam)
    S = gae_error_scale(offs, mask, V, rew, g, lam, skip)
    adv, ret = adv.cpu().numpy().astype(np.float64), ret.cpu().numpy().astype(np.float64)
    assert np.all(adv[:3] == 7) and np.all(ret[-5:] == 7)  # outside every span: not written
    sl = slice(3, T - 5)
    check_gae(adv[sl], ret[sl], a_ref[sl], r_ref[sl], V[sl], S[sl], mask[sl], 2300, f"n {n_traj} skip {skip}")
    assert R.rl_query_status(ws)[1] == 0


@pytest.mark.parametrize("lead", [0, 1])
@pytest.mark.parametrize("n_groups,lo,hi", [(1, 8, 8), (300, 1, 9), (1500, 3, 5), (40, 2, 70)])
def test_advantage_segments_and_spans(R, n_groups, lo, hi, lead):
    """Group sizes on both sides of the lanes a group gets (with one far above the mean), spans of 0
    to 700 tokens counted by a warp or by a CTA, arrays that start off the 16-byte boundary."""
    rng = np.random.default_rng(n_groups + lead)
    sizes = rng.integers(lo, hi + 1, n_groups)
    sizes[n_groups // 2] = 8 * hi + 3
    go = np.zeros(n_groups + 1, np.int32)
    np.cumsum(sizes, out=go[1:])
    n = int(go[-1])
    lens = rng.integers(0, 30, n)
    lens[: min(n, 40)] = rng.integers(60, 700, min(n, 40))
    offs = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=offs[1:])
    T = int(offs[-1])
    rew = rng.integers(0, 3, n).astype(np.float32)
    valid = (rng.random(n) < 0.9).astype(np.uint8)
    mask = (rng.integers(0, 4, T) * 60).astype(np.uint8)
    owner = np.repeat(np.arange(n, dtype=np.int32), lens)
    ws = R.new_workspace(0, 0)
    P = R.make_params()
    OP = O.LossParams()
    a_ref, c_ref, L_ref, _ = O.advantages_and_coefficients(rew, go, offs, (mask != 0).astype(np.uint8), valid, OP)
    tt = dev(np.full(T, -1, np.int32), lead)
    spans = R.rl_group_advantages(dev(go), dev(rew), dev(offs), dev(mask, lead), P, ws, traj_valid=dev(valid),
                                  token_traj_out=tt)
    perm = rng.permutation(T)
    by_owner = R.rl_group_advantages_by_owner(dev(go), dev(rew), dev(owner[perm]), dev(mask[perm]), P, ws,
                                              traj_valid=dev(valid))
    assert np.array_equal(spans[3].cpu().numpy(), owner)
    for got in (spans, by_owner):
        assert np.array_equal(got[2].cpu().numpy(), L_ref)
        for x, ref in ((got[0], a_ref), (got[1], c_ref)):  # double arithmetic, rounded once to float32
            x = x.cpu().numpy().astype(np.float64)
            assert np.all(np.abs(x - ref) <= 2.0 ** -24 * np.abs(ref) * 1.001 + 1e-30)
    assert R.rl_query_status(ws)[1] == 0


@pytest.mark.parametrize("lead", [0, 1])
@pytest.mark.parametrize("rows", [1, 3, 4, 1023, 1025, 700001])
def test_value_loss_vector_tails(R, rows, lead):
    """Four rows per load with up to three left over, and arrays that rule the wide loads out."""
    rng = np.random.default_rng(rows + lead)
    v, g = (rng.normal(0, 1, rows).astype(np.float32) for _ in range(2))
    mask = (rng.random(rows) < 0.6).astype(np.uint8)
    tt = rng.integers(0, 7, rows).astype(np.int32)
    coef = np.array([0.5, 0, 1e-3, 1, 0.25, 3e-5, 0.1], np.float32)
    ws, loss = R.new_workspace(rows, 0), torch.zeros(1, dtype=torch.float64, device="cuda")
    d = R.rl_value_loss_fwd_bwd(dev(v, lead), dev(g, lead), dev(mask, lead), dev(tt, lead), dev(coef), ws, loss)
    l_ref, d_ref, _ = PO.value_loss_fwd_bwd(v, g, mask, tt, coef.astype(np.float64))
    assert abs(loss.item() - l_ref) <= 4 * 2.0 ** -24 * abs(l_ref) + 1e-30  # two float32 roundings per term
    assert np.all(np.abs(d.cpu().numpy() - d_ref) <= 4 * 2.0 ** -24 * np.abs(d_ref) + 1e-30)
    tt[0], mask[0] = 9, 1
    R.rl_value_loss_fwd_bwd(dev(v), dev(g), dev(mask), dev(tt), dev(coef), ws, loss)
    assert R.rl_query_status(ws)[1] == R.RL_DEV_BAD_TRAJ


@pytest.mark.parametrize("lead", [0, 1])
@pytest.mark.parametrize("order", ["runs", "short", "pairs", "random"])
@pytest.mark.parametrize("T", [1, 127, 130, 50003])
def test_owner_sums_orders(R, T, order, lead):
    """Owners in long runs, in runs of 8, alternating, and in random order: the same sums, and the
    bits of the double-rounded differences (values near 0, above 2^12 and clamped ones among them)."""
    rng = np.random.default_rng(T + lead)
    n = 23
    owner = {"runs": np.arange(T) * n // T, "short": np.arange(T) // 8 % n, "pairs": np.arange(T) % 2,
             "random": rng.integers(0, n, T)}[order].astype(np.int32)
    old = -rng.exponential(1.0, T).astype(np.float32)
    old[rng.random(T) < 0.1] *= np.float32(1e-7)
    old[rng.random(T) < 0.05] = 0.0
    roll = (old + rng.normal(0, 0.01, T)).astype(np.float32)
    old[0] = -9000.25
    mask = (rng.random(T) < 0.7).astype(np.uint8)
    fixed = np.rint((old.astype(np.float64) - roll.astype(np.float64)) * 2.0 ** 40)
    S = np.zeros(n, np.int64)
    np.add.at(S, owner[mask != 0], fixed[mask != 0].astype(np.int64))
    ws = R.new_workspace(n, 0)
    w, ratio = R.rl_sequence_is_weights(dev(owner, lead), dev(mask, lead), dev(old, lead), dev(roll, lead), n, ws,
                                        cap=2.0, want_log_ratio=True)
    assert np.array_equal(ratio.cpu().numpy(), (S / 2.0 ** 40).astype(np.float32))
    ref = np.minimum(np.exp(S / 2.0 ** 40), 2.0)
    assert np.all(np.abs(w.cpu().numpy() - ref) <= 2.0 ** -23 * ref + 1e-30)
    assert R.rl_query_status(ws)[1] == 0
