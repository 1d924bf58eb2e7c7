"""The work that a training program has this library do, as cases that can be timed and compared.

A case is one pass through the public binding (``paper_2608_16798_gb300.rl_loss``) on inputs that
already lie on the GPU, with the workspace and output buffers that a training loop keeps:

  step          advantages and coefficients of a small batch, then the policy loss and its gradient
  loss          the policy loss and its gradient over one microbatch of logits rows
  logprobs      forward-only log-probabilities (the pi_old / pi_ref recompute)
  head_loss     the loss through the fused LM head: d hidden and d W
  head_logprobs forward-only log-probabilities through the fused LM head
  batch         everything a batch needs besides the logits: advantages, sequence-level weights,
                masked GAE (or R - V for tokens in any order), the value loss, the statistics

Inputs follow the laws of ``workloads.py`` (normal logits, Gumbel-max sampled ids, log-ratios
kept 1e-4 away from the clip bounds so that every correct implementation takes the same clip
branch) and are drawn on the device from the seed. ``exact`` states every result in float64 with
plain torch.
"""

import math

import numpy as np
import torch

import paper_2608_16798_gb300.rl_loss as R

DEV = "cuda"
EPS_LOW, EPS_HIGH = 0.2, 0.28
RATIO_BAND = 1e-4
ADV_EPS = 1e-6
TIS_CAP = 2.0
CHUNK_ELEMS = 1 << 27  # logits elements handled at once by prepare() and exact()


def _loss(name, rows, V, dtype, law, std, kl=0.0, ent=0.0, tis=False, stats=False, ld=0):
    c = dict(kind="loss", rows=rows, V=V, ld=ld or V, dtype=dtype, law=law, std=std, kl=kl, ent=ent, tis=tis,
             stats=stats)
    return dict(c, name=name) if name else c


def _logprobs(name, rows, V, dtype, std, ent, ld=0):
    c = dict(kind="logprobs", rows=rows, V=V, ld=ld or V, dtype=dtype, std=std, ent=ent)
    return dict(c, name=name) if name else c


def _head(name, kind, T, D, V, ent=False, kl=0.0, dh="bf16"):
    c = dict(kind=kind, T=T, D=D, V=V, ent=ent, kl=kl, dh=dh)
    return dict(c, name=name) if name else c


def _batch(name, groups, size, lo, hi, law, packing, gamma=1.0, lam=1.0, cap=TIS_CAP):
    c = dict(kind="batch", groups=groups, size=size, lo=lo, hi=hi, law=law, packing=packing, gamma=gamma, lam=lam,
             cap=cap)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a whole update step at the smallest configuration: latency and launches
        dict(name="step_tiny", kind="step", groups=1, size=8, lo=64, hi=64, V=4096, dtype="bf16", std=3.0),
        # the benchmark's microbatch of a multi-turn agent batch
        _loss("loss_multiturn", 16384, 151936, "bf16", "spans", 2.0),
        # a long-horizon microbatch: entropy bonus, reference KL, monitored statistics
        _loss("loss_longhorizon", 8192, 151936, "bf16", "spans", 2.0, kl=1e-3, ent=1e-3, stats=True),
        # the edge batch's fp32 logits: near-one-hot rows, rows of -1e4 entries, both clip bounds
        _loss("loss_edge_f32", 32768, 32000, "f32", "edge", 2.0),
        # a model that upcasts its logits to fp32, at the full vocabulary, with the rollout weight
        _loss("loss_wide_f32", 2048, 151936, "f32", "spans", 2.0, tis=True),
        # packed rows of a vocabulary with three added tokens: rows start at any element
        _loss("loss_added_tokens", 8192, 32003, "bf16", "spans", 2.0),
        # pi_old recompute of a microbatch, with the entropy that training monitors
        _logprobs("logprobs_multiturn", 8192, 151936, "bf16", 2.0, True),
        # the fused head on a ragged microbatch of more than one chunk, at the full model
        _head("head_loss_large", "head_loss", 6000, 4096, 151936),
        # the fused head of a small model on a short last microbatch
        _head("head_loss_small", "head_loss", 500, 1024, 32000),
        # pi_old recompute through the fused head
        _head("head_logprobs", "head_logprobs", 2048, 2048, 151936, ent=True),
        # a long-horizon PPO batch: 512 trajectories of 512 to 8,192 tokens
        _batch("batch_longhorizon", 32, 16, 512, 8192, "spans", "spans", gamma=1.0, lam=0.97),
        # many short trajectories: 4,096 groups of 4 x 8 tokens
        _batch("batch_edge", 4096, 4, 8, 8, "edge", "spans"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "loss", "loss", "loss", "logprobs", "logprobs", "head_loss", "head_logprobs", "batch"])
    if kind == "step":
        size = rng.choice([4, 8, 16])
        lo = _log_int(rng, 16, 256)
        return dict(kind=kind, groups=rng.randint(1, 4), size=size, lo=lo, hi=lo + rng.randint(0, lo),
                    V=rng.choice([1000, 1003, 2048, 4096, 8192]), dtype="bf16", std=3.0)
    if kind in ("loss", "logprobs"):
        dtype = rng.choice(["bf16", "bf16", "f32"])
        V = _log_int(rng, 1000, 200000)
        if rng.random() < 0.6:
            V = max(64, V // 64 * 64)  # padded vocabularies are the common ones
        ld = (V + 63) // 64 * 64 if rng.random() < 0.25 else V
        es = 2 if dtype == "bf16" else 4
        rows = max(1, min(65536, _log_int(rng, 1 << 21, 3 << 30) // (V * es)))
        if kind == "loss":
            return _loss(None, rows, V, dtype, rng.choice(["spans", "spans", "none", "edge"]), 2.0,
                         kl=rng.choice([0.0, 1e-3]), ent=rng.choice([0.0, 0.0, 1e-3]), tis=rng.random() < 0.3,
                         stats=rng.random() < 0.3, ld=ld)
        return _logprobs(None, rows, V, dtype, 2.0, rng.random() < 0.5, ld=ld)
    if kind in ("head_loss", "head_logprobs"):
        D = 64 * rng.randint(8, 64)
        V = _log_int(rng, 16000, 151936)
        T = _log_int(rng, 64, 6000)
        if kind == "head_loss":
            return _head(None, kind, T, D, V, ent=rng.random() < 0.3, kl=rng.choice([0.0, 1e-3]),
                         dh=rng.choice(["bf16", "bf16", "f32"]))
        return _head(None, kind, T, D, V, ent=rng.random() < 0.5)
    lo = _log_int(rng, 8, 512)
    hi = lo * rng.choice([1, 4, 16])
    size = rng.choice([4, 8, 16])
    groups = max(1, min(4096, _log_int(rng, 1 << 13, 1 << 20) // (size * (lo + hi) // 2)))
    return _batch(None, groups, size, lo, hi, "spans" if lo >= 64 else "edge", rng.choice(["spans", "owners"]),
                  gamma=rng.choice([1.0, 0.99]), lam=rng.choice([1.0, 0.97]), cap=rng.choice([0.0, TIS_CAP]))


# ----------------------------------------------------------------------------- inputs

def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1_000_003 + stream * 7919) & 0x7FFFFFFFFFFF)
    return g


def _mask_np(lengths, law, rng):
    """Trainable spans U{64..752} and masked spans U{32..512} in turn; edge: whole trajectories
    masked (1/4), whole ones trained on (1/2), the rest mixed token by token."""
    T = int(lengths.sum())
    if law == "none":
        return np.ones(T, np.uint8)
    if law == "edge":
        kind = np.repeat(rng.random(len(lengths)), lengths)
        coin = rng.random(T) < 0.5
        return np.where(kind < 0.25, 0, np.where(kind < 0.75, 1, coin)).astype(np.uint8)
    m = np.empty(T, np.uint8)
    pos = 0
    for n in lengths:
        end, on = pos + int(n), True
        while pos < end:
            k = min(end - pos, int(rng.integers(64, 753)) if on else int(rng.integers(32, 513)))
            m[pos:pos + k] = on
            pos += k
            on = not on
    return m


def _layout(case, seed, T=None):
    """Trajectories in groups: offsets, rewards and mask (with T: as many groups of 8 of 256 to
    2,048 tokens as cover T tokens, the mask and owners of the first T of them)."""
    rng = np.random.default_rng([int(seed) & 0xFFFFFFFF, 17])
    law = case.get("law", "none")
    if T is None:
        groups, size = case["groups"], case["size"]
        # log-uniform lengths: the case's own set of them (so its sizes do not depend on the seed),
        # in an order of the seed's
        u = np.random.default_rng([groups, size, case["lo"], case["hi"]]).uniform(
            math.log(case["lo"]), math.log(case["hi"] + 1), groups * size)
        lengths = rng.permutation(np.clip(np.floor(np.exp(u)), case["lo"], case["hi"]).astype(np.int64))
    else:
        lo, hi, size = (8, 8, 4) if law == "edge" else (256, 2048, 8)
        lengths = rng.integers(lo, hi + 1, (T // lo // size + 1) * size).astype(np.int64)
        need = int(np.searchsorted(np.cumsum(lengths), T)) + 1
        groups = -(-need // size)
        lengths = lengths[:groups * size]
    n = groups * size
    offs = np.zeros(n + 1, np.int64)
    np.cumsum(lengths, out=offs[1:])
    rewards = (rng.random(n) < (0.5 if law == "edge" else 0.3)).astype(np.float32)
    rewards[0], rewards[size - 1] = 1.0, 0.0  # at least one group that learns something
    return dict(offs=offs, go=(np.arange(groups + 1) * size).astype(np.int32), rewards=rewards,
                mask=_mask_np(lengths, law, rng), owner=np.repeat(np.arange(n, dtype=np.int32), lengths))


def _advantages64(go, rewards, L, agg):
    """Group-relative advantages (population sigma) and the coefficients of the batch, float64."""
    adv = np.zeros(len(rewards))
    for b, e in zip(go[:-1], go[1:]):
        r = rewards[b:e].astype(np.float64)
        if r.min() != r.max():
            adv[b:e] = (r - r.mean()) / (r.std() + float(np.float32(ADV_EPS)))
    N, S = int((L > 0).sum()), int(L.sum())
    if agg == R.AGG_TOKEN_MEAN:
        coef = np.where(L > 0, 1.0 / max(S, 1), 0.0)
    else:
        coef = np.where(L > 0, 1.0 / (max(N, 1) * np.maximum(L, 1)), 0.0)
    return adv, coef


def _log_ratios(n, seed, law):
    """delta = logp - old_logp, away from the clip bounds: N(0, 0.1^2), or U[-0.7, 0.7] (edge)."""
    g = _gen(seed, 4)
    d = torch.rand(n, generator=g, device=DEV) * 1.4 - 0.7 if law == "edge" else \
        torch.randn(n, generator=g, device=DEV) * 0.1
    for b in (math.log(1 - EPS_LOW), math.log(1 + EPS_HIGH)):
        d = torch.where((d - b).abs() <= RATIO_BAND, d + 4 * RATIO_BAND, d)
    return d


def _rows_of(rows, V):
    step = max(1, CHUNK_ELEMS // V)
    return [(r, min(rows, r + step)) for r in range(0, rows, step)]


def _logits(case, rows, seed, law):
    """Logits rows in a [rows, ld] buffer, the ids sampled from them, and their log-probs."""
    V, ld = case["V"], case.get("ld", case["V"])
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    z = torch.empty(rows, ld, dtype=dt, device=DEV)[:, :V]
    ids = torch.empty(rows, dtype=torch.int32, device=DEV)
    logp = torch.empty(rows, dtype=torch.float32, device=DEV)
    g = _gen(seed, 2)
    for r0, r1 in _rows_of(rows, V):
        x = torch.randn(r1 - r0, V, generator=g, device=DEV).mul_(case["std"])
        if law == "edge":  # 1% of rows with one +40 logit, 1% with half of their entries at -1e4
            kind = torch.rand(r1 - r0, generator=g, device=DEV)
            spike = torch.nonzero(kind < 0.01).flatten()
            x[spike, torch.randint(0, V, (len(spike),), generator=g, device=DEV)] = 40.0
            low = torch.nonzero(kind > 0.99).flatten()
            x[low] = torch.where(torch.rand(len(low), V, generator=g, device=DEV) < 0.5, -1e4, x[low])
        z[r0:r1] = x
        x = z[r0:r1].float()
        u = torch.rand(r1 - r0, V, generator=g, device=DEV)
        a = u.clamp_(min=1e-30).log_().neg_().log_().neg_().add_(x).argmax(1)
        ids[r0:r1] = a
        logp[r0:r1] = x.gather(1, a[:, None])[:, 0] - torch.logsumexp(x, 1)
    return z, ids, logp


def _t(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def _objective_inputs(case, n, logp, seed):
    """Per-token and per-trajectory inputs of the loss over n rows of the packed stream."""
    lay = _layout(case, seed, T=n)
    L = np.bincount(lay["owner"], weights=lay["mask"], minlength=len(lay["rewards"])).astype(np.int64)
    adv, coef = _advantages64(lay["go"], lay["rewards"], L, R.AGG_SEQ_MEAN_TOKEN_MEAN)
    old = logp - _log_ratios(n, seed, case.get("law", "spans"))
    kl = case["kl"]
    return dict(mask=_t(lay["mask"][:n]), tt=_t(lay["owner"][:n]), adv=_t(adv.astype(np.float32)),
                coef=_t(coef.astype(np.float32)), old=old,
                ref=logp + torch.randn(n, generator=_gen(seed, 5), device=DEV) * 0.2 if kl else None,
                roll=old + torch.randn(n, generator=_gen(seed, 6), device=DEV) * 0.05 if case.get("tis") else None)


def _params(case, agg=R.AGG_SEQ_MEAN_TOKEN_MEAN):
    kl = case.get("kl", 0.0)
    ent = case.get("ent", 0.0) if not isinstance(case.get("ent"), bool) else (1e-3 if case["ent"] else 0.0)
    return R.make_params(EPS_LOW, EPS_HIGH, kl, 3 if kl else 0, ent, TIS_CAP if case.get("tis") else 0.0, ADV_EPS, agg)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "step":
        lay = _layout(case, seed)
        n = int(lay["offs"][-1])
        z, ids, logp = _logits(case, n, seed, "none")
        s.update(z=z, ids=ids, old=logp - _log_ratios(n, seed, "none"), mask=_t(lay["mask"]), go=_t(lay["go"]),
                 offs=_t(lay["offs"]), rewards=_t(lay["rewards"]), lay=lay, params=_params(case),
                 grad=torch.empty_like(z), loss=torch.zeros(1, dtype=torch.float64, device=DEV),
                 ws=R.new_workspace(n, case["V"]))
    elif kind == "loss":
        n = case["rows"]
        z, ids, logp = _logits(case, n, seed, case["law"])
        s.update(z=z, ids=ids, params=_params(case), grad=torch.empty_strided(z.shape, z.stride(), dtype=z.dtype, device=DEV),
                 loss=torch.zeros(1, dtype=torch.float64, device=DEV), ws=R.new_workspace(n, case["V"]),
                 stats=torch.empty(n, 5, dtype=torch.float32, device=DEV) if case["stats"] else None,
                 **_objective_inputs(case, n, logp, seed))
    elif kind == "logprobs":
        z, ids, _ = _logits(case, case["rows"], seed, "none")
        s.update(z=z, ids=ids, ws=R.new_workspace(case["rows"], case["V"]))
    elif kind in ("head_loss", "head_logprobs"):
        T, D, V = case["T"], case["D"], case["V"]
        g = _gen(seed, 3)
        h = torch.randn(T, D, generator=g, device=DEV).bfloat16()
        w = torch.empty(V, D, dtype=torch.bfloat16, device=DEV)
        for v0, v1 in _rows_of(V, D):
            w[v0:v1] = torch.randn(v1 - v0, D, generator=g, device=DEV).mul_(1.28 / math.sqrt(D))
        ids = torch.randint(0, V, (T,), generator=g, device=DEV, dtype=torch.int32)
        s.update(h=h, w=w, ids=ids, ws=R.new_workspace(T, V, D))
        if kind == "head_loss":
            logp = torch.empty(T, device=DEV)
            wf = w.float()
            for r0, r1 in _rows_of(T, V):
                x = h[r0:r1].float() @ wf.T
                logp[r0:r1] = x.gather(1, ids[r0:r1, None].long())[:, 0] - torch.logsumexp(x, 1)
            dh = torch.bfloat16 if case["dh"] == "bf16" else torch.float32
            s.update(params=_params(case), loss=torch.zeros(1, dtype=torch.float64, device=DEV),
                     d_w=torch.zeros(V, D, dtype=torch.float32, device=DEV),
                     d_h=torch.empty(T, D, dtype=dh, device=DEV), **_objective_inputs(dict(case, law="spans"), T, logp, seed))
    else:
        lay = _layout(case, seed)
        if case["packing"] == "owners":  # each rollout's tokens interleaved with its group's others
            p = np.random.default_rng([int(seed) & 0xFFFFFFFF, 18]).permutation(case["size"] * 4)
            order = np.argsort(lay["owner"] // (case["size"] * 4) * len(p) * 64 + p[np.arange(len(lay["owner"])) // 64 % len(p)],
                               kind="stable")
            lay["owner"], lay["mask"] = lay["owner"][order], lay["mask"][order]
        T, g = len(lay["mask"]), _gen(seed, 7)
        old = -1.0 - torch.rand(T, generator=g, device=DEV)
        val = torch.randn(T, generator=g, device=DEV) * 0.25 + 0.3
        stats = torch.rand(T, 5, generator=g, device=DEV) + torch.tensor([-2.0, 0.5, 0.0, 2.0, 0.0], device=DEV)
        stats[:, 2] = ((stats[:, 1] > 1 + EPS_HIGH) | (stats[:, 1] < 1 - EPS_LOW)).float()
        s.update(lay=lay, mask=_t(lay["mask"]), go=_t(lay["go"]), offs=_t(lay["offs"]), rewards=_t(lay["rewards"]),
                 owner=_t(lay["owner"]), old=old, roll=old + torch.randn(T, generator=g, device=DEV) * 0.02, val=val,
                 val_new=val + torch.randn(T, generator=g, device=DEV) * 0.1, stats=stats,
                 params=_params(case, R.AGG_TOKEN_MEAN), ws=R.new_workspace(T, 0),
                 loss=torch.zeros(1, dtype=torch.float64, device=DEV),
                 summary=torch.zeros(5, dtype=torch.float64, device=DEV))
    return s


# ----------------------------------------------------------------------------- one pass

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        adv, coef, n_tok, tt = R.rl_group_advantages(s["go"], s["rewards"], s["offs"], s["mask"], s["params"], s["ws"])
        s["loss"].zero_()
        g = R.rl_policy_loss_fwd_bwd(s["z"], s["ids"], s["mask"], tt, adv, coef, s["old"], s["params"], s["ws"],
                                     s["loss"], grad_out=s["grad"])
        return dict(loss=s["loss"], grad=g, adv=adv, coef=coef, n_tok=n_tok, owner=tt)
    if kind == "loss":
        s["loss"].zero_()
        g = R.rl_policy_loss_fwd_bwd(s["z"], s["ids"], s["mask"], s["tt"], s["adv"], s["coef"], s["old"], s["params"],
                                     s["ws"], s["loss"], grad_out=s["grad"], ref_logp=s["ref"], rollout_logp=s["roll"],
                                     token_stats=s["stats"])
        return dict(loss=s["loss"], grad=g, stats=s["stats"])
    if kind == "logprobs":
        logp, ent, lse = R.rl_token_logprobs(s["z"], s["ids"], s["ws"], want_entropy=case["ent"], want_lse=True)
        return dict(logp=logp, ent=ent, lse=lse)
    if kind == "head_loss":
        s["loss"].zero_()
        s["d_w"].zero_()
        dh = R.rl_fused_head_loss_fwd_bwd(s["h"], s["w"], s["ids"], s["mask"], s["tt"], s["adv"], s["coef"], s["old"],
                                          s["params"], s["ws"], s["loss"], s["d_w"], d_hidden=s["d_h"], ref_logp=s["ref"])
        return dict(loss=s["loss"], d_h=dh, d_w=s["d_w"])
    if kind == "head_logprobs":
        logp, ent, lse = R.rl_fused_head_token_logprobs(s["h"], s["w"], s["ids"], s["ws"], want_entropy=case["ent"],
                                                        want_lse=True)
        return dict(logp=logp, ent=ent, lse=lse)
    n = s["rewards"].numel()
    if case["packing"] == "spans":
        adv, coef, n_tok, tt = R.rl_group_advantages(s["go"], s["rewards"], s["offs"], s["mask"], s["params"], s["ws"])
    else:
        tt = s["owner"]
        adv, coef, n_tok = R.rl_group_advantages_by_owner(s["go"], s["rewards"], tt, s["mask"], s["params"], s["ws"])
    w, ratio = R.rl_sequence_is_weights(tt, s["mask"], s["old"], s["roll"], n, s["ws"], cap=case["cap"],
                                        want_log_ratio=True, traj_adv_inout=adv)
    if case["packing"] == "spans":
        tadv, ret = R.rl_masked_gae(s["offs"], s["mask"], s["val"], s["ws"], case["gamma"], case["lam"], True,
                                    traj_rewards=s["rewards"])
    else:
        tadv, ret = R.rl_rollout_value_advantages(tt, s["mask"], s["val"], s["rewards"], s["ws"])
    s["loss"].zero_()
    s["summary"].zero_()
    d_v = R.rl_value_loss_fwd_bwd(s["val_new"], ret, s["mask"], tt, coef, s["ws"], s["loss"])
    R.rl_token_stats_summary(s["stats"], s["mask"], tt, coef, s["ws"], s["summary"])
    return dict(adv=adv, coef=coef, n_tok=n_tok, owner=tt, weight=w, log_ratio=ratio, token_adv=tadv, returns=ret,
                value_loss=s["loss"], d_values=d_v, summary=s["summary"])


# ----------------------------------------------------------------------------- what a pass cannot do without

# share of the rows that are trained on, by the law of the mask
ACTIVE = {"none": 1.0, "spans": 0.62, "edge": 0.62}


def work(case):
    kind = case["kind"]
    if kind == "step":
        T = case["groups"] * case["size"] * (case["lo"] + case["hi"]) / 2
        return dict(bytes=T * (2 * case["V"] * 2 + 17), flops=T * case["V"] * 8)
    if kind in ("loss", "logprobs"):
        es = 2 if case["dtype"] == "bf16" else 4
        n = case["rows"] * case["V"]
        if kind == "logprobs":
            return dict(bytes=n * es + case["rows"] * 16, flops=n * 4)
        on = ACTIVE[case["law"]]
        return dict(bytes=n * es * (1 + on) + case["rows"] * 17, flops=n * on * 8)
    if kind in ("head_loss", "head_logprobs"):
        T, D, V = case["T"], case["D"], case["V"]
        if kind == "head_logprobs":
            return dict(bytes=2 * D * (T + V) + 16 * T, flops=2 * T * D * V)
        # only trained tokens have a loss and a gradient
        return dict(bytes=4 * D * T + 2 * D * V + 4 * D * V, flops=6 * T * D * V * ACTIVE["spans"])
    mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"]) if case["hi"] > case["lo"] else case["lo"]
    T = case["groups"] * case["size"] * mean
    # mask, owner (written and read), log-probs, values, returns, advantages, statistics, d values
    return dict(bytes=T * 50 + case["groups"] * case["size"] * 40, flops=T * 40)


def tolerance(case):
    kind = case["kind"]
    if kind in ("step", "loss"):
        # bf16 gradients round once (2^-9 of each value on average over its binade, 2^-8 at most)
        return {"rel": 7e-3, "max": 1.6e-2} if case["dtype"] == "bf16" else {"rel": 1e-5, "max": 4e-4}
    if kind == "head_loss":
        # dZ rounds twice to bf16, the products sum them in fp32, d hidden rounds again
        return {"rel": 1e-2, "max": 1e-1}
    return {"rel": 1e-5, "max": 4e-4}


# ----------------------------------------------------------------------------- the results in 64 bits

def _terms64(logp, H, s, ent, kl, tis):
    """Per-token loss and d loss / d logp (Sec. 2.3.2 with the k3 KL and the rollout weight)."""
    tt = s["tt"].long()
    A, c = s["adv"].double()[tt], s["coef"].double()[tt]
    on = (s["mask"] != 0) & (c != 0)
    rho = torch.exp(logp - s["old"].double())
    lo, hi = 1.0 - float(np.float32(EPS_LOW)), 1.0 + float(np.float32(EPS_HIGH))
    surr = torch.minimum(rho * A, rho.clamp(lo, hi) * A)
    cut = ((A > 0) & (rho > hi)) | ((A < 0) & (rho < lo))
    w = torch.exp(s["old"].double() - s["roll"].double()).clamp(max=TIS_CAP) if tis else torch.ones_like(A)
    beta, alpha = float(np.float32(kl)), float(np.float32(ent))
    K, dK = torch.zeros_like(A), torch.zeros_like(A)
    if kl:
        d = s["ref"].double() - logp
        K, dK = torch.exp(d) - d - 1, 1 - torch.exp(d)
    ell = -w * surr + beta * K - alpha * H
    g = torch.where(cut, torch.zeros_like(A), -w * A * rho) + beta * dK
    z = torch.zeros_like(A)
    stats = torch.stack([logp, rho, cut.double(), H, K], 1) * on[:, None]
    return torch.where(on, c, z), torch.where(on, c * ell, z).sum().reshape(1), g, alpha, stats


def _softmax64(x, ids):
    x = x.double()
    lse = torch.logsumexp(x, 1)
    lp = x - lse[:, None]
    p = lp.exp()
    H = -torch.where(p > 0, p * lp, torch.zeros_like(p)).sum(1)
    return x.gather(1, ids.long()[:, None])[:, 0] - lse, H, lse, p, lp


def _dz64(p, lp, H, ids, c, g, alpha):
    """c [g (delta_a - p) + alpha p (log p + H)] per row."""
    dz = p * (-g[:, None])
    if alpha:
        dz += alpha * torch.where(p > 0, p * (lp + H[:, None]), torch.zeros_like(p))
    dz.scatter_add_(1, ids.long()[:, None], g[:, None])
    return dz * c[:, None]


def _loss64(s, logits_of, n, V, ent, kl, tis, grad_of):
    """Two passes over blocks of rows: the softmax statistics, then the gradient of the logits."""
    logp, H = torch.empty(n, dtype=torch.float64, device=DEV), torch.empty(n, dtype=torch.float64, device=DEV)
    blocks = _rows_of(n, V)
    for r0, r1 in blocks:
        logp[r0:r1], H[r0:r1] = _softmax64(logits_of(r0, r1), s["ids"][r0:r1])[:2]
    c, loss, g, alpha, stats = _terms64(logp, H, s, ent, kl, tis)
    for r0, r1 in blocks:
        _, h, _, p, lp = _softmax64(logits_of(r0, r1), s["ids"][r0:r1])
        grad_of(r0, r1, _dz64(p, lp, h, s["ids"][r0:r1], c[r0:r1], g[r0:r1], alpha))
    return loss, stats


def _exact_logits(s, ent, kl, tis):
    n, V = s["z"].shape
    grad = torch.empty(n, V, dtype=torch.float64, device=DEV)

    def put(r0, r1, dz):
        grad[r0:r1] = dz
    loss, stats = _loss64(s, lambda r0, r1: s["z"][r0:r1], n, V, ent, kl, tis, put)
    return loss, grad, stats


def _exact_head(case, s):
    """float64 products; d W is left out (None) where the three together would take too long."""
    T, D, V = case["T"], case["D"], case["V"]
    flops = 2.0 * T * D * V
    if flops > 1e13:
        return None
    w = s["w"].double()
    if case["kind"] == "head_logprobs":
        out = [torch.empty(T, dtype=torch.float64, device=DEV) for _ in range(3)]
        for r0, r1 in _rows_of(T, V):
            logp, H, lse, _, _ = _softmax64(s["h"][r0:r1].double() @ w.T, s["ids"][r0:r1])
            for o, x in zip(out, (logp, H, lse)):
                o[r0:r1] = x
        return dict(logp=out[0], ent=out[1] if case["ent"] else None, lse=out[2])
    want_w = flops <= 3e12
    d_h = torch.empty(T, D, dtype=torch.float64, device=DEV)
    d_w = torch.zeros(V, D, dtype=torch.float64, device=DEV) if want_w else None
    z = torch.empty(T, V, dtype=torch.float64, device=DEV)
    for r0, r1 in _rows_of(T, V):
        z[r0:r1] = s["h"][r0:r1].double() @ w.T

    def put(r0, r1, dz):
        d_h[r0:r1] = dz @ w
        if want_w:
            d_w.addmm_(dz.T, s["h"][r0:r1].double())
    loss, _ = _loss64(s, lambda r0, r1: z[r0:r1], T, V, 1e-3 if case["ent"] else 0.0, case["kl"], False, put)
    return dict(loss=loss, d_h=d_h, d_w=d_w)


def _exact_batch(case, s):
    lay = s["lay"]
    owner, M, offs = lay["owner"], lay["mask"] != 0, lay["offs"]
    n = len(lay["rewards"])
    Ri = lay["rewards"].astype(np.float64)
    L = np.bincount(owner, weights=M, minlength=n).astype(np.int64)
    adv, coef = _advantages64(lay["go"], lay["rewards"], L, R.AGG_TOKEN_MEAN)
    f = {k: s[k].double().cpu().numpy() for k in ("old", "roll", "val", "val_new", "stats")}
    S = np.bincount(owner, weights=np.where(M, f["old"] - f["roll"], 0.0), minlength=n)
    w = np.exp(S)
    if case["cap"] > 0:
        w = np.minimum(w, float(np.float32(case["cap"])))
    V = f["val"]
    if case["packing"] == "owners":
        tadv, ret = np.where(M, Ri[owner] - V, 0.0), np.where(M, Ri[owner], 0.0)
    else:  # the backward recursion over trainable tokens, all trajectories at once
        gamma = float(np.float32(case["gamma"]))
        gl = float(np.float32(case["gamma"]) * np.float32(case["lam"]))
        tadv, ret = np.zeros(len(V)), np.zeros(len(V))
        x, vn, seen = np.zeros(n), np.zeros(n), np.zeros(n, bool)
        for back in range(1, int((offs[1:] - offs[:-1]).max()) + 1):
            t = offs[1:] - back
            i = np.nonzero(t >= offs[:-1])[0]
            i = i[M[t[i]]]
            t = t[i]
            x[i] = np.where(seen[i], 0.0, Ri[i]) + gamma * vn[i] - V[t] + gl * x[i]
            vn[i], seen[i] = V[t], True
            tadv[t], ret[t] = x[i], x[i] + V[t]
    c = np.where(M, coef[owner], 0.0)
    d = f["val_new"] - ret
    on = c != 0
    st = f["stats"][on]
    summary = np.array([on.sum(), st[:, 2].sum(), st[:, 3].sum(), st[:, 4].sum(), st[:, 1].sum()], np.float64)
    return dict(adv=adv * w, coef=coef, n_tok=None, owner=None, weight=w, log_ratio=S, token_adv=tadv, returns=ret,
                value_loss=np.array([(c * d * d).sum()]), d_values=2 * c * d, summary=summary)


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "step":
        lay = s["lay"]
        L = np.bincount(lay["owner"], weights=lay["mask"], minlength=len(lay["rewards"])).astype(np.int64)
        adv, coef = _advantages64(lay["go"], lay["rewards"], L, R.AGG_SEQ_MEAN_TOKEN_MEAN)
        s.update(adv=_t(adv), coef=_t(coef), tt=_t(lay["owner"]))
        loss, grad, _ = _exact_logits(s, 0.0, 0.0, False)
        return dict(loss=loss, grad=grad, adv=adv, coef=coef, n_tok=None, owner=None)
    if kind == "loss":
        loss, grad, stats = _exact_logits(s, case["ent"], case["kl"], case["tis"])
        return dict(loss=loss, grad=grad, stats=stats if case["stats"] else None)
    if kind == "logprobs":
        out = [torch.empty(case["rows"], dtype=torch.float64, device=DEV) for _ in range(3)]
        for r0, r1 in _rows_of(case["rows"], case["V"]):
            logp, H, lse, _, _ = _softmax64(s["z"][r0:r1], s["ids"][r0:r1])
            for o, x in zip(out, (logp, H, lse)):
                o[r0:r1] = x
        return dict(logp=out[0], ent=out[1] if case["ent"] else None, lse=out[2])
    if kind in ("head_loss", "head_logprobs"):
        return _exact_head(case, s)
    return _exact_batch(case, s)
