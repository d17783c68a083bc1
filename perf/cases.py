"""What a user of this library runs, as cases that can be timed and compared.

A training program builds the segment layout of a batch of trajectories, gathers the packed
Q, K and V rows (or reads them through the gather map), runs the attention forward and
backward, and evaluates the RL objective over the segments' token streams.  Each case is one of
those calls, or a whole small step, on layouts drawn like the library's own workloads: a
trajectory of `steps` steps, each a screenshot of `img` tokens and a response of `txt` tokens,
cut with `window` new and `keep` retained screenshots.

The step counts that fix a case's shapes come from its own `shape` number, the tensors from the
seed; a layout case's inputs are the step counts, which the seed deals in another order.
"""
import math

import numpy as np
import torch

from paper_2607_11185_gb300 import vcs

DEV = "cuda"


def _case(name, kind, traj, steps, img, txt, window, keep, heads=(0, 0, 0), outliers=False, shape=1):
    return dict(name=name, kind=kind, traj=traj, steps_lo=steps[0], steps_hi=steps[1], img_lo=img[0], img_hi=img[1],
                txt_lo=txt[0], txt_hi=txt[1], window=window, keep=keep, hq=heads[0], hkv=heads[1], d=heads[2],
                outliers=outliers, shape=shape)


def listed():
    short = ((5, 15), (1024, 1024), (64, 256))        # eight short rollouts: steps, img, txt
    mixed = ((10, 50), (1500, 2700), (64, 512))       # full-screen rollouts of up to 50 steps
    long = ((50, 50), (2700, 2700), (512, 512))       # long-horizon rollouts
    return [
        # the layout of one small batch, rebuilt for every batch of rollouts: launches and latency
        _case("layout_small", "layout", 8, *short, 3, 0),
        # the layout of a whole collection of long rollouts at once (126 M segment tokens)
        _case("layout_batch", "layout", 512, *long, 8, 0),
        # the packed Q/K/V rows of one long rollout, at the largest row size
        _case("gather_long", "gather", 1, *long, 8, 0, (40, 8, 128)),
        # a whole step (layout, gather, forward, backward) of one four-step rollout through the
        # allocating calls: what a debugging run or the smallest model does, latency only
        _case("step_tiny", "step", 1, (4, 4), (256, 256), (32, 32), 2, 0, (2, 1, 64)),
        # forward (reference-policy log-probabilities, scoring) over a small batch of rollouts
        _case("fwd_short", "fwd", 8, *short, 3, 0, (28, 4, 128), shape=2),
        # the backward of that batch's actor update
        _case("bwd_short", "bwd", 8, *short, 3, 0, (28, 4, 128), shape=2),
        # forward and backward over the longest segments (25,696 to 46,176 tokens), with the
        # large-logit keys of such contexts
        _case("fwd_long", "fwd", 1, *long, 8, 0, (40, 8, 128), outliers=True),
        _case("bwd_long", "bwd", 1, *long, 8, 0, (40, 8, 128), outliers=True),
        # the training pass of a model with 64-wide heads on the small batch
        _case("train_d64", "train", 8, *short, 3, 0, (14, 2, 64), shape=2),
        # the training pass without segment-layout copies of Q/K/V, one screenshot retained
        _case("train_gathered", "gathered", 8, *short, 3, 1, (28, 4, 128), shape=2),
        # forward scoring that computes the rows consecutive segments share once, step-wise layout
        _case("fwd_reuse_stepwise", "reuse", 1, *mixed, 1, 0, (28, 4, 128), shape=6),
        # token stream, trainable tokens, group advantages and the RL objective over 2 M tokens
        _case("objective", "objective", 8, *long, 8, 0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))

    kind = rng.choice(["layout", "gather", "step", "fwd", "bwd", "fwd", "bwd", "train", "gathered", "reuse",
                       "objective"])
    d = rng.choice([64, 128, 128])
    hkv = rng.choice([1, 2, 4, 8])
    hq = hkv * rng.choice([1, 2, 3, 5, 7])
    traj = {"layout": log_int(8, 512), "objective": log_int(1, 512), "step": 1}.get(kind, log_int(1, 16))
    lo, img, txt = rng.randint(1, 50), log_int(200, 2700), log_int(16, 512)
    if kind == "step":
        lo, img, txt = rng.randint(1, 8), log_int(64, 512), log_int(16, 128)
    window, keep = rng.choice([1, 2, 3, 5, 8]), rng.choice([0, 0, 1, 5, 8])
    while True:
        c = _case("", kind, traj, (max(1, lo // 2), lo), (max(1, img // 2), img), (max(1, txt // 4), txt), window,
                  keep, (hq, hkv, d) if kind not in ("layout", "objective") else (0, 0, 0),
                  outliers=d == 128 and rng.random() < 0.3, shape=rng.randrange(1, 1 << 20))
        del c["name"]
        w = work(c)
        if w["flops"] <= 1.5e13 and w["bytes"] <= 7e9:
            return c
        if traj > 1:  # too large: fewer rollouts, then shorter ones
            traj = max(1, traj // 2)
        else:
            lo = max(1, lo * 2 // 3)


# ---------------------------------------------------------------- shapes (host arithmetic)

def _steps(case, seed):
    """cu_steps, step_img, step_txt (int32).  Attention shapes depend on the case alone."""
    rng = np.random.default_rng(case["shape"])
    t = rng.integers(case["steps_lo"], case["steps_hi"], size=case["traj"], endpoint=True)
    n = int(t.sum())
    img = rng.integers(case["img_lo"], case["img_hi"], size=n, endpoint=True).astype(np.int32)
    txt = rng.integers(case["txt_lo"], case["txt_hi"], size=n, endpoint=True).astype(np.int32)
    cu = np.concatenate([[0], np.cumsum(t)])
    if case["kind"] == "layout":
        # a fixed screen still yields a few tokens more or fewer after patch merging; the seed
        # deals the same rollouts in another order, so that the outputs keep their sizes
        img = np.maximum(img + rng.integers(-8, 8, size=n, endpoint=True).astype(np.int32), 1)
        perm = np.random.default_rng(seed).permutation(case["traj"])
        order = np.concatenate([np.arange(cu[b], cu[b + 1]) for b in perm])
        img, txt, cu = img[order], txt[order], np.concatenate([[0], np.cumsum(t[perm])])
    return cu.astype(np.int32), img, txt


def _segments(case, seed):
    """Per segment (trajectory, its first step, first step with a screenshot, first new step, end)."""
    cu, _, _ = _steps(case, seed)
    first, step = case["keep"] + case["window"], case["window"]
    out = []
    for b in range(case["traj"]):
        g0, g1 = int(cu[b]), int(cu[b + 1])
        s = g0
        while s < g1:
            e = min(s + (first if s == g0 else step), g1)
            out.append((b, g0, max(g0, s - case["keep"]), s, e))
            s = e
    return out


def _lengths(case, seed=0):
    _, img, txt = _steps(case, seed)
    ct = np.concatenate([[0], np.cumsum(txt, dtype=np.int64)])
    ci = np.concatenate([[0], np.cumsum(img, dtype=np.int64)])
    return np.array([ct[e] - ct[g0] + ci[e] - ci[a] for _, g0, a, _, e in _segments(case, seed)], np.int64)


def _layout(case, seed):
    """The whole layout in numpy: cu_seqlens, seg_traj, gather, source step, position, mask."""
    _, img, txt = _steps(case, seed)
    off = np.concatenate([[0], np.cumsum(img.astype(np.int64) + txt)])
    cu, traj, gat, src, pos, msk = [0], [], [], [], [], []
    for b, g0, a, s, e in _segments(case, seed):
        n0 = cu[-1]
        parts = [(u, off[u] + (img[u] if u < a else 0), off[u + 1]) for u in range(g0, e)]
        for u, lo, hi in parts:
            gat.append(np.arange(lo, hi, dtype=np.int32))
            src.append(np.full(hi - lo, u, np.int32))
            msk.append(((gat[-1] >= off[u] + img[u]) & (u >= s)).astype(np.uint8))
            n0 += int(hi - lo)
        pos.append(np.arange(n0 - cu[-1], dtype=np.int32))
        cu.append(n0)
        traj.append(b)
    cat = np.concatenate
    return np.array(cu, np.int32), np.array(traj, np.int32), cat(gat), cat(src), cat(pos), cat(msk)


# ---------------------------------------------------------------- state

def _randn(gen, shape):
    out = torch.empty(shape, dtype=torch.bfloat16, device=DEV)
    for r in range(0, shape[0], 1 << 15):
        out[r:r + (1 << 15)] = torch.randn((min(1 << 15, shape[0] - r),) + shape[1:], generator=gen, device=DEV)
    return out


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _qkv(case, seed, rows):
    g = _gen(seed)
    q = _randn(g, (rows, case["hq"], case["d"]))
    k = _randn(g, (rows, case["hkv"], case["d"]))
    v = _randn(g, (rows, case["hkv"], case["d"]))
    if case["outliers"]:  # 5% of the keys with logits eight times as large
        k.mul_(torch.where(torch.rand(k.shape[:2], generator=g, device=DEV) < 0.05, 8.0, 1.0).bfloat16()[..., None])
    return q, k, v, g


def _objective_inputs(case, seed, traj_tokens, tokens):
    g = _gen(seed)
    n = case["traj"]
    lp = -torch.rand(tokens, generator=g, device=DEV) * 3
    return dict(traj_ids=torch.randint(0, 150000, (traj_tokens,), generator=g, device=DEV, dtype=torch.int32),
                traj_logp=-torch.rand(traj_tokens, generator=g, device=DEV) * 3, new=lp,
                # an importance ratio that leaves [0.8, 1.28] for some tokens
                old=lp + 0.2 * torch.randn(tokens, generator=g, device=DEV),
                ref=lp + 0.1 * torch.randn(tokens, generator=g, device=DEV),
                rewards=(torch.rand(n, generator=g, device=DEV) < 0.4).float())


def _dev(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in arrays]


def prepare(case, seed):
    st = dict(case=case)
    kind = case["kind"]
    cu_steps, img, txt = _steps(case, seed)
    st["steps"] = _dev(cu_steps, img, txt)
    traj_tokens = int(img.sum(dtype=np.int64) + txt.sum(dtype=np.int64))
    if kind == "layout":
        return st
    if kind == "step":  # dO arrives after the forward in a real step; here it is drawn beforehand
        st["q"], st["k"], st["v"], g = _qkv(case, seed, traj_tokens)
        st["do"] = _randn(g, (int(_lengths(case).sum()), case["hq"], case["d"]))
        return st
    lay = vcs.build_segments(*st["steps"], case["window"], case["keep"])
    st["lay"] = lay
    ns, nt, mx = lay["num_segments"], lay["num_tokens"], lay["max_seqlen"]
    hq, hkv, d = case["hq"], case["hkv"], case["d"]
    if kind == "objective":
        st["in"] = _objective_inputs(case, seed, traj_tokens, nt)
        return st
    in_traj = kind in ("gather", "gathered", "reuse")
    st["q"], st["k"], st["v"], g = _qkv(case, seed, traj_tokens if in_traj else nt)
    if kind == "reuse":  # the packed rows are copies of the rollout's rows, so prefixes repeat
        st["q"], st["k"], st["v"] = (x[lay["tok_gather"].long()] for x in (st["q"], st["k"], st["v"]))
    if kind == "gather":
        st["out"] = [torch.empty((nt, h, d), dtype=torch.bfloat16, device=DEV) for h in (hq, hkv, hkv)]
        st["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        return st
    nb = vcs.vcs_attn_fwd_workspace_size(ns, nt, mx, hq, hkv, d)
    st["o"] = torch.empty((nt, hq, d), dtype=torch.bfloat16, device=DEV)
    st["lse"] = torch.empty((hq, nt), dtype=torch.float32, device=DEV)
    if kind in ("bwd", "train", "gathered"):
        st["do"] = _randn(g, (nt, hq, d))
        st["grads"] = [torch.empty_like(st[x]) for x in ("q", "k", "v")]
        nb = max(nb, vcs.vcs_attn_bwd_gathered_workspace_size(ns, nt, mx, traj_tokens, hq, hkv, d)
                 if kind == "gathered" else vcs.vcs_attn_bwd_workspace_size(ns, nt, mx, hq, hkv, d))
    st["ws"], st["ws_bytes"] = torch.empty(nb, dtype=torch.uint8, device=DEV), nb
    if kind == "reuse":
        st["shared"] = torch.empty(ns, dtype=torch.int32, device=DEV)
    if kind == "bwd":  # the backward's inputs are a forward's outputs
        _fwd(st)
    return st


def _ok(status):
    if status != 0:
        raise RuntimeError(vcs.vcs_status_string(status))


def _dims(st):
    c, lay = st["case"], st["lay"]
    return (lay["num_segments"], lay["num_tokens"], lay["max_seqlen"], c["hq"], c["hkv"], c["d"], 0.0)


def _fwd(st):
    _ok(vcs.vcs_attn_fwd(st["q"], st["k"], st["v"], st["lay"]["cu_seqlens"], *_dims(st), st["o"], st["lse"],
                         st["ws"], st["ws_bytes"]))


def _bwd(st):
    _ok(vcs.vcs_attn_bwd(st["q"], st["k"], st["v"], st["o"], st["lse"], st["do"], st["lay"]["cu_seqlens"],
                         *_dims(st), *st["grads"], st["ws"], st["ws_bytes"]))


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "layout":
        lay = vcs.build_segments(*state["steps"], case["window"], case["keep"])
        return [lay[n] for n in ("cu_seqlens", "seg_traj", "tok_gather", "tok_src_step", "tok_pos", "tok_loss_mask")]
    if kind == "step":
        lay = vcs.build_segments(*state["steps"], case["window"], case["keep"])
        q, k, v = vcs.gather(state["q"], state["k"], state["v"], lay["tok_gather"])
        o, lse = vcs.attn_fwd(q, k, v, lay["cu_seqlens"], lay["max_seqlen"])
        return [o, lse, *vcs.attn_bwd(q, k, v, o, lse, state["do"], lay["cu_seqlens"], lay["max_seqlen"])]
    lay = state["lay"]
    if kind == "gather":
        _ok(vcs.vcs_gather(state["q"], state["k"], state["v"], state["q"].shape[0], lay["tok_gather"],
                           lay["num_tokens"], case["hq"], case["hkv"], case["d"], *state["out"], state["status"]))
        return state["out"]
    if kind == "fwd":
        _fwd(state)
        return [state["o"], state["lse"]]
    if kind == "bwd":
        _bwd(state)
        return state["grads"]
    if kind == "train":
        _fwd(state)
        _bwd(state)
        return [state["o"], state["lse"], *state["grads"]]
    if kind == "gathered":
        qkv = (state["q"], state["k"], state["v"], state["q"].shape[0], lay["tok_gather"])
        _ok(vcs.vcs_attn_fwd_gathered(*qkv, lay["cu_seqlens"], *_dims(state), state["o"], state["lse"], state["ws"],
                                      state["ws_bytes"]))
        _ok(vcs.vcs_attn_bwd_gathered(*qkv, state["o"], state["lse"], state["do"], lay["cu_seqlens"], *_dims(state),
                                      *state["grads"], state["ws"], state["ws_bytes"]))
        return [state["o"], state["lse"], *state["grads"]]
    if kind == "reuse":
        _ok(vcs.vcs_shared_prefix(lay["cu_seqlens"], lay["seg_traj"], lay["tok_gather"], lay["num_segments"],
                                  lay["num_tokens"], state["shared"]))
        _ok(vcs.vcs_attn_fwd_reuse(state["q"], state["k"], state["v"], lay["cu_seqlens"], state["shared"],
                                   *_dims(state), state["o"], state["lse"], state["ws"], state["ws_bytes"]))
        return [state["shared"], state["o"], state["lse"]]
    i = state["in"]
    ids, logp = vcs.stream_fields(i["traj_ids"], i["traj_logp"], lay["tok_gather"], lay["tok_loss_mask"])
    idx = vcs.compact_trainable(lay["tok_loss_mask"])
    adv = vcs.group_advantage(i["rewards"], case["traj"])
    loss, dlogp = vcs.grpo_loss(i["new"], i["old"], i["ref"], lay["tok_loss_mask"], lay["cu_seqlens"],
                                lay["seg_traj"], adv)
    return [ids, logp, idx, adv, loss, dlogp]


# ---------------------------------------------------------------- work, tolerance, exact values

def work(case):
    lens = _lengths(case)
    nt, ns = int(lens.sum()), len(lens)
    _, img, txt = _steps(case, 0)
    tt, n = int(img.sum(dtype=np.int64) + txt.sum(dtype=np.int64)), len(img)
    hq, hkv, d = case["hq"], case["hkv"], case["d"]
    layout, row, lse = 13 * nt + 8 * ns + 8 * n, (hq + 2 * hkv) * d * 2, 4 * hq * nt
    pairs = float((lens * (lens + 1) // 2).sum()) * hq * d
    o = 2 * hq * d * nt
    kind = case["kind"]
    if kind == "layout":
        return {"bytes": layout, "flops": 0}
    if kind == "gather":
        return {"bytes": (tt + nt) * row + 4 * nt, "flops": 0}
    if kind == "objective":
        trainable = int(txt.sum(dtype=np.int64))
        return {"bytes": 4 * tt + (4 + 1 + 8 + 4) * nt + (4 + 4 + 12) * trainable, "flops": 0}
    if kind == "fwd":
        return {"bytes": nt * row + o + lse, "flops": 4 * pairs}
    if kind == "reuse":
        seg, ct = _segments(case, 0), np.concatenate([[0], np.cumsum(txt, dtype=np.int64)])
        # rows already in the previous segment: the history it carried as text
        shared = [0] + [int(ct[p[2]] - ct[p[1]]) if p[0] == s[0] else 0 for p, s in zip(seg, seg[1:])]
        pairs -= float(sum(x * (x + 1) // 2 for x in shared)) * hq * d
        return {"bytes": nt * row + o + lse + 4 * nt, "flops": 4 * pairs}
    if kind == "bwd":
        return {"bytes": 2 * nt * row + 2 * o + lse, "flops": 8 * pairs}
    if kind == "train":
        return {"bytes": 2 * nt * row + 2 * o + lse, "flops": 12 * pairs}
    if kind == "gathered":
        return {"bytes": 2 * tt * row + 2 * o + lse + 4 * nt, "flops": 12 * pairs}
    return {"bytes": layout + 2 * tt * row + 2 * nt * row + 2 * o + lse, "flops": 12 * pairs}  # step


def tolerance(case):
    kind = case["kind"]
    if kind in ("layout", "gather"):
        return "exact"
    if kind == "objective":  # fp32 terms, fp64 sum
        return {"rel": 1e-5}
    # bf16 P, dS and outputs: 0.002 to 0.0025 of each output's norm measured against fp64, up to
    # 0.0065 for gradients over segments of a few tile rows, where few terms average
    return {"rel": 1e-2 if kind in ("fwd", "reuse") or _lengths(case).mean() >= 1000 else 2.5e-2}


def _attention64(q, k, v, lens, do=None):
    """fp64 attention over packed segments, in query blocks; the gradients too when do is given."""
    nt, hq, d = q.shape
    hkv, scale = k.shape[1], 1 / math.sqrt(d)
    o = torch.empty((nt, hq, d), dtype=torch.float64, device=DEV)
    lse = torch.empty((hq, nt), dtype=torch.float64, device=DEV)
    grads = [torch.zeros(x.shape, dtype=torch.float64, device=DEV) for x in (q, k, v)] if do is not None else None
    s0 = 0
    for n in lens.tolist():
        for h in range(hq):
            g = h // (hq // hkv)
            kh, vh = k[s0:s0 + n, g].double(), v[s0:s0 + n, g].double()
            for a in range(0, n, 1024):
                b = min(a + 1024, n)
                qh = q[s0 + a:s0 + b, h].double()
                s = qh @ kh[:b].T * scale
                s[:, a:b].masked_fill_(torch.ones((b - a, b - a), dtype=torch.bool, device=DEV).triu_(1), -math.inf)
                l = torch.logsumexp(s, 1)
                p = s.sub_(l[:, None]).exp_()
                oh = p @ vh[:b]
                o[s0 + a:s0 + b, h], lse[h, s0 + a:s0 + b] = oh, l
                if do is not None:
                    dh = do[s0 + a:s0 + b, h].double()
                    grads[2][s0:s0 + b, g] += p.T @ dh
                    ds = p.mul_((dh @ vh[:b].T).sub_((dh * oh).sum(1, keepdim=True))).mul_(scale)
                    grads[0][s0 + a:s0 + b, h] = ds @ kh[:b]
                    grads[1][s0:s0 + b, g] += ds.T @ qh
        s0 += n
    return o, lse, grads


def _objective64(case, seed, lay):
    cu, seg_traj, gat, _, _, msk = lay
    _, img, txt = _steps(case, seed)
    i = _objective_inputs(case, seed, int(img.sum(dtype=np.int64) + txt.sum(dtype=np.int64)), len(gat))
    gat, msk, cu, seg_traj = _dev(gat.astype(np.int64), msk, cu.astype(np.int64), seg_traj.astype(np.int64))
    on = msk != 0
    r = i["rewards"].double()
    adv = (r - r.mean()) / (r.std(correction=0) + 1e-6)
    a = adv.float().double()[seg_traj.repeat_interleave(cu.diff())]
    new, old, ref = (i[x].double() for x in ("new", "old", "ref"))
    # the ratio's logarithm is the fp32 difference of the two inputs, as the call defines it
    rho = (i["new"] - i["old"]).double().exp()
    lo, hi, cap = float(np.float32(0.8)), float(np.float32(1.28)), 3.0
    pos = a >= 0
    live = torch.where(pos, rho <= hi, (rho >= lo) & (rho <= cap))
    flat = torch.where(pos, hi, torch.where(rho < lo, lo, cap))
    kl, e = float(np.float32(1e-4)), torch.expm1((i["ref"] - i["new"]).double())
    obj = torch.where(live, rho, flat) * a
    loss = torch.where(on, -obj + kl * (e - (ref - new)), 0.0).sum()[None] / case["traj"]
    dlogp = torch.where(on, -torch.where(live, rho * a, 0.0) - kl * e, 0.0) / case["traj"]
    return [i["traj_ids"][gat], torch.where(on, i["traj_logp"][gat], 0.0), on.nonzero()[:, 0].int(), adv, loss, dlogp]


def exact(case, seed):
    kind = case["kind"]
    w = work(case)
    if w["flops"] > 1.2e13 or w["bytes"] > 1.6e9 and kind in ("layout", "gather"):
        return None
    lay = _layout(case, seed)
    if kind == "layout":
        return _dev(*lay)
    if kind == "objective":
        return _objective64(case, seed, lay)
    gat, lens = _dev(lay[2].astype(np.int64))[0], _lengths(case)
    _, img, txt = _steps(case, seed)
    tt, nt = int(img.sum(dtype=np.int64) + txt.sum(dtype=np.int64)), len(lay[2])
    packed = kind in ("fwd", "bwd", "train")
    q, k, v, g = _qkv(case, seed, nt if packed else tt)
    if not packed:
        q, k, v = q[gat], k[gat], v[gat]
    if kind == "gather":
        return [q, k, v]
    do = None if kind in ("fwd", "reuse") else _randn(g, (nt, case["hq"], case["d"]))
    o, lse, grads = _attention64(q, k, v, lens, do)
    if kind == "fwd":
        return [o, lse]
    if kind == "reuse":
        cu, seg_traj = lay[0], lay[1]
        shared = np.zeros(len(lens), np.int32)
        for s in range(1, len(lens)):
            if seg_traj[s] == seg_traj[s - 1]:
                n = int(min(lens[s], lens[s - 1]))
                same = lay[2][cu[s]:cu[s] + n] == lay[2][cu[s - 1]:cu[s - 1] + n]
                shared[s] = n if same.all() else int(np.argmin(same))
        return [_dev(shared)[0], o, lse]
    if kind == "bwd":
        return grads
    if kind == "gathered":  # a rollout row's gradient is the sum over its copies
        grads = [torch.zeros((tt,) + x.shape[1:], dtype=torch.float64, device=DEV).index_add_(0, gat, x)
                 for x in grads]
    return [o, lse, *grads]
