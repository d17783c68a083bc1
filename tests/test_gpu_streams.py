"""The allocating calls on a stream of the caller's choice, given in any form the raw calls take."""
import types

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

BUSY = 40_000_000  # cycles a stream is kept busy ahead of a call, about 20 ms


def inputs():
    g = torch.Generator(device="cuda").manual_seed(7)
    cu, img, txt = (torch.tensor(x, dtype=torch.int32, device="cuda")
                    for x in ([0, 3, 7], [40, 33, 57, 64, 20, 90, 31], [9, 12, 5, 30, 7, 8, 16]))
    rows = int((img + txt).sum())
    q, k, v = (torch.randn((rows, h, 64), generator=g, device="cuda").bfloat16() for h in (2, 1, 1))
    return cu, img, txt, q, k, v


def calls(x, stream):
    """Every allocating call with the given stream; the results as one flat list."""
    from paper_2607_11185_gb300 import vcs
    cu, img, txt, q, k, v = x
    kw = {} if stream is None else dict(stream=stream)
    out = [torch.tensor(vcs.plan_segments(cu, img, txt, 2, 1, **kw))]
    lay = vcs.build_segments(cu, img, txt, 2, 1, **kw)
    names = ("cu_seqlens", "seg_traj", "tok_gather", "tok_src_step", "tok_pos", "tok_loss_mask")
    cu_seq, seg_traj, gat, _, _, mask = seg = [lay[n] for n in names]
    mx = lay["max_seqlen"]
    qs, ks, vs = vcs.gather(q, k, v, gat, **kw)
    o, lse = vcs.attn_fwd(qs, ks, vs, cu_seq, mx, **kw)
    shared = vcs.shared_prefix(cu_seq, seg_traj, gat, **kw)
    traj_ids = torch.arange(len(q), dtype=torch.int32, device="cuda")
    traj_lp = -torch.arange(len(q), dtype=torch.float32, device="cuda") / len(q)
    torch.cuda.synchronize()
    ids, lp = vcs.stream_fields(traj_ids, traj_lp, gat, mask, **kw)
    old, adv = lp + 0.1, vcs.group_advantage(torch.tensor([0.0, 1.0], device="cuda"), 2, **kw)
    torch.cuda.synchronize()
    loss, dlogp = vcs.grpo_loss(lp, old, lp, mask, cu_seq, seg_traj, adv, **kw)
    out += seg + [qs, ks, vs, o, lse, shared, ids, lp, adv, loss, dlogp, vcs.compact_trainable(mask, **kw)]
    out += vcs.attn_fwd_reuse(qs, ks, vs, cu_seq, shared, mx, **kw)
    out += vcs.attn_fwd_gathered(q, k, v, gat, cu_seq, mx, **kw)
    grads = [*vcs.attn_bwd(qs, ks, vs, o, lse, o, cu_seq, mx, **kw),
             *vcs.attn_bwd_gathered(q, k, v, gat, o, lse, o, cu_seq, mx, **kw)]
    torch.cuda.synchronize()
    return out, grads


def check(got, want):
    for a, b in zip(got[0], want[0], strict=True):
        assert torch.equal(a, b)
    for a, b in zip(got[1], want[1], strict=True):  # fp32 sums in any order
        assert (a.double() - b.double()).norm() <= 1e-2 * b.double().norm()


def test_default_stream_by_its_handle():
    # the words of the builder, the gather, the fields and the compaction are read after this very
    # stream has been waited for, though it is busy when the call is made
    from paper_2607_11185_gb300 import vcs
    x = inputs()
    want = calls(x, None)
    assert torch.cuda.default_stream().cuda_stream == 0
    torch.cuda._sleep(BUSY)
    assert vcs.plan_segments(*x[:3], 2, 1, stream=0) == tuple(want[0][0].tolist())
    torch.cuda._sleep(BUSY)
    lay = vcs.build_segments(*x[:3], 2, 1, stream=0)
    assert torch.equal(lay["tok_gather"], want[0][3])
    check(calls(x, 0), want)
    check(calls(x, types.SimpleNamespace(cuda_stream=0)), want)
