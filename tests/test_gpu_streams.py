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


def calls(x, stream, before=lambda: None):
    """Every allocating call with the given stream, `before` ahead of each: (exact results, gradients)."""
    from paper_2607_11185_gb300 import vcs
    cu, img, txt, q, k, v = x
    traj_ids = torch.arange(len(q), dtype=torch.int32, device="cuda")
    traj_lp = -torch.arange(len(q), dtype=torch.float32, device="cuda") / len(q)
    rewards = torch.tensor([0.0, 1.0], device="cuda")

    def call(fn, *args):
        torch.cuda.synchronize()  # the arguments may come from another stream
        before()
        return fn(*args) if stream is None else fn(*args, stream=stream)

    lay = call(vcs.build_segments, cu, img, txt, 2, 1)
    names = ("cu_seqlens", "seg_traj", "tok_gather", "tok_src_step", "tok_pos", "tok_loss_mask")
    cu_seq, seg_traj, gat, _, _, mask = seg = [lay[n] for n in names]
    mx = lay["max_seqlen"]
    qs, ks, vs = call(vcs.gather, q, k, v, gat)
    o, lse = call(vcs.attn_fwd, qs, ks, vs, cu_seq, mx)
    shared = call(vcs.shared_prefix, cu_seq, seg_traj, gat)
    ids, lp = call(vcs.stream_fields, traj_ids, traj_lp, gat, mask)
    adv = call(vcs.group_advantage, rewards, 2)
    torch.cuda.synchronize()
    loss, dlogp = call(vcs.grpo_loss, lp, lp + 0.1, lp, mask, cu_seq, seg_traj, adv)
    out = [torch.tensor(call(vcs.plan_segments, cu, img, txt, 2, 1)), *seg, qs, ks, vs, o, lse, shared, ids, lp, adv,
           loss, dlogp, call(vcs.compact_trainable, mask), *call(vcs.attn_fwd_reuse, qs, ks, vs, cu_seq, shared, mx),
           *call(vcs.attn_fwd_gathered, q, k, v, gat, cu_seq, mx)]
    grads = [*call(vcs.attn_bwd, qs, ks, vs, o, lse, o, cu_seq, mx),
             *call(vcs.attn_bwd_gathered, q, k, v, gat, o, lse, o, cu_seq, mx)]
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


def poison(stream):
    """Leaves words that are no status in the stream's free memory."""
    with torch.cuda.stream(stream):
        junk = [torch.full((1 << n,), 0x5f5f5f5f, dtype=torch.int32, device="cuda") for n in range(6, 21)
                for _ in range(4)]
        torch.cuda.synchronize()
        del junk


@pytest.mark.parametrize("form", ["stream", "handle"])
def test_busy_stream_other_than_the_current(form):
    # every word is read behind the call's kernels, though the call's stream is busy and the current
    # one is not, and the workspace holds words that are no status
    x = inputs()
    want = calls(x, None)
    side = torch.cuda.Stream()

    def before():
        poison(torch.cuda.current_stream())
        poison(side)
        with torch.cuda.stream(side):
            torch.cuda._sleep(BUSY)

    check(calls(x, side if form == "stream" else side.cuda_stream, before), want)


def test_workspace_of_a_running_call_is_not_handed_out(monkeypatch):
    from paper_2607_11185_gb300 import vcs
    q, k, v = inputs()[3:]
    cu = torch.tensor([0, len(q)], dtype=torch.int32, device="cuda")
    taken, ws = [], vcs._ws

    def keep(*args):
        t = ws(*args)
        taken.append((t.data_ptr(), t.numel()))
        return t

    monkeypatch.setattr(vcs, "_ws", keep)
    side = torch.cuda.Stream()
    want = vcs.attn_fwd(q, k, v, cu, len(q))
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(BUSY)
    got = vcs.attn_fwd(q, k, v, cu, len(q), stream=side, check=False)
    ptr, n = taken[-1]
    assert all(torch.empty(n, dtype=torch.int32, device="cuda").data_ptr() != ptr for _ in range(4))
    assert not side.query()
    torch.cuda.synchronize()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("name", ["plan_segments", "build_segments", "gather", "shared_prefix", "stream_fields",
                                  "compact_trainable"])
def test_failed_call_is_waited_for(name, monkeypatch):
    # a call that launched a kernel and then failed: its pinned words stay until the kernel is done
    from paper_2607_11185_gb300 import vcs
    x = inputs()
    lay = vcs.build_segments(*x[:3], 2, 1)
    gat, mask = lay["tok_gather"], lay["tok_loss_mask"]
    args = dict(plan_segments=(*x[:3], 2, 1), build_segments=(*x[:3], 2, 1), gather=(*x[3:], gat),
                shared_prefix=(lay["cu_seqlens"], lay["seg_traj"], gat),
                stream_fields=(gat, gat.float(), gat, mask), compact_trainable=(mask,))[name]
    real = getattr(vcs, "vcs_" + name)

    def fails(*a, **kw):
        torch.cuda._sleep(BUSY)
        assert real(*a, **kw) == 0
        return 5

    monkeypatch.setattr(vcs, "vcs_" + name, fails)
    with pytest.raises(vcs.VcsError):
        getattr(vcs, name)(*args)
    assert torch.cuda.current_stream().query()
