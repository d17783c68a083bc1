"""GPU attention backward vs the fp64 oracle.

Tolerance (from the method's precision: bf16 inputs, fp32 accumulation):
relative L2 error <= 1e-2 per gradient tensor over all checked rows; where
the reference norm is below 1e-6 (exact zeros of one-token segments) the
absolute error must be <= 1e-3.
"""
import numpy as np
import pytest
import torch

from oracle import attention as oatt
from oracle import segments as oseg
from paper_2607_11185_gb300 import workloads
from tests.gpu_cases import bench_chunks, cu_from_lengths

pytestmark = pytest.mark.gpu

REL = 1e-2


def rel_err(got, ref):
    got = np.asarray(got, np.float64)
    ref = np.asarray(ref, np.float64)
    nr = np.linalg.norm(ref)
    if nr < 1e-6:
        return np.abs(got - ref).max() / 1e-1      # abs <= 1e-3 maps to <= 1e-2
    return np.linalg.norm(got - ref) / nr


def run(q, k, v, do, cu):
    from paper_2607_11185_gb300 import vcs
    dcu = torch.from_numpy(np.asarray(cu, np.int32)).cuda()
    mx = int(np.diff(cu).max())
    o, lse = vcs.attn_fwd(q, k, v, dcu, mx)
    dq, dk, dv = vcs.attn_bwd(q, k, v, o, lse, do, dcu, mx)
    return o, lse, dq, dk, dv


CASES = [
    ([1, 127, 128, 129, 255, 256, 257, 300], 2, 1, 64),
    ([1, 127, 128, 129, 255, 256, 257, 300], 2, 1, 128),
    ([600, 1, 383, 513], 7, 1, 128),
    ([640, 129], 4, 4, 64),
    ([1000], 6, 2, 128),
]


@pytest.mark.parametrize("lengths,hq,hkv,d", CASES)
def test_small_shapes_full_oracle(lengths, hq, hkv, d):
    cu = cu_from_lengths(lengths)
    q, k, v, do = workloads.draw_dense(31 + d + hq, int(cu[-1]), hq, hkv, d, device="cuda")
    _, _, dq, dk, dv = run(q, k, v, do, cu)
    rq, rk, rv = oatt.attn_bwd(q.cpu(), k.cpu(), v.cpu(), do.cpu(), cu)
    for name, got, ref in (("dq", dq, rq), ("dk", dk, rk), ("dv", dv, rv)):
        e = rel_err(got.float().cpu().numpy(), ref)
        assert e <= REL, (name, e)


def test_tiny_workload_full_oracle():
    w = workloads.WORKLOADS["tiny"]
    cu_s, img, txt = workloads.draw_steps(w)
    lay = oseg.build(cu_s, img, txt, w.window, w.keep)
    qt, kt, vt = workloads.draw_traj_qkv(w, workloads.trajectory_tokens(img, txt), device="cuda")
    g = torch.from_numpy(lay["tok_gather"].astype(np.int64)).cuda()
    q, k, v = qt[g], kt[g], vt[g]
    do = workloads.draw_dout(w, q.shape[0], device="cuda")
    _, _, dq, dk, dv = run(q, k, v, do, lay["cu_seqlens"])
    rq, rk, rv = oatt.attn_bwd(q.cpu(), k.cpu(), v.cpu(), do.cpu(), lay["cu_seqlens"])
    for got, ref in ((dq, rq), (dk, rk), (dv, rv)):
        assert rel_err(got.float().cpu().numpy(), ref) <= REL


def test_single_token_segments():
    cu = cu_from_lengths([1] * 24)
    q, k, v, do = workloads.draw_dense(9, 24, 4, 2, 64, device="cuda")
    _, _, dq, dk, dv = run(q, k, v, do, cu)
    assert dq.abs().max().item() <= 1e-3 and dk.abs().max().item() <= 1e-3
    ref_dv = do.float().view(24, 2, 2, 64).sum(2)
    assert rel_err(dv.float().cpu().numpy(), ref_dv.cpu().numpy()) <= REL


def test_large_logits_stress():
    cu = cu_from_lengths([700, 333])
    q, k, v, do = workloads.draw_dense(22, int(cu[-1]), 2, 1, 128, device="cuda", scale=6.0)
    _, _, dq, dk, dv = run(q, k, v, do, cu)
    rq, rk, rv = oatt.attn_bwd(q.cpu(), k.cpu(), v.cpu(), do.cpu(), cu)
    for got, ref in ((dq, rq), (dk, rk), (dv, rv)):
        assert rel_err(got.float().cpu().numpy(), ref) <= REL


def check_sampled_grads(q, k, v, do, cu, dq, dk, dv, rng, n_seg=4, n_rows=6, tail=48):
    """dQ on sampled rows; dK/dV on the last `tail` keys of sampled segments; gradient sums."""
    nseg = len(cu) - 1
    lens = np.diff(cu)
    hq, hkv = q.shape[1], k.shape[1]
    G = hq // hkv
    segs = sorted({int(np.argmin(lens)), int(np.argmax(lens)), 0, nseg - 1,
                   *[int(x) for x in rng.integers(0, nseg, size=n_seg)]})
    got_q, ref_q, got_k, ref_k, got_v, ref_v = [], [], [], [], [], []
    for s in segs:
        b, e = int(cu[s]), int(cu[s + 1])
        L = e - b
        heads = sorted({0, hq - 1, int(rng.integers(0, hq))})
        rows = sorted({0, L - 1, *[int(x) for x in rng.integers(0, L, size=n_rows)]})
        ref = oatt.rows_dq(q, k, v, do, (b, e), heads, rows)
        idx = torch.tensor([b + r for r in rows], device=dq.device)
        got_q.append(dq[idx][:, heads].float().cpu().numpy())
        ref_q.append(ref)
        g = int(rng.integers(0, hkv))
        keys = list(range(max(0, L - tail), L))
        rk, rv = oatt.keys_dkdv(q, k, v, do, (b, e), g, keys)
        kidx = torch.tensor([b + j for j in keys], device=dk.device)
        got_k.append(dk[kidx, g].float().cpu().numpy())
        ref_k.append(rk)
        got_v.append(dv[kidx, g].float().cpu().numpy())
        ref_v.append(rv)
        # sum_j dK_j = 0 and sum_j dV_j = sum_i dO_i over the group, per segment (any size)
        sdk = dk[b:e].float().sum(0)
        assert (sdk.abs().max() / dk[b:e].float().abs().sum(0).max().clamp_min(1e-6)).item() < 1e-2
        sdv = dv[b:e].float().sum(0)
        sdo = do[b:e].float().view(L, hkv, G, -1).sum((0, 2))
        assert ((sdv - sdo).norm() / sdo.norm()).item() < 1e-2
    for name, got, ref in (("dq", got_q, ref_q), ("dk", got_k, ref_k), ("dv", got_v, ref_v)):
        e = rel_err(np.concatenate([x.ravel() for x in got]), np.concatenate([x.ravel() for x in ref]))
        assert e <= REL, (name, e)


def _layout_inputs(name, first_chunk=False):
    """The workload's inputs in segment layout; with first_chunk, only the segments of the
    benchmark's first launch (its first trajectory chunk)."""
    w = workloads.WORKLOADS[name]
    cu_s, img, txt = workloads.draw_steps(w)
    lay = oseg.build(cu_s, img, txt, w.window, w.keep)
    qt, kt, vt = workloads.draw_traj_qkv(w, workloads.trajectory_tokens(img, txt), device="cuda")
    cu = lay["cu_seqlens"]
    if first_chunk:
        cu = cu[: bench_chunks(w, lay, len(cu_s) - 1)[0][1] + 1]
    nt = int(cu[-1])
    g = torch.from_numpy(lay["tok_gather"][:nt].astype(np.int64)).cuda()
    q, k, v = qt[g], kt[g], vt[g]
    do = workloads.draw_dout(w, len(lay["tok_gather"]), device="cuda")[:nt].contiguous()
    return q, k, v, do, cu


def test_traj8_full_size_sampled():
    q, k, v, do, cu = _layout_inputs("traj8_w3")
    _, _, dq, dk, dv = run(q, k, v, do, cu)
    check_sampled_grads(q, k, v, do, cu, dq, dk, dv, np.random.default_rng(8))


def test_traj32_first_chunk_sampled():
    q, k, v, do, cu = _layout_inputs("traj32_w3", first_chunk=True)
    _, _, dq, dk, dv = run(q, k, v, do, cu)
    check_sampled_grads(q, k, v, do, cu, dq, dk, dv, np.random.default_rng(32), n_seg=2, n_rows=4, tail=16)


def test_long_horizon_first_chunk_sampled():
    q, k, v, do, cu = _layout_inputs("traj16x50_w8", first_chunk=True)
    _, _, dq, dk, dv = run(q, k, v, do, cu)
    check_sampled_grads(q, k, v, do, cu, dq, dk, dv, np.random.default_rng(50), n_seg=1, n_rows=3, tail=8)


def test_long_horizon_early_and_middle_key_tiles():
    """dK, dV at full size where the backward does the most work: one kv head of the shortest
    segment of the benchmark's first long-horizon chunk (L = 25,696), on the first key tile
    (keys 0-127: every query tile of the segment and all five heads of the group reach it), a
    tile in the middle of the segment and the ragged last tile, against the oracle evaluated
    for those keys over all their query rows."""
    q, k, v, do, cu = _layout_inputs("traj16x50_w8", first_chunk=True)
    _, _, dq, dk, dv = run(q, k, v, do, cu)
    lens = np.diff(cu)
    s = int(np.argmin(lens))
    b, e = int(cu[s]), int(cu[s + 1])
    L = e - b
    mid = (L // 2) // 128 * 128
    last = (L - 1) // 128 * 128
    keys = list(range(0, 128)) + list(range(mid, mid + 128)) + list(range(last, L))
    g = 3
    rk, rv = oatt.keys_dkdv_blocked(q, k, v, do, (b, e), g, keys, row_block=1024)
    kidx = torch.tensor([b + j for j in keys], device=dk.device)
    for name, got, ref in (("dk", dk[kidx, g], rk), ("dv", dv[kidx, g], rv)):
        got = got.float().cpu().numpy()
        for lo, hi in ((0, 128), (128, 256), (256, len(keys))):   # each tile on its own
            err = rel_err(got[lo:hi], ref[lo:hi])
            assert err <= REL, (name, lo, err)


def test_traj8_longest_segment_every_key_and_row():
    """The 8-trajectory workload's longest segment (5,671 tokens) for one kv head in full: dK,
    dV of every key and dQ of every row of the group's seven query heads, against the full
    oracle on that group."""
    q, k, v, do, cu = _layout_inputs("traj8_w3")
    _, _, dq, dk, dv = run(q, k, v, do, cu)
    lens = np.diff(cu)
    s = int(np.argmax(lens))
    b, e = int(cu[s]), int(cu[s + 1])
    hq, hkv = q.shape[1], k.shape[1]
    G = hq // hkv
    g = 2
    heads = slice(g * G, (g + 1) * G)
    rq, rk, rv = oatt.attn_bwd(q[b:e, heads].cpu(), k[b:e, g:g + 1].cpu(), v[b:e, g:g + 1].cpu(),
                               do[b:e, heads].cpu(), [0, e - b])
    for name, got, ref in (("dq", dq[b:e, heads], rq), ("dk", dk[b:e, g:g + 1], rk), ("dv", dv[b:e, g:g + 1], rv)):
        err = rel_err(got.float().cpu().numpy(), ref)
        assert err <= REL, (name, err)


@pytest.mark.parametrize("hq,hkv,d", [(1, 1, 64), (1, 1, 128), (2, 1, 64), (3, 1, 128), (5, 1, 64), (5, 1, 128)])
def test_query_tile_counts_around_the_rings(hq, hkv, d):
    """Key tiles with 1 .. 25 query tiles (head by head: 1, 2, 3, 5 of each row block), so that the
    Q/dO rings, the row-term buffers and the first and last tile of the two chains meet every count,
    with full and ragged last tiles."""
    cu = cu_from_lengths([1, 128, 129, 256, 260, 384, 511, 640])
    q, k, v, do = workloads.draw_dense(77 + d + hq, int(cu[-1]), hq, hkv, d, device="cuda")
    _, _, dq, dk, dv = run(q, k, v, do, cu)
    rq, rk, rv = oatt.attn_bwd(q.cpu(), k.cpu(), v.cpu(), do.cpu(), cu)
    for name, got, ref in (("dq", dq, rq), ("dk", dk, rk), ("dv", dv, rv)):
        e = rel_err(got.float().cpu().numpy(), ref)
        assert e <= REL, (name, e)


def test_dk_dv_summed_in_query_order_d64():
    """At d = 64 dK and dV are fp32 sums over the group's heads in turn, each from the key tile's own
    rows to the segment end, 16 query rows a term.  Every dim gets a 1, a 2^30 and a -2^30 in three of
    the terms, whose sum is 1 or 0 by their order, so the result is that order's, exactly."""
    d, G, L, big = 64, 2, 384 + 40, float(2 ** 30)
    rng = np.random.default_rng(3)
    groups = (L + 15) // 16
    order = [(h, c) for h in range(G) for c in range(groups)]

    def column():
        terms = np.zeros(len(order), np.float32)
        at = rng.choice(len(order), 3, replace=False)
        terms[at] = rng.permutation([1.0, big, -big])
        total = np.float32(0)
        for t in terms:
            total = np.float32(total + t)
        return terms, total

    # keys 0 and 1 share every later row (P = 1/2 each), with opposite values: O = 0, dS = +-1
    q = torch.zeros(L, G, d)
    do = torch.zeros(L, G, d)
    k = torch.zeros(L, 1, d)
    v = torch.zeros(L, 1, d)
    q[:, :, 0], do[:, :, 0], k[:2, 0, 0], k[2:, 0, 0] = 16, 16, 16, -16
    v[0, 0, 0], v[1, 0, 0] = 1, -1
    want = np.zeros((2, d), np.float32)  # dK_0 and dV_0
    for b in range(1, d):
        for which, (x, unit) in enumerate(((q, 1.0), (do, 2.0))):
            terms, want[which, b] = column()
            for (h, c), t in zip(order, terms):
                x[min(16 * c + 1 + int(rng.integers(0, 15)), L - 1), h, b] = unit * float(t)
    _, _, _, dk, dv = run(*(x.bfloat16().cuda() for x in (q, k, v, do)), [0, L])
    assert 8 < want[0].sum() < d - 8 and 8 < want[1].sum() < d - 8  # both outcomes occur
    assert np.array_equal(dk[0, 0, 1:].float().cpu().numpy(), want[0, 1:])
    assert np.array_equal(dv[0, 0, 1:].float().cpu().numpy(), want[1, 1:])


@pytest.mark.parametrize("d", [64, 128])
def test_segment_ends_around_the_drains_row_groups(d):
    """At d = 128 the last query tile's rows past the segment end are left out of the dQ reductions 16 at a
    time, and warps without rows skip the epilogue: ends on both sides of each, against the oracle, and
    the gathered backward (rows in trajectory order) against the same gradients."""
    from paper_2607_11185_gb300 import vcs
    lengths = [1, 7, 8, 9, 15, 16, 17, 24, 25, 31, 32, 33, 48, 49, 64, 65, 96, 97, 112, 113, 120, 121, 127, 128, 129,
               144, 145, 161, 256 + 33]
    cu = cu_from_lengths(lengths)
    q, k, v, do = workloads.draw_dense(77 + d, int(cu[-1]), 2, 1, d, device="cuda")
    o, lse, *grads = run(q, k, v, do, cu)
    want = oatt.attn_bwd(q.cpu(), k.cpu(), v.cpu(), do.cpu(), cu)
    for s, e in zip(cu, cu[1:]):
        for name, got, ref in zip(("dq", "dk", "dv"), grads, want):
            # a segment of a few rows averages few bf16 roundings
            assert rel_err(got[s:e].float().cpu().numpy(), ref[s:e]) <= 2.5 * REL, (name, e - s)
    gat = torch.arange(int(cu[-1]), dtype=torch.int32, device="cuda")
    got = vcs.attn_bwd_gathered(q, k, v, gat, o, lse, do, torch.from_numpy(cu).cuda(), max(lengths))
    for name, a, b in zip(("dq", "dk", "dv"), got, grads):
        assert (a.double() - b.double()).norm() <= 5e-3 * b.double().norm(), name


def test_d64_keeps_the_exact_difference_of_dp_and_d():
    """One-token segments: P = 1, O = v and dP = D exactly for small whole numbers, so dS, and with it dQ
    and dK, is 0, at any scale.  (-D scale) rounded on its own left a residue at scales that are not a
    power of two."""
    from paper_2607_11185_gb300 import vcs
    n, d = 9, 64
    g = torch.Generator(device="cuda").manual_seed(4)
    q, k = (torch.randn((n, h, d), generator=g, device="cuda").bfloat16() for h in (2, 1))
    v, do = (torch.randint(-3, 4, (n, h, d), generator=g, device="cuda").bfloat16() for h in (1, 2))
    cu = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    for scale in (0.1, 0.3, 0.125):
        o, lse = vcs.attn_fwd(q, k, v, cu, 1, softmax_scale=scale)
        assert torch.equal(o, v.expand(n, 2, d))
        dq, dk, dv = vcs.attn_bwd(q, k, v, o, lse, do, cu, 1, softmax_scale=scale)
        assert not dq.any() and not dk.any()
        assert torch.equal(dv.float(), do.float().sum(1, keepdim=True))
