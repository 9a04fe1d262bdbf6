"""Sizes at which a kernel's split of the work changes: row lengths around the register budgets of the ranking, blocks per
head around the pooling splits, lists whose segments are shorter or longer than the rings and slots they run through.

Bars as in test_gpu_parity.py (its checks are used): descriptors, codes, scales and lists exact, outputs within the bf16
tolerance of the oracle.
"""
import ctypes

import numpy as np
import pytest
import torch

import da2_inputs
import oracle
import paper_2609_32628_b200 as da2
from helpers import Workspace, oracle_all, run_gpu
from test_gpu_parity import _check_attention, _check_prepare

pytestmark = pytest.mark.gpu
W = da2_inputs.Workload


# R = T * tiles from the smallest rows there are to beyond 2,048 entries (longer rows are ranked by a whole thread block), whole
# calls; the edges of every register count of the ranking: test_rows_at_every_register_count
@pytest.mark.parametrize("T,Hg,Wg", [(1, 8, 8), (1, 9, 8), (4, 32, 32), (13, 8, 40), (32, 8, 40), (23, 8, 56), (107, 8, 24),
                                     (29, 24, 56), (23, 24, 104), (61, 24, 56), (128, 32, 32), (683, 8, 24)])
def test_row_lengths(T, Hg, Wg):
    w = W("rows", 1, 1, 64, T, Hg, Wg, 0.0, 0.10, 0.20, seed=31)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    plan, ws, out = run_gpu(w, q, k, v)
    ref = oracle_all(w, q, k, v)
    bad = _check_prepare(w, plan, ws, ref)
    R = plan.info.R
    sel = [(0, a) for a in sorted({0, R // 2, R - 1})]
    if sum(int(x) for x in plan.info.quota):
        _check_attention(w, out, ref, sel, bad)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("f16,f8,f4", [(0.15, 0.25, 0.30), (0.15, 0.25, 0.0), (0.15, 0.0, 0.30), (0.02, 0.03, 0.30),
                                       (0.30, 0.02, 0.02), (0.4, 0.0, 0.0)])
def test_segments_of_three_tiers(d, f16, f8, f4):
    """Many heads at once (the order in which warps meet varies), segments of 1 to 23 blocks: bit-identical over repeated
    runs, and equal to the oracle on sampled blocks."""
    w = W("segments", 1, 21, d, 5, 23, 40, f16, f8, f4, seed=32, k_outlier_channels=(3, 35), k_outlier_gain=5.0)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    plan, ws, out = run_gpu(w, q, k, v)
    again = torch.empty_like(out)
    for _ in range(4):
        again.fill_(float("nan"))
        da2.da2_attention_fwd(plan, q, k, v, ws, again)
        assert torch.equal(out, again)
    heads = [0, 20]
    ref = oracle_all(w, q, k, v, heads=heads)
    bad = _check_prepare(w, plan, ws, ref, heads=heads)
    sel = [(h, int(a)) for h in range(2) for a in np.random.default_rng(3).choice(plan.info.R, 10, replace=False)]
    _check_attention(w, out, ref, sel, bad, heads=heads)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n16,n8,n4", [(0, 0, 1), (0, 1, 0), (0, 1, 1), (0, 2, 3), (0, 3, 2), (0, 33, 4), (0, 1, 34), (1, 0, 0),
                                       (1, 1, 0), (1, 0, 1), (2, 1, 2), (3, 2, 1), (1, 32, 3), (5, 16, 17), (0, 0, 31), (0, 0, 32),
                                       (0, 1, 31), (0, 3, 31), (0, 3, 32), (4, 0, 31), (4, 0, 32), (3, 15, 16), (3, 14, 17),
                                       (1, 15, 16), (31, 0, 0), (32, 0, 0), (33, 0, 0), (2, 31, 0), (1, 0, 30)])
def test_lists_of_odd_and_even_segments(n16, n8, n4, d):
    """Blocks of a list are fetched in pairs (those of the 16-bit tier one by one): segments and lists that end in the middle of a
    pair, and one below, at and above the 32 entries that a loader holds, on ragged tiles."""
    w = W("pairs", 1, 2, d, 5, 12, 28, n16 / 40, n8 / 40, n4 / 40, seed=37)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    plan, ws, out = run_gpu(w, q, k, v)
    assert [int(x) for x in plan.info.quota] == [n4, n8, n16] and plan.info.R == 40
    ref = oracle_all(w, q, k, v)
    bad = _check_prepare(w, plan, ws, ref)
    _check_attention(w, out, ref, [(h, a) for h in range(2) for a in (0, 3, 20, 39)], bad)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("f16,f8,f4", [(0.1, 0.2, 0.45), (0.0, 0.25, 0.5), (0.25, 0.5, 0.0)])
def test_head_scope_lists_that_end_at_a_loaders_batch(f16, f8, f4, d):
    """The same with one ranking per head: every row whose segments or list end one below, at or above 32 entries."""
    w = W("batch", 1, 8, d, 5, 12, 28, f16, f8, f4, seed=40)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    plan, ws, out = run_gpu(w, q, k, v, rank_scope=1)
    ref = oracle_all(w, q, k, v, rank_scope=1)
    bad = _check_prepare(w, plan, ws, ref)
    _, cnt = Workspace(plan, ws).lists()
    ends = np.cumsum(cnt, 2)
    sel = [(int(h), int(a)) for h, a in np.argwhere(((ends >= 31) & (ends <= 33)).any(2))]
    assert all((ends == n).any() for n in (31, 32, 33))
    _check_attention(w, out, ref, sel, bad)


@pytest.mark.parametrize("H", [1, 8, 30])
def test_pooling_splits(H):
    """80 blocks a head: eight and two warps per block (two twice)."""
    w = W("pool", 1, H, 128, 5, 27, 30, 0.1, 0.2, 0.2, seed=33)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    plan, ws, _ = run_gpu(w, q, k, v)
    heads = sorted({0, H - 1})
    _check_prepare(w, plan, ws, oracle_all(w, q, k, v, heads=heads), heads=heads)


# 80 blocks a head: 4, 2 and 1 warps per block at d = 128; 8, 8, 4, 2 and 1 at d = 64
@pytest.mark.parametrize("H,d", [(5, 128), (8, 128), (20, 128), (2, 64), (5, 64), (8, 64), (20, 64), (30, 64)])
def test_pooling_by_waves(H, d):
    w = W("pool", 1, H, d, 5, 27, 30, 0.1, 0.2, 0.2, seed=36)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    plan, ws, _ = run_gpu(w, q, k, v)
    heads = sorted({0, H - 1})
    _check_prepare(w, plan, ws, oracle_all(w, q, k, v, heads=heads), heads=heads)


# rows of half a tile and one more, and the grids of one and of two CTAs per SM with the next larger ones
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("H,R", [(16, 32), (16, 33), (74, 33), (75, 33), (148, 33), (149, 33)])
def test_draft_logits_by_grid(H, R, d):
    """Logits against their definition in fp64 (one rounding to fp32; an fp64 sum of d terms errs by d half ulps of its largest
    partial sum at most), and what runs beside them against the oracle."""
    w = W("logits", 1, H, d, R, 8, 8, 0.0, 0.1, 0.3, seed=39)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    plan, ws, _ = run_gpu(w, q, k, v)
    I = plan.info
    desc = [ws[I.off_desc[i]:I.off_desc[i] + H * R * d * 4].view(torch.float32).view(H, R, d).double() for i in range(4)]
    for i in range(2):
        got = ws[I.off_logits[i]:I.off_logits[i] + H * R * R * 4].view(torch.float32).view(H, R, R).double()
        exp = float(I.softmax_scale) * desc[i] @ desc[2 + i].transpose(1, 2)
        mag = float(I.softmax_scale) * desc[i].abs() @ desc[2 + i].abs().transpose(1, 2)
        assert ((got - exp).abs() <= exp.abs() * 2.0 ** -24 + mag * (2 * d * 2.0 ** -53 + 2.0 ** -52)).all()
    heads = [0, H - 1]
    _check_prepare(w, plan, ws, oracle_all(w, q, k, v, heads=heads), heads=heads)


@pytest.mark.parametrize("T,Hg,Wg", [(1, 8, 8), (3, 9, 20), (13, 8, 40), (23, 24, 56), (683, 8, 24)])
@pytest.mark.parametrize("f16,f8,f4", [(0.1, 0.2, 0.3), (0.0, 0.1, 0.2)])
def test_head_scope_sizes(T, Hg, Wg, f16, f8, f4):
    if T == 683 and f16:
        pytest.skip("one budget is enough for the longest rows")
    w = W("head", 1, 2, 64, T, Hg, Wg, f16, f8, f4, seed=34)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    plan, ws, out = run_gpu(w, q, k, v, rank_scope=1)
    ref = oracle_all(w, q, k, v, rank_scope=1)
    bad = _check_prepare(w, plan, ws, ref)
    R = plan.info.R
    _check_attention(w, out, ref, [(h, a) for h in range(2) for a in sorted({0, R // 2, R - 1})], bad)


@pytest.mark.parametrize("rank_scope", [0, 1])
@pytest.mark.parametrize("T,Hg,Wg", [(2, 16, 16), (9, 24, 40), (2, 24, 352)])
def test_ties_go_to_the_lower_index(T, Hg, Wg, rank_scope):
    """Constant Q and K: every score of the map is the same, so every boundary is a tie (the bisection of a row and the
    radix passes of a head run to their last bit)."""
    w = W("ties", 1, 2, 64, T, Hg, Wg, 0.1, 0.2, 0.3, seed=35)
    _, _, v = da2_inputs.make_qkv(w, "cuda")
    q = torch.ones_like(v)
    k = torch.ones_like(v)
    plan, ws, out = run_gpu(w, q, k, v, rank_scope=rank_scope)
    ref = oracle_all(w, q, k, v, rank_scope=rank_scope)
    assert _check_prepare(w, plan, ws, ref) == []
    _check_attention(w, out, ref, [(1, 0), (1, plan.info.R - 1)], [])


@pytest.mark.parametrize("rank_scope", [0, 1])
@pytest.mark.parametrize("H,T,Hg,Wg", [(2, 2, 8, 296), (2, 5, 24, 40), (4, 5, 24, 40), (5, 5, 24, 40), (6, 5, 24, 40)])
def test_last_wave_of_blocks(H, T, Hg, Wg, rank_scope):
    """One query block per CTA in the last wave: 148 blocks (all of them), 150 (none), 300 and 375 in heads of 75 (the last 7
    and 82), 450 (none: 157 would be left)."""
    w = W("wave", 1, H, 64, T, Hg, Wg, 0.0, 0.1, 0.2, seed=35)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    plan, ws, out = run_gpu(w, q, k, v, rank_scope=rank_scope)
    ref = oracle_all(w, q, k, v, rank_scope=rank_scope)
    bad = _check_prepare(w, plan, ws, ref)
    R = plan.info.R
    sel = [(h, a) for h in range(H) for a in (0, 1, 66, 67, 68, 69, R - 2, R - 1)]
    _check_attention(w, out, ref, sel, bad)
    again = torch.full_like(out, float("nan"))
    da2.da2_attention_fwd(plan, q, k, v, ws, again)
    assert torch.equal(out, again)


@pytest.mark.parametrize("fixed", [False, True])
@pytest.mark.parametrize("H,T,Hg,Wg", [(1, 1, 8, 8), (2, 4, 16, 16), (12, 8, 32, 32)])
def test_operands_follow_their_own_call(H, T, Hg, Wg, fixed):
    """The operand kernel runs beside the draft logits on scales that the kernels before those wrote: calls on inputs of very
    different range, enqueued one after the other on one workspace, leave what each leaves when it runs alone."""
    w = W("order", 1, H, 128, T, Hg, Wg, 0.1, 0.2, 0.3, seed=36)
    x = da2_inputs.make_qkv(w, "cuda")
    inputs = [x, [t * 512 for t in x], [t.flip(2) / 256 for t in x]]
    g = [np.full(H, s, np.float32) for s in (0.002, 0.003, 0.004)] if fixed else (None, None, None)
    plan = da2.da2_plan(1, H, T, Hg, Wg, 128, 0.1, 0.2, 0.3, g_q=g[0], g_k=g[1], g_v=g[2])
    I = plan.info
    kept = lambda ws: torch.cat([ws[I.off_gscale:I.off_gscale + H * 16],
                                 *(ws[I.off_qrec[t]:I.off_qrec[t] + H * I.R * I.qrec_bytes[t]] for t in range(3)),
                                 *(ws[I.off_kvrec[t]:I.off_kvrec[t] + H * I.R * I.kvrec_bytes[t]] for t in range(3)),
                                 ws[I.off_dq8:I.off_dq8 + H * I.R * 4], ws[I.off_dv8:I.off_dv8 + H * 128 * 4]])
    alone = []
    for qkv in inputs:
        ws = torch.zeros(int(I.workspace_bytes), dtype=torch.uint8, device="cuda")
        da2.da2_prepare(plan, *qkv, ws)
        torch.cuda.synchronize()
        alone.append(kept(ws))
    ws = torch.zeros(int(I.workspace_bytes), dtype=torch.uint8, device="cuda")
    got = []
    for i in range(60):
        da2.da2_prepare(plan, *inputs[i % 3], ws)
        if i % 4 == 3:
            got.append((i % 3, kept(ws)))
    torch.cuda.synchronize()
    for i, g_ in got:
        assert torch.equal(g_, alone[i])


@pytest.mark.parametrize("rank_scope", [0, 1])
@pytest.mark.parametrize("T,Hg,Wg", [(2, 16, 16), (5, 24, 40)])
@pytest.mark.parametrize("call", ["prepare", "refresh", "cached", "cached_reselect"])
def test_a_call_starts_behind_all_earlier_work(call, T, Hg, Wg, rank_scope):
    """The first kernel of a preparation depends on the completion of what the caller enqueued before it; only the kernels behind
    it may start early.  Read off the edges of a captured graph, whose nodes are as many as the launches reported; a replay
    leaves the same bits in the workspace (8 and 75 blocks a head: logits in plain and in spread grids)."""
    w = W("edges", 1, 2, 64, T, Hg, Wg, 0.1, 0.2, 0.3, seed=38)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    plan, ws, _ = run_gpu(w, q, k, v, rank_scope=rank_scope, zero_ws=True)
    rt = ctypes.CDLL("libcudart.so.12")
    stream = torch.cuda.Stream()
    handle, graph, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        assert rt.cudaStreamBeginCapture(handle, 2) == 0          # relaxed mode
        q.mul_(1.0)                                               # a kernel of the caller's
        {"prepare": lambda: da2.da2_prepare(plan, q, k, v, ws), "refresh": lambda: da2.da2_refresh_operands(plan, q, k, v, ws),
         "cached": lambda: da2.da2_prepare_cached_scales(plan, q, k, v, ws, reselect=False),
         "cached_reselect": lambda: da2.da2_prepare_cached_scales(plan, q, k, v, ws, reselect=True)}[call]()
        assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetEdges_v2(graph, None, None, None, ctypes.byref(n)) == 0
    src, dst = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)()
    data = (ctypes.c_uint8 * (8 * n.value))()                     # 8 bytes an edge; the third says: 0 full, 1 programmatic
    assert rt.cudaGraphGetEdges_v2(graph, src, dst, data, ctypes.byref(n)) == 0
    kinds = {src[i]: data[8 * i + 2] for i in range(n.value)}     # a chain: one edge out of every node but the last
    caller = set(src) - set(dst)
    assert len(kinds) == n.value and len(caller) == 1 and kinds[caller.pop()] == 0 and 1 in kinds.values()
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    assert n.value == 1 + da2.da2_last_launch_count(plan)
    I, ref, run = plan.info, ws.clone(), ctypes.c_void_p()
    ws[I.off_qrec[0]:I.off_dq8].zero_()
    torch.cuda.synchronize()
    assert rt.cudaGraphInstantiate(ctypes.byref(run), graph, ctypes.c_ulonglong(0)) == 0
    assert rt.cudaGraphLaunch(run, handle) == 0
    torch.cuda.synchronize()
    assert torch.equal(ws[I.off_vmax:I.off_select], ref[I.off_vmax:I.off_select])
    assert torch.equal(ws[I.off_qrec[0]:], ref[I.off_qrec[0]:])
    assert rt.cudaGraphExecDestroy(run) == 0 and rt.cudaGraphDestroy(graph) == 0


_HELD = (2, 4, 6, 8, 10, 12, 14, 16, 20, 24, 28, 32, 40, 48, 56, 64)  # entries per lane a row may be held in


@pytest.mark.parametrize("lam", [0.0, 1.0])
@pytest.mark.parametrize("R", [1, 33] + [32 * e + x for e in _HELD for x in (0, 1)])
def test_rows_at_every_register_count(R, lam):
    """The last register of a row full and the first of the next size, three boundaries at once.  Scores: at lambda 0 and 1 the
    map is the quotient of one branch, so its bits follow from the stored logits by correctly rounded steps: exponentials,
    their sum in the order of 256 threads (whatever kernel takes the row), one division.  The logits are spread so that
    exponentials from 1 to below 2^-100 occur.  Lists: exactly the oracle's ranking of the stored map."""
    w = W("registers", 1, 1, 64, R, 8, 8, 0.1, 0.2, 0.3, seed=37)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    plan, ws, _ = run_gpu(w, q * 40, k, v, lam=lam)
    I = plan.info
    V = Workspace(plan, ws)
    A = V.draft_map()
    logits = ws[I.off_logits[int(lam)]:I.off_logits[int(lam)] + R * R * 4].view(torch.float32).view(R, R)
    x = torch.exp(logits - logits.max(1, keepdim=True).values)
    if R > 64:
        assert ((x > 0) & (x < 2.0 ** -100)).any()
    y = torch.zeros(R, -(-R // 256) * 256, device="cuda")
    y[:, :R] = x
    y = y.view(R, -1, 256)
    z = torch.zeros(R, 256, device="cuda")
    for i in range(y.shape[1]):
        z = z + y[:, i]
    z = z.view(R, 8, 32)
    lane = torch.arange(32, device="cuda")
    for o in (16, 8, 4, 2, 1):
        z = z + z[:, :, lane ^ o]
    total = torch.zeros(R, device="cuda")
    for i in range(8):
        total = total + z[:, i, 0]
    exp = x.cpu().numpy() / total.cpu().numpy()[:, None]
    assert np.array_equal(A[0].view(np.int32), exp.view(np.int32))
    k4, k8, k16 = (int(n) for n in I.quota)
    ids, cnt = V.lists()
    ids_o, cnt_o = oracle.lists(oracle.rank_row(A, k16, k8, k4))
    n = k4 + k8 + k16
    assert np.array_equal(cnt, cnt_o) and np.array_equal(ids[:, :, :n], ids_o[:, :, :n])
