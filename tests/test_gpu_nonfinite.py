"""A NaN among the inputs: it takes no part in the maxima that the quantiser scales come from (App. C.3 as the oracle
computes it), so that scales, codes and outputs of blocks that do not hold or attend to it stay what they are without it.
"""
import numpy as np
import pytest
import torch

import da2_inputs
import oracle
import paper_2609_32628_b200 as da2
from helpers import Workspace, compare_lists, oracle_all, run_gpu
from test_gpu_parity import _check_attention

pytestmark = pytest.mark.gpu
W = da2_inputs.Workload


def _same(got, exp, keep, what):
    assert np.array_equal(got[keep], exp[keep]), what


def _check_operands(plan, ws, ref, dv=None, g=None):
    """Scales and codes against the oracle, the NaN elements' own codes left out.  g, dv: scales that were carried over."""
    V, pl = Workspace(plan, ws), ref["pl"]
    st = np.maximum(pl.slot_token, 0)
    num = {n: np.where((pl.slot_token >= 0)[None, :, :, None], (ref[n][:, st] & 0x7fff) <= 0x7f80, True) for n in ("q", "k", "v")}
    if g is None:
        g = np.stack([oracle.nvfp4_global_scale(ref[n]) for n in ("q", "k", "v")], 1)
    assert np.array_equal(V.gscale(), g)
    for i, n in enumerate(("q", "k")):
        codes, delta = oracle.quant_int8(ref[n], pl)
        assert np.array_equal(V.dq8() if n == "q" else V.dk8(), delta), n
        _same(V.q_or_k_int8(n), codes, num[n], f"int8 {n}")
        codes, sf = oracle.quant_nvfp4_qk(ref[n], pl, np.ascontiguousarray(g[:, i]))
        gc, gsf = V.q_or_k_fp4(n)
        assert np.array_equal(gsf, sf), n
        _same(gc, codes, num[n], f"nvfp4 {n}")
    codes, dc = oracle.quant_v_e4m3(ref["v"], pl)
    if dv is not None:
        dc, codes = dv, oracle.quant_v_e4m3_given(ref["v"], pl, dv)
    assert np.array_equal(V.dv8(), dc)
    _same(V.v_e4m3(), codes, num["v"], "e4m3 v")
    codes, sf = oracle.quant_nvfp4_v(ref["v"], pl, np.ascontiguousarray(g[:, 2]))
    gc, gsf = V.v_fp4()
    assert np.array_equal(gsf, sf), "v"
    _same(gc, codes, num["v"], "nvfp4 v")


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("channels", [(0,), (1,), (0, 1)])
@pytest.mark.parametrize("which", ["q", "k", "v"])
def test_nan_stays_out_of_the_scales(which, channels, d):
    """The NaN sits in a low, a high or both halves of a packed pair; the largest values of the head are in channels 2 and 3."""
    w = W("nan", 1, 2, d, 3, 12, 20, 0.1, 0.2, 0.3, seed=41)
    x = dict(zip("qkv", da2_inputs.make_qkv(w, "cuda")))
    for t in x.values():
        t[..., 2:4] *= 6.0
    clean = {n: t.clone() for n, t in x.items()}
    pl = oracle.plan(w.T, w.Hg, w.Wg)
    block = pl.R - 1
    for c in channels:
        x[which][0, 0, int(pl.slot_token[block, 1]), c] = float("nan")
    plan, ws, out = run_gpu(w, x["q"], x["k"], x["v"])
    ref = oracle_all(w, x["q"], x["k"], x["v"])
    _check_operands(plan, ws, ref)
    ids, cnt = Workspace(plan, ws).lists()
    # a row of scores that are no numbers is a tie throughout: the lower indices
    bad, _ = compare_lists(np.nan_to_num(ref["A"], nan=0.0), ref["ids"], ref["counts"], ids, cnt)
    sel = [(h, a) for h in range(2) for a in range(pl.R)
           if h == 1 or (a != block if which == "q" else block not in ids[0, a])]
    _check_attention(w, out, ref, sel, bad)
    # carried-over scales: the block's own scale and the group scales are still derived
    da2.da2_prepare(plan, clean["q"], clean["k"], clean["v"], ws)
    V = Workspace(plan, ws)
    g, dv = V.gscale(), V.dv8()
    da2.da2_prepare_cached_scales(plan, x["q"], x["k"], x["v"], ws, reselect=True)
    _check_operands(plan, ws, ref, dv=dv, g=g)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("slot_of", ["full", "edge"])
def test_nan_key_reaches_every_query_that_attends_to_it(slot_of, d):
    """bf16 products carry a NaN key into each output row that keeps its block, whether or not the block has padding slots
    beside it; the other head is untouched."""
    w = W("nan16", 1, 2, d, 3, 12, 20, 1.0, 0.0, 0.0, seed=42)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    pl = oracle.plan(w.T, w.Hg, w.Wg)
    full = int((pl.slot_token >= 0).sum(1).argmax())
    block = full if slot_of == "full" else pl.R - 1
    assert ((pl.slot_token[block] < 0).any()) == (slot_of == "edge")
    k[0, 0, int(pl.slot_token[block, 0]), 5] = float("nan")
    plan, ws, out = run_gpu(w, q, k, v)
    assert torch.isnan(out[0, 0]).all()
    ref = oracle_all(w, q, k, v)
    _check_attention(w, out, ref, [(1, a) for a in range(pl.R)], [])


@pytest.mark.parametrize("f16,f8,f4", [(0.1, 0.2, 0.3), (0.0, 0.3, 0.0), (0.5, 0.25, 0.25)])
@pytest.mark.parametrize("T,Hg,Wg", [(1, 8, 8), (1, 24, 56), (13, 8, 40), (23, 24, 56), (61, 24, 56), (683, 8, 24)])
def test_rows_of_nan_scores_keep_the_lower_indices(T, Hg, Wg, f16, f8, f4):
    """A NaN in K makes every score of its head NaN: all rows of head 0 are one tie; head 1 has its ordinary lists."""
    w = W("nanrows", 1, 2, 64, T, Hg, Wg, f16, f8, f4, seed=43)
    q, k, v = da2_inputs.make_qkv(w, "cuda")
    k[0, 0, w.N // 2, 7] = float("nan")
    plan = da2.da2_plan(w.B, w.H, w.T, w.Hg, w.Wg, w.head_dim, f16, f8, f4)
    ws = torch.empty(int(plan.info.workspace_bytes), dtype=torch.uint8, device="cuda")
    da2.da2_prepare(plan, q, k, v, ws)
    torch.cuda.synchronize()
    ids, cnt = Workspace(plan, ws, [0]).lists()
    k4, k8, k16 = (int(x) for x in plan.info.quota)
    n = k4 + k8 + k16
    assert (cnt == np.array([k4, k8, k16])).all()
    assert (ids[0, :, :n] == np.r_[k16 + k8:n, k16:k16 + k8, 0:k16]).all()
    ref = oracle_all(w, q, k, v, heads=[1])
    compare_lists(ref["A"], ref["ids"], ref["counts"], *Workspace(plan, ws, [1]).lists())
