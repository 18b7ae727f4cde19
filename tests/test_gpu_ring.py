"""The rescan kernel's ring of tiles (CTA ranges above 16,384 ends) at the sizes where it can go wrong, against
the oracle: a range one past the one-copy form, ranges that end at, just before and just after a tile and
after the ring has gone round, appends that cross a tile's end, each filter depth, each verification rule, W
candidates, the two-layer probe, a length bound, and a row past 2^25 tokens (the one-copy form's match keys
hold an end below that)."""
import numpy as np
import pytest

import synth
from tests import lockstep
from tests.test_gpu_candidates import compare as cand_compare, gpu_loop as cand_gpu_loop, \
    oracle_loop as cand_oracle_loop

pytestmark = pytest.mark.gpu

W = synth.WORKLOADS


@pytest.mark.parametrize("L0,n_min,sampled", [(16400, 3, False), (24574, 2, False), (24577, 1, True), (32765, 3, True),
                                              (40960, 3, False), (57341, 2, True)])
def test_one_cta_rows(L0, n_min, sampled):
    wl = W["mixed_128k"].scaled(name=f"ring_{L0}", B=3, L0=L0, steps=5, n_min=n_min, k=12)
    o_trace, o_ctx, _ = lockstep.oracle_trace(wl, range(wl.B), wl.steps, sampled=sampled)
    g_trace, g_ctx, _ = lockstep.gpu_trace(wl, wl.steps, split=1, fused=True, sampled=sampled)
    _, stats = lockstep.compare(wl, o_trace, g_trace, range(wl.B), o_ctx, g_ctx)
    assert stats["checked"] == wl.B * wl.steps


@pytest.mark.parametrize("name,L0,split", [("zipf_32k", 40001, 1), ("code_16k", 34001, 2)])
def test_candidates_and_two_layer_probe(name, L0, split):
    wl = W[name].scaled(name=f"{name}_ring", B=3, L0=L0, steps=3)
    if wl.probe_kind == 1:
        o_trace, o_ctx, _ = lockstep.oracle_trace(wl, range(wl.B), wl.steps)
        g_trace, g_ctx, _ = lockstep.gpu_trace(wl, wl.steps, split=split, fused=True)
        lockstep.compare(wl, o_trace, g_trace, range(wl.B), o_ctx, g_ctx)
    o_trace, o_ctx = cand_oracle_loop(wl, range(wl.B), wl.steps, 10, 20)
    g_trace, g_ctx = cand_gpu_loop(wl, wl.steps, 10, 20, split=split, fused=True)
    checked, _ = cand_compare(wl, o_trace, g_trace, range(wl.B), o_ctx, g_ctx)
    assert checked > 0


def test_length_bound_and_prefetch():
    """A bound far above the lengths (tiles past every row's end are staged and skipped) and the prefetch bits:
    bit-identical to the plain call."""
    import torch
    from paper_2609_20186_gb300 import Session, binding as bd, bf16_tensor
    wl = W["zipf_32k"].scaled(name="ring_bound", B=4, L0=33333, steps=600)
    ctx, lens = wl.contexts()
    lens[1] = 16000
    lens[2] = 1
    res = []
    for bound, prefetch in ((0, 0), (ctx.shape[1], bd.PREFETCH_CONTEXT | bd.PREFETCH_PROBE)):
        s = Session(ctx, lens, wl.probe_weights(), k=wl.k, n_min=wl.n_min, n_max=wl.n_max, d=wl.d, split=1,
                    len_bound=bound, prefetch=prefetch)
        s.step(bf16_tensor(wl.hidden(0), s.device))
        torch.cuda.synchronize()
        res.append(s.step_outputs())
    for key in ("len", "mode", "score", "match_n", "match_end", "status"):
        assert np.array_equal(res[0][key], res[1][key]), key
    for b in range(wl.B):
        n = int(res[0]["len"][b])
        assert np.array_equal(res[0]["draft"][b, :n], res[1]["draft"][b, :n])


def test_row_past_the_key_range():
    """One row of 2^25 + 64 tokens; the only earlier occurrence of its suffix lies past 2^25 - 64, then near
    the row's start."""
    import torch
    from paper_2609_20186_gb300 import Session, bf16_tensor
    L = (1 << 25) + 64
    x = np.arange(L, dtype=np.int32)
    for end in (L - 60, 5000):
        row = x.copy()
        row[L - 6:] = row[end - 5:end + 1]
        s = Session(row[None, :], np.array([L], np.int32), np.zeros(8, np.uint16), k=8, n_min=3, n_max=8,
                    logit_tau=float("-inf"), d=8)
        s.step(bf16_tensor(np.zeros((1, 8), np.uint16), s.device))
        torch.cuda.synchronize()
        o = s.step_outputs()
        assert (int(o["match_n"][0]), int(o["match_end"][0]), int(o["mode"][0])) == (6, end, 1)
        assert o["draft"][0, :8].tolist() == row[end + 1:end + 9].tolist()
