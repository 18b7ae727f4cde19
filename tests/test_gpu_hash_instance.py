"""The rescan kernel's hash instance against the oracle, through the C ABI.

The library takes the instance that hashes every old end before the grid-dependency wait (one byte an
end; the scan after the wait then compares bytes and tests only the ends whose byte matches) when a
launch's context is prefetched, its grid has at least one CTA per SM and the extra shared memory keeps the
resident CTAs per SM.  The small lockstep cases of the other files prefetch nothing and run grids below the SM
count, so the cases here set the prefetch bits and force grids above it (rows x CTAs per row >= the SM count) on
short rows: filter depths 3, 2 and 1 (n_min 3, 2, 1), greedy, sampled and W-candidate verification, fused and
separate, the linear and the two-layer probe.  test_instance_taken holds that such a launch is the hash instance,
and that the same rows without the context prefetch take the other one, which runs beside it against the oracle.
"""
import ctypes

import numpy as np
import pytest

import synth
from tests import lockstep
from tests.test_gpu_candidates import compare as cand_compare, gpu_loop as cand_gpu_loop, \
    oracle_loop as cand_oracle_loop

pytestmark = pytest.mark.gpu

W = synth.WORKLOADS
PREFETCH = 3  # context and probe

# (workload, CTAs per row): rows x CTAs >= 152 SMs takes the hash instance
HASHED = {
    "zipf_f3": (W["zipf_32k"].scaled(name="zipf_f3", B=48, L0=5001, steps=12), 4),
    "mixed_f2": (W["mixed_128k"].scaled(name="mixed_f2", B=40, L0=6003, steps=10), 4),
    "uniform_f1": (W["uniform_8k"].scaled(name="uniform_f1", B=48, L0=3001, steps=12, n_min=1), 4),
    "code_mlp": (W["code_16k"].scaled(name="code_mlp", B=160, L0=2001, steps=6), 1),
}


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


CANDS = [(10, 20), (3, 8)]


def _instance(wl, split, prefetch, mode, Wc=0, D=0):
    """The template arguments (sampled, candidates, scan, two-layer probe) of the rescan kernel that a fused call
    launches."""
    import re
    import torch
    from paper_2609_20186_gb300 import binding as bd
    lib = bd.load()
    B, cap, k, d = wl.B, wl.cap, wl.k, wl.d
    i32 = dict(dtype=torch.int32, device="cuda")
    ctx, lens = torch.zeros(B, cap, **i32), torch.full((B,), wl.L0, **i32)
    W_, D_ = max(Wc, 1), max(D, k)
    draft, target, vlen = torch.zeros(B, W_, D_, **i32), torch.zeros(B, W_, D_ + 1, **i32), torch.zeros(B, **i32)
    clen, out, o1, o2 = torch.zeros(B, W_, **i32), torch.zeros(B, W_, D_, **i32), torch.zeros(B, W_, **i32), torch.zeros(B, **i32)
    acc, ch, mode_o = torch.zeros(B, **i32), torch.zeros(B, **i32), torch.zeros(B, **i32)
    f, score = torch.zeros(B, k, device="cuda"), torch.zeros(B, device="cuda")
    hidden = torch.zeros(B, d, dtype=torch.bfloat16, device="cuda")
    w = torch.zeros(max(d, (d + 1) * wl.probe_hidden), dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(max(256, bd.switchsd_workspace_bytes(B, wl.probe_kind, wl.probe_hidden, d)), dtype=torch.uint8,
                     device="cuda")

    def call(stream):
        p = bd.switchsd_params()
        p.B, p.cap, p.d, p.k, p.n_min, p.n_max, p.kappa = B, cap, d, k, wl.n_min, wl.n_max, wl.kappa
        p.probe_kind, p.probe_hidden, p.split, p.prefetch = wl.probe_kind, wl.probe_hidden, split, prefetch
        p.workspace, p.workspace_bytes, p.stream = ws.data_ptr(), ws.numel(), stream.cuda_stream
        state = (ctx.data_ptr(), lens.data_ptr(), hidden.data_ptr(), w.data_ptr(), ctypes.byref(p))
        tail = (mode_o.data_ptr(), score.data_ptr())
        if mode == "candidates":
            code = lib.switchsd_verify_candidates_step(
                draft.data_ptr(), target.data_ptr(), clen.data_ptr(), vlen.data_ptr(), acc.data_ptr(), ch.data_ptr(), *state,
                Wc, D, out.data_ptr(), o1.data_ptr(), o2.data_ptr(), *tail)
        elif mode == "sampled":
            code = lib.switchsd_verify_sampled_step(
                draft.data_ptr(), f.data_ptr(), f.data_ptr(), f.data_ptr(), target.data_ptr(), vlen.data_ptr(),
                acc.data_ptr(), *state, out.data_ptr(), o2.data_ptr(), *tail)
        else:
            code = lib.switchsd_verify_step(draft.data_ptr(), target.data_ptr(), vlen.data_ptr(), acc.data_ptr(), *state,
                                            out.data_ptr(), o2.data_ptr(), *tail)
        assert code == bd.OK
    names = [n for n in lockstep.kernel_names(call) if "rescan_kernel" in n]
    assert len(set(names)) == 1, names
    m = re.search(r"rescan_kernelILb(\d)ELb(\d)ELi(\d)ELb(\d)E", names[0])
    return tuple(int(x) for x in m.groups())


@pytest.mark.parametrize("mode,Wc,D", [("greedy", 0, 0), ("sampled", 0, 0)] + [("candidates", *c) for c in CANDS])
@pytest.mark.parametrize("name", list(HASHED))
def test_instance_taken(name, mode, Wc, D):
    wl, split = HASHED[name]
    assert wl.B * split >= _sms()  # with the context prefetch, the grid that selects the hash instance
    kind = (int(mode == "sampled"), int(mode == "candidates"))
    assert _instance(wl, split, PREFETCH, mode, Wc, D) == (*kind, 1, wl.probe_kind)
    assert _instance(wl, split, PREFETCH & ~1, mode, Wc, D) == (*kind, 0, wl.probe_kind)


def test_instance_of_the_full_size_workloads():
    """The prefetched full-size parity tests run the benchmark's instances: the hash one but where the grid is smaller
    (uniform_8k) or the hash bytes would cost a resident CTA (code_16k)."""
    from tests.test_gpu_parity import PREFETCHED_STEPS
    for name, scan in (("zipf_32k", 1), ("mixed_128k", 1), ("code_16k", 0), ("uniform_8k", 0)):
        wl = W[name].scaled(steps=PREFETCHED_STEPS)
        assert _instance(wl, 0, PREFETCH, "greedy") == (0, 0, scan, wl.probe_kind), name


@pytest.mark.parametrize("fused", [False, True], ids=["separate", "fused"])
@pytest.mark.parametrize("name", list(HASHED))
def test_hash_instance_lockstep(name, fused):
    wl, split = HASHED[name]
    rows = range(wl.B)
    o_trace, o_ctx, _ = lockstep.oracle_trace_rows(wl, wl.B, wl.steps)
    g_trace, g_ctx, _ = lockstep.gpu_trace(wl, wl.steps, split=split, fused=fused, prefetch=PREFETCH)
    flips, stats = lockstep.compare(wl, o_trace, g_trace, rows, o_ctx, g_ctx)
    assert stats["checked"] > 0 and len(flips) <= 1
    # the same rows and grid without the prefetch (the instance without the hash bytes)
    g2, g2_ctx, _ = lockstep.gpu_trace(wl, wl.steps, split=split, fused=fused)
    lockstep.compare(wl, o_trace, g2, rows, o_ctx, g2_ctx)


@pytest.mark.parametrize("name", ["zipf_f3", "mixed_f2"])
def test_hash_instance_sampled(name):
    wl, split = HASHED[name]
    rows = range(wl.B)
    o_trace, o_ctx, _ = lockstep.oracle_trace(wl, rows, wl.steps, sampled=True)
    g_trace, g_ctx, _ = lockstep.gpu_trace(wl, wl.steps, sampled=True, split=split, fused=True, prefetch=PREFETCH)
    flips, stats = lockstep.compare(wl, o_trace, g_trace, rows, o_ctx, g_ctx)
    assert stats["checked"] > 0 and len(flips) <= 1


@pytest.mark.parametrize("name,Wc,D", [(n, *c) for n in ("zipf_f3", "uniform_f1") for c in CANDS] + [("code_mlp", *CANDS[0])])
def test_hash_instance_candidates(name, Wc, D):
    wl, split = HASHED[name]
    wl = wl.scaled(k=max(wl.k, D))  # row capacity for appends of up to D + 1 tokens a step
    rows = range(0, wl.B, 4 if wl.probe_kind else 1)
    o_trace, o_ctx = cand_oracle_loop(wl, rows, wl.steps, Wc, D)
    g_trace, g_ctx = cand_gpu_loop(wl, wl.steps, Wc, D, split=split, fused=True, prefetch=PREFETCH)
    checked, _ = cand_compare(wl, o_trace, g_trace, rows, o_ctx, g_ctx)
    assert checked > 0
