"""The rescan kernel's hash instance, which a launch takes when the context is prefetched and the grid has at
least one CTA per SM, against the instance that the same rows take without the prefetch (itself held to the
oracle by the lockstep tests): bit-identical outputs for every filter depth, greedy and sampled verification, W
candidates and the two-layer probe, at a range that ends inside a round of the first pass."""
import ctypes

import numpy as np
import pytest

import synth
from tests.test_gpu_hash_instance import HASHED

pytestmark = pytest.mark.gpu


def _session(wl, split, prefetch):
    from paper_2609_20186_gb300 import Session
    ctx, lens = wl.contexts()
    return Session(ctx, lens, wl.probe_weights(), k=wl.k, n_min=wl.n_min, n_max=wl.n_max, kappa=wl.kappa,
                   logit_tau=wl.logit_tau, probe_kind=wl.probe_kind, probe_hidden=wl.probe_hidden, future=wl.future(),
                   harness=wl.harness_params(), d=wl.d, split=split, prefetch=prefetch)


@pytest.mark.parametrize("sampled", [False, True], ids=["greedy", "sampled"])
@pytest.mark.parametrize("name", list(HASHED))
def test_chain(name, sampled):
    import torch
    from paper_2609_20186_gb300 import bf16_tensor
    wl, split = HASHED[name]
    a, b = _session(wl, split, 0), _session(wl, split, 3)
    hidden = bf16_tensor(np.stack([wl.hidden(t) for t in range(wl.steps)]), a.device)
    torch.cuda.synchronize()
    for t in range(wl.steps):
        for s in (a, b):
            if t == 0:
                s.step(hidden[0])
            elif sampled:
                s.verify_sampled_step(hidden[t])
            else:
                s.verify_step(hidden[t])
        for key in ("len", "mode", "score", "match_n", "match_end", "status", "accept", "lens"):
            assert torch.equal(getattr(a, key), getattr(b, key)), (t, key)
        live = torch.arange(wl.k, device="cuda") < a.len[:, None]
        assert torch.equal(a.draft[live], b.draft[live]), t
        for s in (a, b):  # the kernel before the next call writes neither contexts nor hidden states
            if sampled:
                s.harness_sampled(t)
            else:
                s.harness(t)
    assert torch.equal(a.ctx, b.ctx)


@pytest.mark.parametrize("name", ["zipf_f3", "mixed_f2", "uniform_f1"])
def test_candidates(name):
    import torch
    from paper_2609_20186_gb300 import binding as bd, bf16_tensor
    lib = bd.load()
    wl, split = HASHED[name]
    ctx, lens = wl.contexts()
    B, cap = ctx.shape
    W, D = 10, 20
    c, ln = torch.from_numpy(ctx).cuda(), torch.from_numpy(lens).cuda()
    h, w = bf16_tensor(wl.hidden(0), "cuda"), bf16_tensor(wl.probe_weights(), "cuda")
    out = []
    for prefetch in (0, 3):
        i32 = dict(dtype=torch.int32, device="cuda")
        o = dict(cand=torch.zeros(B, W, D, **i32), cand_len=torch.zeros(B, W, **i32), ncand=torch.zeros(B, **i32),
                 mode=torch.zeros(B, **i32), score=torch.zeros(B, device="cuda"), n=torch.zeros(B, **i32),
                 e=torch.zeros(B, **i32))
        p = bd.switchsd_params()
        p.B, p.cap, p.d, p.k, p.n_min, p.n_max, p.split, p.prefetch = B, cap, wl.d, D, wl.n_min, wl.n_max, split, prefetch
        p.logit_tau = float("-inf")
        p.out_match_n, p.out_match_end = o["n"].data_ptr(), o["e"].data_ptr()
        p.stream = torch.cuda.current_stream().cuda_stream
        assert lib.switchsd_step_candidates(c.data_ptr(), ln.data_ptr(), h.data_ptr(), w.data_ptr(), ctypes.byref(p), W, D,
                                            o["cand"].data_ptr(), o["cand_len"].data_ptr(), o["ncand"].data_ptr(),
                                            o["mode"].data_ptr(), o["score"].data_ptr()) == bd.OK
        out.append(o)
    a, b = out
    for key in ("ncand", "mode", "score", "n", "e"):
        assert torch.equal(a[key], b[key]), key
    assert int(a["ncand"].max()) > 0
    live = torch.arange(W, device="cuda") < a["ncand"][:, None]
    assert torch.equal(a["cand_len"][live], b["cand_len"][live])
    tok = live[:, :, None] & (torch.arange(D, device="cuda") < a["cand_len"][:, :, None])
    assert torch.equal(a["cand"][tok], b["cand"][tok])
