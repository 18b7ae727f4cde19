"""Kernels launched right behind a step that appends, with no synchronisation between: every kernel starts while the
one before it runs, so each must read what that one wrote.  After each fused step the labels of the grown rows are
taken and the index is rebuilt and searched; the search must agree with the rescan that the fused step made over
the same context, the labels with the oracle's."""
import ctypes

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

W = synth.WORKLOADS


@pytest.mark.parametrize("name,B,L0,n", [("zipf_32k", 40, 3001, 5), ("code_16k", 16, 20001, 8), ("uniform_8k", 3, 17001, 3)])
def test_labels_and_index_behind_an_append(name, B, L0, n):
    import torch
    from paper_2609_20186_gb300 import Session, bf16_tensor, binding as bd
    wl = W[name].scaled(name=f"{name}_behind", B=B, L0=L0, steps=8, probe_kind=0, d=512)
    ctx, lens = wl.contexts()
    s = Session(ctx, lens, wl.probe_weights(), k=wl.k, n_min=wl.n_min, n_max=wl.n_max, kappa=wl.kappa,
                logit_tau=wl.logit_tau, future=wl.future(), harness=wl.harness_params(), d=wl.d)
    hidden = bf16_tensor(np.stack([wl.hidden(t) for t in range(wl.steps)]), s.device)
    cap = s.cap
    index = bd.NgramIndex(B, cap, wl.n_min, wl.n_max)
    ws = torch.empty(int(s.lib.switchsd_labels_workspace_bytes(B, cap)), dtype=torch.uint8, device="cuda")
    lab = torch.zeros((wl.steps, B, cap), dtype=torch.uint8, device="cuda")
    rec = {key: torch.zeros((wl.steps, B), dtype=torch.int32, device="cuda") for key in ("n", "e", "in", "ie", "lens")}
    i32 = dict(dtype=torch.int32, device="cuda")
    idraft, ilen, imode = torch.zeros(B, wl.k, **i32), torch.zeros(B, **i32), torch.zeros(B, **i32)
    iscore = torch.zeros(B, device="cuda")
    torch.cuda.synchronize()
    for t in range(wl.steps):
        if t == 0:
            s.step(hidden[0])
        else:
            s.verify_step(hidden[t])
        bd.switchsd_copy_labels(s.ctx, s.lens, lab[t], n=n, workspace=ws)
        index.build(s.ctx, s.lens)
        p = bd.switchsd_params()
        p.B, p.cap, p.d, p.k, p.n_min, p.n_max, p.kappa = B, cap, wl.d, wl.k, wl.n_min, wl.n_max, wl.kappa
        p.index = index.handle
        p.out_match_n, p.out_match_end = rec["in"][t].data_ptr(), rec["ie"][t].data_ptr()
        p.stream = torch.cuda.current_stream().cuda_stream
        assert s.lib.switchsd_step(s.ctx.data_ptr(), s.lens.data_ptr(), hidden[t].data_ptr(), s.probe_w.data_ptr(),
                                   ctypes.byref(p), idraft.data_ptr(), ilen.data_ptr(), imode.data_ptr(),
                                   iscore.data_ptr()) == bd.OK
        rec["n"][t].copy_(s.match_n), rec["e"][t].copy_(s.match_end), rec["lens"][t].copy_(s.lens)
        s.harness(t)
    torch.cuda.synchronize()
    r = {key: v.cpu().numpy() for key, v in rec.items()}
    final, got = s.ctx.cpu().numpy(), lab.cpu().numpy()
    assert (r["lens"][-1] > lens).all()  # every row grew
    assert np.array_equal(r["n"], r["in"]) and np.array_equal(r["e"], r["ie"])
    for t in (0, 1, wl.steps - 1):  # contexts only grow: a step's context is a prefix of the last one
        for b in (0, B // 2, B - 1):
            L = int(r["lens"][t, b])
            assert np.array_equal(got[t, b, :L], oracle.copy_labels(final[b, :L], n)), (t, b)
            assert not got[t, b, L:].any()
    index.close()
