"""The two-layer probe's first layer at the sizes where its split of K changes, against the oracle's probe in
double precision: one and two parts of K a CTA with tiles of 64 and 128 units (past 10 MB of partial sums; two parts
where enough CTAs are left: 330 x 512 at d = 4096 and 8192 stand on either side), parts without a chunk of K
(17 chunks over 16 parts), one and two chunks of K in all, ragged last tiles of rows and units, several units a
thread of the rescan kernel, a bias, and the grids that stage all, three or two chunks at once.

The sums run over d products of bf16 values in fp32 (parts of at most d / 16 terms, added in order) and H1
units; |Delta z| <= 1e-3 is the repository's bar for the logit (values of order one).
"""
import numpy as np
import pytest

import oracle
from tests.lockstep import SCORE_TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H1,d", [(330, 512, 1096), (330, 509, 4096), (170, 1024, 2048), (16, 100, 64), (129, 65, 136),
                                    (700, 256, 512), (64, 256, 5120), (300, 128, 8192), (330, 512, 8192), (256, 768, 5120),
                                    (400, 448, 4096), (4, 512, 8192), (1300, 128, 5120)])
@pytest.mark.parametrize("prefetch", [0, 2])
def test_first_layer_parts(B, H1, d, prefetch):
    import torch
    from paper_2609_20186_gb300 import binding as bd, bf16_tensor
    from synth.rng import bf16_bits_from_f32
    rng = np.random.default_rng(B * 1000003 + H1 * 1009 + d)
    h = bf16_bits_from_f32(rng.standard_normal((B, d), dtype=np.float32))
    W1 = bf16_bits_from_f32(rng.standard_normal((H1, d), dtype=np.float32) / np.float32(d ** 0.5))
    w2 = bf16_bits_from_f32(rng.standard_normal(H1, dtype=np.float32) / np.float32(H1 ** 0.5))
    b1 = rng.standard_normal(H1).astype(np.float32)
    ctx = torch.from_numpy(rng.integers(0, 50, (B, 64)).astype(np.int32)).cuda()
    lens = torch.full((B,), 60, dtype=torch.int32, device="cuda")
    out = {n: torch.zeros(B, dtype=torch.int32, device="cuda") for n in ("len", "mode")}
    draft = torch.zeros(B, 4, dtype=torch.int32, device="cuda")
    score = torch.zeros(B, device="cuda")
    w = bf16_tensor(np.concatenate([W1.reshape(-1), w2]), "cuda")
    hd = bf16_tensor(h, "cuda")
    b1d = torch.from_numpy(b1).cuda()
    ws = torch.empty(bd.switchsd_workspace_bytes(B, bd.PROBE_MLP, H1, d), dtype=torch.uint8, device="cuda")
    for _ in range(3):  # back to back: with the prefetch bit the first layer runs beside the call before it
        bd.switchsd_step(ctx, lens, hd, w, draft, out["len"], out["mode"], score, k=4, n_min=3, n_max=5,
                         probe_kind=bd.PROBE_MLP, probe_hidden=H1, b1=b1d, b2=0.25,
                         workspace=ws, prefetch=prefetch)
    z = score.cpu().numpy()
    for b in (0, 1, 126, 127, 128, B // 2, B - 2, B - 1):
        if 0 <= b < B:
            assert abs(float(z[b]) - oracle.probe_mlp(h[b], W1, w2, b1=b1, b2=0.25)) <= SCORE_TOL, b


@pytest.mark.parametrize("B,H1,d", [(330, 512, 8192), (330, 512, 4096), (4, 512, 8192), (130, 64, 5120)])
def test_first_layer_with_the_index(B, H1, d):
    """The same before the index kernel, where nothing else runs beside it and a CTA stages all the chunks that fit."""
    import ctypes
    import torch
    from paper_2609_20186_gb300 import binding as bd, bf16_tensor
    from synth.rng import bf16_bits_from_f32
    rng = np.random.default_rng(B + H1 + d)
    h = bf16_bits_from_f32(rng.standard_normal((B, d), dtype=np.float32))
    W1 = bf16_bits_from_f32(rng.standard_normal((H1, d), dtype=np.float32) / np.float32(d ** 0.5))
    w2 = bf16_bits_from_f32(rng.standard_normal(H1, dtype=np.float32) / np.float32(H1 ** 0.5))
    ctx = torch.from_numpy(rng.integers(0, 50, (B, 64)).astype(np.int32)).cuda()
    lens = torch.full((B,), 60, dtype=torch.int32, device="cuda")
    index = bd.NgramIndex(B, 64, 3, 5)
    index.build(ctx, lens)
    ln, mode, draft = (torch.zeros(*s, dtype=torch.int32, device="cuda") for s in ((B,), (B,), (B, 4)))
    score = torch.zeros(B, device="cuda")
    w, hd = bf16_tensor(np.concatenate([W1.reshape(-1), w2]), "cuda"), bf16_tensor(h, "cuda")
    ws = torch.empty(bd.switchsd_workspace_bytes(B, bd.PROBE_MLP, H1, d), dtype=torch.uint8, device="cuda")
    p = bd.switchsd_params()
    p.B, p.cap, p.d, p.k, p.n_min, p.n_max = B, 64, d, 4, 3, 5
    p.probe_kind, p.probe_hidden, p.workspace, p.workspace_bytes = bd.PROBE_MLP, H1, ws.data_ptr(), ws.numel()
    p.index, p.stream = index.handle, torch.cuda.current_stream().cuda_stream
    assert bd.load().switchsd_step(ctx.data_ptr(), lens.data_ptr(), hd.data_ptr(), w.data_ptr(), ctypes.byref(p),
                                   draft.data_ptr(), ln.data_ptr(), mode.data_ptr(), score.data_ptr()) == bd.OK
    z = score.cpu().numpy()
    for b in (0, 1, 127, 128, B // 2, B - 1):
        if b < B:
            assert abs(float(z[b]) - oracle.probe_mlp(h[b], W1, w2, b1=None, b2=0.0)) <= SCORE_TOL, b
    index.close()
