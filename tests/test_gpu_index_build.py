"""switchsd_index_build against the oracle at the sizes where its chunked radix pass can go wrong.

The build takes a row in chunks (4,096, 8,192 or 16,384 positions for capacities up to those, else 32,768), splits the
buckets over several CTAs (few rows, or more than 2^17 buckets), and drops the positions below n - 1.  The
rows here end just below, at and above those sizes, and hold a period-1 and a period-7 run (one bucket takes
everything), a small alphabet (dense repeats) and uniform ids.  Every chain is read back through the
candidate step: for every gate length kappa it lists the W most recent ends of the kappa-gram, at the built
length and at shorter ones (ends past the length are skipped).

Rows of up to 256 tokens, many rows of up to 2,048, and many of more than 262,144 are built by a warp per row and n
instead (capacity 260 with 240 and 300 of them stands on either side).
"""
import ctypes

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

# (length, rows, n_min, n_max)
SHAPES = [(1, 2, 1, 3), (7, 3, 3, 8), (33, 5, 2, 12), (255, 9, 3, 8), (257, 40, 3, 8), (258, 50, 3, 8), (1000, 40, 3, 8),
          (1001, 170, 3, 8), (1801, 310, 3, 8), (4096, 5, 2, 5),
          (4097, 4, 3, 5), (8192, 4, 3, 5), (8193, 5, 2, 4), (16383, 4, 3, 8), (16385, 4, 3, 8),
          (32768, 4, 2, 4), (32769, 5, 1, 2), (70001, 4, 3, 5), (140003, 4, 2, 3),
          # rows enough that a CTA takes all of an item's buckets (its links go out through shared memory), of every
          # instance, with one chunk and with a second one
          (4095, 40, 3, 6), (8192, 40, 3, 5), (16384, 40, 3, 5), (32768, 40, 3, 5), (32770, 40, 3, 5), (40001, 40, 3, 5),
          (65536, 40, 3, 5)]


def _rows(L, B, rng):
    x = np.zeros((B, L), np.int32)
    for b in range(B):
        kind = b % 4
        if kind == 0:
            x[b] = rng.integers(0, 12, L)
        elif kind == 1:
            x[b] = 7
        elif kind == 2:
            x[b] = np.tile(rng.integers(0, 1 << 30, 7), L // 7 + 1)[:L]
        else:
            x[b] = rng.integers(-(1 << 31), 1 << 31, L)
            if L > 600:
                x[b, L - 200:] = x[b, 100:300]
    return x


@pytest.mark.parametrize("L,B,n_min,n_max", SHAPES, ids=[f"L{s[0]}_{s[1]}" for s in SHAPES])
def test_built_chains(L, B, n_min, n_max):
    import torch
    from paper_2609_20186_gb300 import binding as bd
    lib = bd.load()
    rng = np.random.default_rng(L)
    cap = (L + 3) // 4 * 4
    W, D, d, k = 16, 4, 8, 4
    ctx = np.zeros((B, cap), np.int32)
    ctx[:, :L] = _rows(L, B, rng)
    lens = np.full(B, L, np.int32)
    if B > 3:
        lens[3] = max(1, L - 5)
    c = torch.from_numpy(ctx).cuda()
    ln = torch.from_numpy(lens).cuda()
    idx = bd.NgramIndex(B, cap, n_min, n_max)
    idx.build(c, ln)
    idx.build(c, ln)  # a rebuild leaves the same index
    h = torch.ones(B, d, dtype=torch.bfloat16, device="cuda")
    w = torch.ones(d, dtype=torch.bfloat16, device="cuda")
    hb = np.full((B, d), 0x3F80, np.uint16)

    def ints(*s):
        return torch.zeros(s, dtype=torch.int32, device="cuda")

    for cut in sorted({0, 1, 2, min(40, L // 2), L // 3}):
        lens_c = np.maximum(lens - cut, 1).astype(np.int32)
        ln.copy_(torch.from_numpy(lens_c))
        for kappa in range(n_min, n_max + 1):
            cand, cl, nc, mode = ints(B, W, D), ints(B, W), ints(B), ints(B)
            mn, me = ints(B), ints(B)
            score = torch.zeros(B, device="cuda")
            p = bd.switchsd_params()
            p.B, p.cap, p.d, p.k, p.n_min, p.n_max, p.kappa = B, cap, d, k, n_min, n_max, kappa
            p.logit_tau = float("-inf")
            p.index = idx.handle
            p.out_match_n, p.out_match_end = mn.data_ptr(), me.data_ptr()
            p.stream = torch.cuda.current_stream().cuda_stream
            assert lib.switchsd_step_candidates(c.data_ptr(), ln.data_ptr(), h.data_ptr(), w.data_ptr(), ctypes.byref(p),
                                                W, D, cand.data_ptr(), cl.data_ptr(), nc.data_ptr(), mode.data_ptr(),
                                                score.data_ptr()) == bd.OK
            o = oracle.step_candidates(ctx, lens_c, hb, hb[0], W=W, D=D, n_min=n_min, n_max=n_max, kappa=kappa,
                                       logit_tau=float("-inf"))
            assert np.array_equal(mn.cpu().numpy(), o["match_n"]), (cut, kappa)
            assert np.array_equal(me.cpu().numpy(), o["match_end"]), (cut, kappa)
            assert np.array_equal(mode.cpu().numpy(), o["mode"]), (cut, kappa)
            assert np.array_equal(nc.cpu().numpy(), o["ncand"]), (cut, kappa)
            g, gl = cand.cpu().numpy(), cl.cpu().numpy()
            for b in range(B):
                for i in range(int(o["ncand"][b])):
                    m = int(o["cand_len"][b, i])
                    assert gl[b, i] == m and np.array_equal(g[b, i, :m], o["cand"][b, i, :m]), (cut, kappa, b, i)
    idx.close()


def test_many_long_rows():
    """34 rows past 262,144 tokens with 31 n: the warp-per-item build, read back for the shortest, a middle and the
    longest n of the first four rows and the last."""
    import torch
    from paper_2609_20186_gb300 import binding as bd
    lib = bd.load()
    B, L, n_min, n_max, W, D, d, k = 34, 262145, 2, 32, 16, 4, 8, 4
    cap = (L + 3) // 4 * 4
    ctx = np.zeros((B, cap), np.int32)
    ctx[:, :L] = _rows(L, B, np.random.default_rng(L))
    lens = np.full(B, L, np.int32)
    c, ln = torch.from_numpy(ctx).cuda(), torch.from_numpy(lens).cuda()
    idx = bd.NgramIndex(B, cap, n_min, n_max)
    idx.build(c, ln)
    h = torch.ones(B, d, dtype=torch.bfloat16, device="cuda")
    hb = np.full((B, d), 0x3F80, np.uint16)

    def ints(*s):
        return torch.zeros(s, dtype=torch.int32, device="cuda")

    for kappa in (n_min, 9, n_max):
        cand, cl, nc, mode, mn, me = ints(B, W, D), ints(B, W), ints(B), ints(B), ints(B), ints(B)
        score = torch.zeros(B, device="cuda")
        p = bd.switchsd_params()
        p.B, p.cap, p.d, p.k, p.n_min, p.n_max, p.kappa = B, cap, d, k, n_min, n_max, kappa
        p.logit_tau = float("-inf")
        p.index = idx.handle
        p.out_match_n, p.out_match_end = mn.data_ptr(), me.data_ptr()
        p.stream = torch.cuda.current_stream().cuda_stream
        assert lib.switchsd_step_candidates(c.data_ptr(), ln.data_ptr(), h.data_ptr(), h.data_ptr(), ctypes.byref(p), W, D,
                                            cand.data_ptr(), cl.data_ptr(), nc.data_ptr(), mode.data_ptr(),
                                            score.data_ptr()) == bd.OK
        for b in (0, 1, 2, 3, B - 1):
            o = oracle.step_candidates(ctx, lens, hb, hb[0], W=W, D=D, n_min=n_min, n_max=n_max, kappa=kappa,
                                       logit_tau=float("-inf"), rows=(b, b + 1))
            assert (int(mn[b]), int(me[b]), int(nc[b])) == (o["match_n"][b], o["match_end"][b], o["ncand"][b]), (kappa, b)
            for i in range(int(o["ncand"][b])):
                m = int(o["cand_len"][b, i])
                assert int(cl[b, i]) == m and cand[b, i, :m].tolist() == o["cand"][b, i, :m].tolist(), (kappa, b, i)
    idx.close()
