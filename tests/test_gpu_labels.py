"""Copy-mode labels (§3.2) on the GPU vs the oracle, through the C ABI.

Labels are integers: bit-exact.  Small rows (several structures, lengths, n) compare every position
with oracle.copy_labels; the full-size contexts of the zipf_32k workload compare sampled positions
with the oracle's single-window test (a position is labelled iff one of the n windows covering it
repeats) and check the runs-of-n invariant everywhere.
"""
import itertools

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _labels(ctx: np.ndarray, lens: np.ndarray, n: int) -> np.ndarray:
    import torch
    from paper_2609_20186_gb300 import binding as bd
    c = torch.from_numpy(np.ascontiguousarray(ctx, np.int32)).cuda()
    ln = torch.from_numpy(np.ascontiguousarray(lens, np.int32)).cuda()
    out = torch.full(c.shape, 7, dtype=torch.uint8, device="cuda")
    bd.switchsd_copy_labels(c, ln, out, n=n)
    return out.cpu().numpy()


def _rows(seed, B, cap):
    rng = np.random.default_rng(seed)
    ctx = np.zeros((B, cap), np.int32)
    lens = np.zeros(B, np.int32)
    for b in range(B):
        L = int(rng.integers(0, cap + 1))
        kind = b % 4
        if kind == 0:                      # small alphabet: many short repeats
            x = rng.integers(0, 3, L)
        elif kind == 1:                    # large alphabet with planted copies of earlier spans
            x = rng.integers(0, 100000, L)
            for _ in range(4):
                if L > 40:
                    ln = int(rng.integers(5, 30))
                    src = int(rng.integers(0, L - ln))
                    dst = int(rng.integers(src, L - ln + 1))
                    x[dst:dst + ln] = x[src:src + ln].copy()
        elif kind == 2:                    # a periodic run
            x = np.tile(rng.integers(0, 5, int(rng.integers(1, 7))), L // 1 + 1)[:L]
        else:                              # Zipf-like ids
            x = np.minimum(rng.zipf(1.3, L), 50000)
        ctx[b, :L] = x
        ctx[b, L:] = rng.integers(0, 3, cap - L)  # garbage past the length must not matter
        lens[b] = L
    return ctx, lens


@pytest.mark.parametrize("n", [5, 1, 3, 8, 32])
def test_small_rows_every_position(n):
    ctx, lens = _rows(10 + n, 24, 700)
    got = _labels(ctx, lens, n)
    for b in range(ctx.shape[0]):
        L = int(lens[b])
        ref = oracle.copy_labels(ctx[b, :L], n)
        assert np.array_equal(got[b, :L], ref), (b, L, n)
        assert not got[b, L:].any()


def test_bad_and_short_lengths():
    ctx, lens = _rows(3, 6, 64)
    lens[:] = [0, 3, 64, -1, 65, 5]
    got = _labels(ctx, lens, 5)
    assert not got[[0, 1, 3, 4]].any()                  # empty, shorter than n, out of range
    assert np.array_equal(got[2], oracle.copy_labels(ctx[2], 5))
    assert np.array_equal(got[5, :5], oracle.copy_labels(ctx[5, :5], 5))


def test_full_size_sampled_positions():
    wl = synth.WORKLOADS["zipf_32k"]
    ctx, lens = wl.contexts()
    got = _labels(ctx, lens, 5)
    rng = np.random.default_rng(0)
    for b in (0, 9, 33, 63):
        L = int(lens[b])
        x = ctx[b, :L]
        y = got[b, :L]
        runs = [len(list(g)) for k, g in itertools.groupby(y.tolist()) if k == 1]
        assert all(r >= 5 for r in runs)
        assert not got[b, L:].any()
        for j in rng.integers(0, L, 60):
            j = int(j)
            ref = any(oracle.window_repeats(x, 5, s) for s in range(max(0, j - 4), j + 1))
            assert bool(y[j]) == ref, (b, j)
        assert 0.02 < y.mean() < 0.98                   # the workload has both kinds of positions


@pytest.mark.parametrize("n", [1, 5])
def test_long_runs_and_short_periods(n):
    """Rows where thousands of windows are equal (one run, period 2, a 2-token alphabet: every insert
    lands on a few table slots) beside ordinary rows in one batch; every position against the oracle."""
    rng = np.random.default_rng(77 + n)
    B, cap = 6, 12000
    ctx = np.zeros((B, cap), np.int32)
    ctx[0] = 7                                          # one run: every window equal
    ctx[1] = np.tile([3, 9], cap // 2)                  # period 2
    ctx[2] = rng.integers(0, 2, cap)                    # two-letter alphabet: few distinct windows
    ctx[3] = rng.integers(0, 100000, cap)               # distinct windows
    ctx[4, :6000] = 5                                   # half a run, then distinct tokens
    ctx[4, 6000:] = rng.integers(0, 100000, cap - 6000)
    ctx[5] = np.minimum(rng.zipf(1.3, cap), 50000)      # Zipf ids
    lens = np.array([cap, cap - 1, cap, cap, cap - 3, 9001], np.int32)
    got = _labels(ctx, lens, n)
    for b in range(B):
        L = int(lens[b])
        assert np.array_equal(got[b, :L], oracle.copy_labels(ctx[b, :L], n)), b
        assert not got[b, L:].any()


def _first_occurrence_labels(x: np.ndarray, n: int) -> np.ndarray:
    """Every position of one row from a dictionary of the windows' first starts (the oracle's definition, in
    time linear in the row)."""
    y = np.zeros(len(x), np.uint8)
    seen = {}
    raw = np.ascontiguousarray(x, np.int32).tobytes()
    for s in range(len(x) - n + 1):
        if seen.setdefault(raw[4 * s:4 * (s + n)], s) < s:
            y[s:s + n] = 1
    return y


# (rows, capacity, n): one and several CTAs a row, tables of every size class, capacities that are no multiple
# of 16, both sides of the lines between the one-kernel form and the two kernels (8,192 tokens for any number of
# rows; then 4 or 22 rows up to 16,384 and 24 up to 32,768, by n; then the share of the grid's waves that is filled,
# up to 65,536), and rows past them
@pytest.mark.parametrize("B,cap,n", [(200, 3001, 5), (3, 513, 32), (40, 8209, 2), (1, 4097, 5), (1, 16384, 5),
                                     (12, 16385, 5), (13, 16385, 5), (23, 32768, 5), (24, 32768, 8), (2, 32769, 5), (70, 16389, 3),
                                     (31, 65536, 5), (32, 65536, 5), (40, 65521, 8), (33, 65537, 5),
                                     (1, 131075, 5), (2, 262144, 7), (1, 262145, 5),
                                     (1, 8192, 5), (21, 8193, 8), (22, 8193, 8), (3, 12289, 8), (4, 12289, 8), (21, 16383, 9), (22, 16383, 9), (24, 20001, 5),
                                     (28, 32768, 9), (29, 32768, 32), (28, 40004, 5), (57, 40004, 5), (66, 33001, 12), (67, 33001, 12)])
def test_size_classes(B, cap, n):
    rng = np.random.default_rng(cap)
    ctx = np.zeros((B, cap), np.int32)
    for b in range(B):
        kind = b % 3
        if kind == 0:                                   # ids that differ in their high bits alone, copies
            ctx[b] = rng.integers(-128, 128, cap) << 24
        elif kind == 1:
            ctx[b] = np.minimum(rng.zipf(1.2, cap), 120000)
        else:
            ctx[b] = np.tile(rng.integers(0, 9, 5), cap // 5 + 1)[:cap]
        if cap > 2000:
            ctx[b, cap - 900:] = ctx[b, 100:1000]
    lens = rng.integers(max(1, cap - 40), cap + 1, B).astype(np.int32)
    assert np.array_equal(_first_occurrence_labels(ctx[0, :400], n), oracle.copy_labels(ctx[0, :400], n))
    got = _labels(ctx, lens, n)
    for b in list(range(min(B, 6))) + [B - 1]:
        L = int(lens[b])
        assert np.array_equal(got[b, :L], _first_occurrence_labels(ctx[b, :L], n)), b
        assert not got[b, L:].any()


def _label_part(ids: np.ndarray, parts: int) -> np.ndarray:
    """The part of a row's cluster that takes the window of one token (label_mix of csrc/labels.cu, n = 1)."""
    with np.errstate(over="ignore"):
        h = ids.astype(np.uint32)
        h = (h ^ (h >> np.uint32(15))) * np.uint32(0x2C1B3C6D)
        h = (h ^ (h >> np.uint32(12))) * np.uint32(0x297A2D39)
        h ^= h >> np.uint32(15)
    return ((h.astype(np.uint64) * np.uint64(parts)) >> np.uint64(32)).astype(np.int64)


def test_full_table():
    """More distinct windows in one part of the hash than its table has slots: those that find the table full
    compare with every earlier window, and repeats of them, and of the ones in the table, are still marked."""
    import torch
    from paper_2609_20186_gb300 import binding as bd
    from tests import lockstep
    B, cap, n = 24, 32768, 1
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    parts = 1
    while parts < 8 and 2 * parts * (B + 5) <= sms and cap // (2 * parts) >= 512:
        parts *= 2
    slots = 2 * (cap // parts) + 64
    rng = np.random.default_rng(3)
    ids = rng.permutation(1 << 20)[:parts * (slots + 4000) * 2].astype(np.int32)
    mine = ids[_label_part(ids, parts) == parts - 1]
    full = mine[:slots + 700]
    rest = np.setdiff1d(ids, mine)
    assert parts > 1 and len(full) == slots + 700
    ctx = np.zeros((B, cap), np.int32)
    for b, order in ((0, 1), (5, -1)):
        again = np.concatenate([full[:300], full[-600:]])  # some of the table's and some of the others
        x = np.concatenate([full[::order], rest[:2000], rng.permutation(again), rest[:50]])
        ctx[b, :len(x)] = x
        ctx[b, len(x):] = rest[2000:2000 + cap - len(x)]
    lens = np.full(B, 7, np.int32)
    lens[[0, 5]] = cap

    def call(stream):
        bd.switchsd_copy_labels(c, ln, out, n=n, workspace=ws, stream=stream)
    c, ln = torch.from_numpy(ctx).cuda(), torch.from_numpy(lens).cuda()
    out = torch.zeros(c.shape, dtype=torch.uint8, device="cuda")
    ws = torch.empty(int(bd.load().switchsd_labels_workspace_bytes(B, cap)), dtype=torch.uint8, device="cuda")
    assert any("label_cluster_kernel" in k for k in lockstep.kernel_names(call))
    got = _labels(ctx, lens, n)
    for b in (0, 5):
        want = _first_occurrence_labels(ctx[b], n)
        assert want.sum() >= 900 and np.array_equal(got[b], want), b
