"""The window table of a pattern (b2sp_prepare_pattern), entry by entry against numpy, where its kernels branch: rows shorter
and longer than a warp's own share, few and many rows, column indices that begin on any 4-byte boundary, batches."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

EDGE_LENS = [0, 1, 2, 3, 7, 8, 9, 31, 255, 256, 257, 259, 511, 513, 2046, 2047, 2048, 2049, 2052, 2303, 2305, 2900]


@pytest.fixture(scope="module")
def b():
    assert torch.cuda.is_available()
    from paper_2311_00368_b200 import binding
    return binding


def make_rows(rng, lens, K):
    rp = np.zeros(len(lens) + 1, np.int32)
    rp[1:] = np.cumsum(lens)
    ci = np.concatenate([np.sort(rng.choice(K, n, replace=False)) for n in lens]).astype(np.int32)
    return rp, ci


def expected(rp, ci, K):
    M, Wk = len(rp) - 1, (K + 31) // 32
    mask = np.zeros((M, Wk), np.uint32)
    rows = np.repeat(np.arange(M), np.diff(rp))
    np.bitwise_or.at(mask, (rows, ci >> 5), np.uint32(1) << (ci & 31).astype(np.uint32))
    count = np.zeros((M, Wk), np.int64)
    np.add.at(count, (rows, ci >> 5), 1)
    return mask, rp[:-1, None] + np.cumsum(count, 1) - count


def table_of(b, ws, M, K, batch=1):
    off, Wk = b.debug_window_table_offset(M), (K + 31) // 32
    t = ws[off:off + 8 * batch * M * Wk].view(torch.int32).cpu().numpy().reshape(batch, M, Wk, 2)
    return t[..., 1].view(np.uint32), t[..., 0]


def flag_of(b, ws):
    off = b.debug_unsorted_flag_offset()
    return int(ws[off:off + 4].view(torch.int32).item())


def device(rp, ci, shift):
    """The arrays on the GPU, the column indices `shift` elements behind a 16-byte boundary, -1 around them."""
    buf = torch.full((ci.size + 16,), -1, dtype=torch.int32, device="cuda")
    view = buf[4 + shift:4 + shift + ci.size]
    view.copy_(torch.from_numpy(ci))
    return torch.from_numpy(rp).cuda(), view


@pytest.mark.parametrize("M,K,shift", [(44, 2999, 0), (44, 2999, 3), (2200, 2999, 0), (2200, 2999, 1), (2201, 3008, 2), (2500, 4096, 3)])
def test_table_entries(b, M, K, shift):
    rng = np.random.default_rng(M + K + shift)
    # (mostly short rows, so that the average keeps the kernel with a warp per row where M is large)
    lens = [EDGE_LENS[i % len(EDGE_LENS)] if i % 3 == 0 or M < 100 else int(rng.integers(0, 300)) for i in range(M)]
    rp, ci = make_rows(rng, lens, K)
    drp, dci = device(rp, ci, shift)
    ws = torch.zeros(1 << 25, dtype=torch.uint8, device="cuda")
    b.prepare_pattern(drp, dci, K, ws)
    mask, pos = table_of(b, ws, M, K)
    want_mask, want_pos = expected(rp, ci, K)
    assert flag_of(b, ws) == 0
    assert np.array_equal(mask[0], want_mask) and np.array_equal(pos[0], want_pos)


@pytest.mark.parametrize("M,K,length", [(2100, 2999, 2500), (2100, 2999, 2047), (2100, 2999, 2049), (2000, 4096, 2100), (1999, 4096, 2100)])
def test_table_entries_of_many_long_rows(b, M, K, length):
    """Either side of the average length and the number of rows at which four warps share a row."""
    rng = np.random.default_rng(M + length)
    rp, ci = make_rows(rng, [length + (i % 3) - 1 for i in range(M)], K)
    drp, dci = device(rp, ci, 3)
    ws = torch.zeros(1 << 25, dtype=torch.uint8, device="cuda")
    b.prepare_pattern(drp, dci, K, ws)
    mask, pos = table_of(b, ws, M, K)
    want_mask, want_pos = expected(rp, ci, K)
    assert flag_of(b, ws) == 0
    assert np.array_equal(mask[0], want_mask) and np.array_equal(pos[0], want_pos)


@pytest.mark.parametrize("M,K", [(2001, 65536), (2001, 65537), (2001, 98304), (2001, 98305)])
def test_table_entries_of_wide_patterns(b, M, K):
    """Either side of the widths at which eight rows' words no longer fit in a block's share of the shared memory."""
    rng = np.random.default_rng(K)
    lens = [int(rng.integers(0, 60)) if i % 50 else 2100 for i in range(M)]
    rp, ci = make_rows(rng, lens, K)
    drp, dci = device(rp, ci, 1)
    ws = torch.zeros(1 << 26, dtype=torch.uint8, device="cuda")
    b.prepare_pattern(drp, dci, K, ws)
    mask, pos = table_of(b, ws, M, K)
    want_mask, want_pos = expected(rp, ci, K)
    assert flag_of(b, ws) == 0
    assert np.array_equal(mask[0], want_mask) and np.array_equal(pos[0], want_pos)


@pytest.mark.parametrize("M", [44, 2200])
@pytest.mark.parametrize("row,entry", [(13, 5), (14, 2045), (17, 2048), (20, 2304), (21, 2899), (21, 2050), (9, 255),
                                       (17, "seam"), (20, "seam"), (21, "seam"), (21, "after the seam"), (20, "before the seam")])
def test_disorder_is_seen_wherever_it_is(b, M, row, entry):
    """Two entries of a row swapped, a repeated entry, a column out of range: each raises the flag.  The seam is the first entry of
    a row that its own warp leaves to the block: 2048 entries after the 16-byte boundary at or before the row."""
    rng = np.random.default_rng([row, len(str(entry))])
    K = 2999
    lens = EDGE_LENS * (M // len(EDGE_LENS)) if M < 100 else EDGE_LENS + [100] * (M - len(EDGE_LENS))
    rp, ci = make_rows(rng, lens, K)
    if isinstance(entry, str):
        begin = int(rp[row]) + 1   # (the arrays begin one element behind a boundary)
        entry = begin // 4 * 4 + 2048 - begin + {"seam": 0, "after the seam": 1, "before the seam": -1}[entry]
    p = int(rp[row]) + min(entry, lens[row] - 1)
    ws = torch.zeros(1 << 25, dtype=torch.uint8, device="cuda")
    for what in ("swap", "repeat", "below", "above"):
        bad = ci.copy()
        if what == "swap":
            bad[p], bad[p - 1] = ci[p - 1], ci[p]
        elif what == "repeat":
            bad[p] = ci[p - 1]
        else:
            bad[p] = -1 if what == "below" else K
        drp, dci = device(rp, bad, 1)
        b.prepare_pattern(drp, dci, K, ws)
        assert flag_of(b, ws) == 1, what
    drp, dci = device(rp, ci, 1)
    b.prepare_pattern(drp, dci, K, ws)
    assert flag_of(b, ws) == 0


@pytest.mark.parametrize("batch,M,K,long", [(3, 30, 700, 0), (7, 333, 257, 0), (5, 500, 4096, 3000), (3, 700, 2600, 2600)])
def test_batched_tables(b, batch, M, K, long):
    """Also with 2000 rows or more in all and some of them longer than a warp's own share, in every problem."""
    rng = np.random.default_rng(batch)
    probs = [make_rows(rng, [long - i % 7 if long and i % 60 == 7 else int(rng.integers(0, min(K, 256))) for i in range(M)], K)
             for _ in range(batch)]
    stride = max(ci.size for _, ci in probs) | 1   # odd: most problems begin off a 16-byte boundary
    # (the last problem's array ends with its last entry, and what lies behind it would break the order if it were read as its own)
    ci = np.full((batch - 1) * stride + probs[-1][1].size, -1, np.int32)
    for i, (_, c) in enumerate(probs):
        ci[i * stride:i * stride + c.size] = c
    rp = np.stack([r for r, _ in probs])
    ws = torch.zeros(1 << 25, dtype=torch.uint8, device="cuda")
    flat = torch.full((ci.size + 64,), -1, dtype=torch.int32, device="cuda")
    flat[:ci.size] = torch.from_numpy(ci)
    b.prepare_pattern_batched(torch.from_numpy(rp).cuda(), flat.as_strided((batch, 1), (stride, 1)), K, ws)
    mask, pos = table_of(b, ws, M, K, batch)
    assert flag_of(b, ws) == 0
    for i, (r, c) in enumerate(probs):
        want_mask, want_pos = expected(r, c, K)
        assert np.array_equal(mask[i], want_mask) and np.array_equal(pos[i], want_pos)


@pytest.mark.parametrize("M,length,long", [
    (5920, 640, 0),      # 740 blocks of eight rows: one wave with five blocks per SM
    (5921, 640, 2900),   # two waves with five, one with six: six
    (7104, 601, 2305),   # the last number of rows for which that holds; just above the length from which it counts
    (7105, 640, 0),      # two waves either way
    (6001, 600, 2900),   # rows not long enough
])
def test_table_entries_on_either_side_of_the_wave_rule(b, M, length, long):
    """A warp per row with five or six blocks on an SM (which differ in how the ends of rows are handled): the table, and a column
    out of order in the first and in the last chunk of a row."""
    K = 2999
    rng = np.random.default_rng(M + length)
    lens = [length + (i % 3) - 1 for i in range(M)]
    if long:   # a row that is finished by its whole block; the average stays
        lens[4000] += long - length
        for i in range(1000):
            lens[i] -= (long - length + 999 - i) // 1000
    assert sum(lens) // M == length or sum(lens) // M == length - 1
    rp, ci = make_rows(rng, lens, K)
    drp, dci = device(rp, ci, 2)
    ws = torch.zeros(1 << 25, dtype=torch.uint8, device="cuda")
    b.prepare_pattern(drp, dci, K, ws)
    mask, pos = table_of(b, ws, M, K)
    want_mask, want_pos = expected(rp, ci, K)
    assert flag_of(b, ws) == 0
    assert np.array_equal(mask[0], want_mask) and np.array_equal(pos[0], want_pos)
    for row, entry in ((4321, 1), (4321, int(lens[4321]) - 1), (M - 1, int(lens[M - 1]) - 1), (4000, int(lens[4000]) - 1)):
        bad, p = ci.copy(), int(rp[row]) + entry
        bad[p - 1], bad[p] = ci[p], ci[p - 1]
        drp, dci = device(rp, bad, 2)
        b.prepare_pattern(drp, dci, K, ws)
        assert flag_of(b, ws) == 1, (row, entry)
