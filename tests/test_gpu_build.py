"""The pair-bitmap build at the edges of its tiles: row counts around its 2,048-row chunks and the
padding of its stored rows, column counts around its 16-column blocks and the pieces they are cut
into (few pieces, many pieces, one row chunk).  Every pair word of a small matrix, a sample of a
large one, and the pair counts, against the oracle's pair words (exact: bits and counts)."""

import numpy as np
import pytest

from oracle.bitmap import pair_words

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,C", [(2047, 15), (2048, 16), (2049, 17), (4097, 31), (4224, 33),
                                 (6145, 130), (8193, 48), (20001, 260), (130, 1024)])
def test_build_at_chunk_and_block_edges(R, C):
    from paper_2105_01196_gb300 import ebic
    g = np.random.default_rng(R + C)
    x = np.round(g.standard_normal((R, C)), 1).astype(np.float32)
    W, wst = (R + 31) // 32, (R + 127) // 128 * 4
    words, cnt = np.zeros(C * C * wst, np.uint32), np.zeros(C * C, np.uint64)
    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        ctx.build_bitmap()
        ctx.copy_bitmap(words)
        ctx.copy_pair_counts(cnt)
    words, cnt = words.reshape(C, C, wst), cnt.reshape(C, C)
    assert not words[:, :, W:].any() and not np.tril(cnt).any()
    assert not words[np.arange(C), np.arange(C)].any()
    pairs = [(a, b) for a in range(C) for b in range(a + 1, C)]
    if len(pairs) > 300:
        edges = [(a, b) for a, b in pairs if (b - a) in (1, 15, 16, 17) and (a + 1) % 16 < 3]
        pick = g.choice(len(pairs), 200, replace=False)
        pairs = edges[:100] + [pairs[k] for k in pick] + [(0, C - 1), (C - 2, C - 1)]
    popc = lambda w: int(np.unpackbits(w.view(np.uint8)).sum())
    for a, b in pairs:
        ab, ba = pair_words(x, a, b), pair_words(x, b, a)
        assert np.array_equal(words[a, b, :W], ab) and np.array_equal(words[b, a, :W], ba), (a, b)
        assert int(cnt[a, b]) == popc(ab) | (popc(ba) << 32), (a, b)


@pytest.mark.parametrize("C", [2, 31, 33, 65, 128, 129, 255, 257, 511, 513, 777, 1023, 1024])
@pytest.mark.parametrize("R", [1, 9, 130])
def test_rank_codes_order_every_pair(R, C):
    """The rank codes' sort at every lane width (1 to 32 keys per lane, full and partly filled) on
    rows that are sorted, reversed, constant, two-valued and random, with infinitely close and
    extreme values: every pair's counts equal the oracle's comparisons (a wrong code shows as a
    wrong pair)."""
    from paper_2105_01196_gb300 import ebic
    g = np.random.default_rng(17 * R + C)
    x = g.standard_normal((R, C)).astype(np.float32)
    kinds = [np.sort, lambda v: np.sort(v)[::-1], lambda v: v * 0 + 1,
             lambda v: np.where(v > 0, np.float32(1), np.float32(-1)), lambda v: v,
             lambda v: np.nextafter(np.float32(1), np.float32(2)) * (1 + (v > 0) * np.float32(1e-7)),
             lambda v: v * np.float32(1e37), lambda v: np.round(v * 3) * np.float32(1e-45)]
    for r in range(R):
        x[r] = kinds[r % len(kinds)](x[r]).astype(np.float32)
    x[:, g.random(C) < 0.1] = -0.0
    cnt = np.zeros(C * C, np.uint64)
    for layout in (ebic.ROW_MAJOR, ebic.COL_MAJOR):
        with ebic.Context(0) as ctx:
            ctx.load_matrix(x if layout == ebic.ROW_MAJOR else np.ascontiguousarray(x.T), layout)
            ctx.build_bitmap()
            ctx.copy_pair_counts(cnt)
        t = cnt.reshape(C, C)
        for a in g.choice(C, size=min(C, 60), replace=False):
            up, down = (x > x[:, a:a + 1]).sum(0), (x < x[:, a:a + 1]).sum(0)
            lo, hi = t[a] & np.uint64(0xFFFFFFFF), t[a] >> np.uint64(32)
            assert np.array_equal(lo[a + 1:], up[a + 1:]) and np.array_equal(hi[a + 1:], down[a + 1:])
