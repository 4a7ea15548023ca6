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
