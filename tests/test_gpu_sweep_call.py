"""One population evaluation through every way its arrays can reach it: host arrays below and above
the size that goes through the context's pinned block, device arrays, outputs partly wanted and on
either side; a bad population leaves every output as it was, and the next call is right.  Counts
and fitness equal the oracle's (sampled for the large population)."""

import numpy as np
import pytest

from oracle import counts as ocounts
from oracle.params import Params as OParams

pytestmark = pytest.mark.gpu
FILL = -7


def _population(g, n, C, hi):
    lens = g.integers(2, hi + 1, size=n)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    return np.concatenate([g.choice(C, size=L, replace=False) for L in lens]).astype(np.int32), off


@pytest.mark.parametrize("n", [1, 7, 257, 13_107, 13_108, 20_000])
@pytest.mark.parametrize("mode", [0, 1, 2, 4])
def test_every_way_in_and_out(n, mode):
    import torch
    from paper_2105_01196_gb300 import ebic
    g = np.random.default_rng(n + mode)
    R, C = 300, 40
    x = g.integers(-3, 4, size=(R, C)).astype(np.float32)
    ci, off = _population(g, n, C, 12)
    p = ebic.Params.make(neg_trends=1, ratio_num=85, ratio_den=100, mode=mode, min_rows=0)
    op = OParams(neg_trends=1, ratio_num=85, ratio_den=100, min_rows=0, col_cap=p.col_cap)
    pick = sorted({0, n - 1} | set(g.integers(0, n, size=40).tolist()))
    want = {i: ocounts.eval_individual(x, [int(c) for c in ci[off[i]:off[i + 1]]], op)
            for i in pick}

    def check(outs, used):
        for k, o in enumerate(outs):
            o = np.asarray(o.cpu() if torch.is_tensor(o) else o).astype(np.int64)
            for i in pick:
                assert o[i] == (want[i][k] if used[k] else FILL), (k, i)

    kinds = [(torch.int32, np.int32)] * 3 + [(torch.int64, np.uint64)]
    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        for dev_in in (0, 1):
            a, o = (torch.from_numpy(ci).cuda(), torch.from_numpy(off).cuda()) if dev_in else (ci, off)
            for dev_out, used in ((0, (1, 1, 1, 1)), (1, (1, 1, 1, 1)), (0, (0, 1, 0, 1)), (1, (1, 0, 1, 0))):
                outs = [torch.full((n,), FILL, dtype=t, device="cuda") if dev_out
                        else np.full(n, FILL, np.int64).astype(d) for t, d in kinds]
                got = [x_ if u else None for x_, u in zip(outs, used)]
                ctx.eval_population(a, o, p, *got)
                if not dev_out:
                    outs = [y.view(np.int64) if y.dtype == np.uint64 else y for y in outs]
                check(outs, used)
                # a repeated column in the last individual: refused, nothing written
                bad = ci.copy()
                bad[off[n - 1] + 1] = bad[off[n - 1]]
                outs = [torch.full((n,), FILL, dtype=t, device="cuda") for t, _ in kinds]
                with pytest.raises(ebic.EbicError) as e:
                    ctx.eval_population(torch.from_numpy(bad).cuda() if dev_in else bad, o, p, *outs)
                assert e.value.code == ebic.EBIC_EINVAL
                check(outs, (0, 0, 0, 0))


def test_contexts_in_turn_share_nothing():
    """Contexts opened and closed in turn and side by side reuse each other's pinned blocks; each
    one's results are its own matrix's."""
    from paper_2105_01196_gb300 import ebic
    g = np.random.default_rng(3)
    p = ebic.Params.make(neg_trends=1, ratio_num=1, ratio_den=1, min_rows=0)
    op = OParams(neg_trends=1, ratio_num=1, ratio_den=1, min_rows=0, col_cap=p.col_cap)
    jobs = []
    for k in range(12):
        x = g.standard_normal((50 + 13 * k, 9)).astype(np.float32)
        ci, off = _population(g, 20 + k, 9, 5)
        jobs.append((x, ci, off, ocounts.eval_population(x, ci, off, op)))
    for width in (1, 12):
        for at in range(0, 12, width):
            ctxs = [ebic.Context(0) for _ in range(width)]
            for ctx, (x, _, _, _) in zip(ctxs, jobs[at:]):
                ctx.load_matrix(x)
            for ctx, (_, ci, off, want) in zip(ctxs, jobs[at:]):
                for a, b in zip(ctx.eval_population(ci, off, p), want):
                    assert np.array_equal(np.asarray(a, np.int64), np.asarray(b, np.int64))
            for ctx in ctxs:
                ctx.close()
