"""Evaluations that read one direction's pair words where no pair of the individual has ties: a
bitmap larger than L2 over distinct values with a few tied column pairs, so that tie-free and tied
individuals meet in one launch.  Chromosome lengths around the eight-row units, exact tests (one
pair from the counts, packed passes, more rows than a unit) and counting ones, ties counting both
ways or not, row counts inside and at the end of a pass; and the generation loop over the same
matrix, children evaluated inside the evolve kernel included.  Equal to the oracle."""

import numpy as np
import pytest

from oracle import counts as ocounts
from oracle import ebic as oebic
from oracle.params import Params as OParams

pytestmark = pytest.mark.gpu


def _matrix(R, C, seed):
    """Distinct values in every row but for 12 columns that repeat the column before them in some
    rows (from one row to all of them)."""
    g = np.random.default_rng(seed)
    x = np.argsort(g.random((R, C)), axis=1).astype(np.float32)
    tied = []
    for k, c in enumerate(range(5, C, C // 12)):
        rows = np.array([R - 1]) if k == 0 else g.choice(R, size=max(1, R * k // 12), replace=False)
        x[rows, c] = x[rows, c - 1]
        tied.append(c)
    return x, tied


@pytest.mark.parametrize("R,C", [(4500, 650), (4096, 700), (8193, 420)])
def test_one_direction_sweep(R, C):
    from paper_2105_01196_gb300 import ebic
    x, tied = _matrix(R, C, R)
    assert C * C * R / 8 > 180e6                       # (larger than L2: the staged forms)
    g = np.random.default_rng(C)
    pop = []
    for L in (2, 3, 4, 5, 6, 7, 8, 9, 10, 16, 17, 18, 25, 33, 34, 64):
        for k in range(3):
            c = g.choice(C, size=L, replace=False)
            if k == 0:                                 # a tied pair somewhere
                t = tied[int(g.integers(len(tied)))]
                c = np.array([v for v in c if v not in (t, t - 1)])[:L - 2]
                at = int(g.integers(0, len(c) + 1))
                c = np.concatenate([c[:at], [t - 1, t], c[at:]])
            pop.append(c)
    off = np.concatenate([[0], np.cumsum([len(c) for c in pop])]).astype(np.int32)
    ci = np.concatenate(pop).astype(np.int32)
    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        for ns in (0, 1):
            for num, den in ((85, 100), (99, 100), (1, 2), (1, 64)):
                p = ebic.Params.make(neg_trends=1, ratio_num=num, ratio_den=den, mode=2,
                                     non_strict=ns, min_rows=0)
                op = OParams(neg_trends=1, ratio_num=num, ratio_den=den, min_rows=0,
                             col_cap=p.col_cap, non_strict=ns)
                want = ocounts.eval_population(x, ci, off, op)
                for got, w in zip(ctx.eval_population(ci, off, p), want):
                    assert np.array_equal(np.asarray(got, np.int64), np.asarray(w, np.int64))


@pytest.mark.parametrize("pop,fuse", [(300, 0), (300, 63), (1400, 0), (1400, 2), (1400, -1)])
@pytest.mark.parametrize("ns", [0, 1])
def test_one_direction_loop(pop, fuse, ns):
    from paper_2105_01196_gb300 import ebic
    R, C = 700, 1000
    x, _ = _matrix(R, C, 5)
    base = dict(neg_trends=1, ratio_num=85, ratio_den=100, max_len=12, init_min_len=2,
                init_max_len=12, pop_size=pop, elite=6, n_biclusters=6, tabu_hit_limit=0, seed=4,
                non_strict=ns)
    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        rep = ctx.run_generations(ebic.Params.make(mode=2, fuse_pairs=fuse, **base), 3)
        top = [(e["cols"], e["f"]) for e in ctx.toplist()]
        cols, lens, _, fit = ctx.population(pop)
    st = oebic.run(x, OParams(**base), 3)
    assert rep.n_evaluated == st.n_evaluated
    assert top == [(tuple(e.cols), e.f) for e in st.top]
    assert [list(c[:n]) for c, n in zip(cols, lens)] == [list(c) for c in st.pop]
    assert fit.tolist() == [int(f) for f in st.fit]
