"""The generation loop's evaluation launch over a bitmap larger than L2 with hardly any ties, so that
it reads one direction's pair words: the launch over every slot (fuse_pairs -1) and over the list
of slots that the evolve kernel left to it (fuse_pairs 2), with its duplicate table and the side
task of the tabu list, one block per slot and one warp per slot, ties counting both ways or not.
Generation by generation, then sixteen in one graph replay, against the oracle."""

import numpy as np
import pytest

from oracle import ebic as oebic
from oracle.params import Params as OParams

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pop", [96, 1400])
@pytest.mark.parametrize("fuse", [-1, 2])
@pytest.mark.parametrize("ns", [0, 1])
def test_loop_reads_one_direction(pop, fuse, ns):
    from paper_2105_01196_gb300 import ebic
    R, C = 4500, 650
    g = np.random.default_rng(31 + ns)
    x = np.argsort(g.random((R, C)), axis=1).astype(np.float32)
    for k, c in enumerate(range(5, C, 60)):           # a few pairs tied, in one to most rows
        x[g.choice(R, size=1 + R * k // 12, replace=False), c] = -1.0
        x[:, c - 1] = np.where(x[:, c] < 0, -1.0, x[:, c - 1])
    assert C * C * R / 8 > 180e6
    num, den = (1, 2) if fuse < 0 else (85, 100)
    base = dict(neg_trends=1, ratio_num=num, ratio_den=den, max_len=20, init_min_len=2,
                init_max_len=20, pop_size=pop, elite=6, n_biclusters=6, tabu_hit_limit=0, seed=23,
                non_strict=ns)
    op = OParams(**base)
    p = ebic.Params.make(mode=2, fuse_pairs=fuse, **base)

    def check(ctx, rep, st):
        assert (rep.gens_done, rep.n_evaluated, rep.last_hits) == (st.gen, st.n_evaluated, st.hits[-1])
        assert [(e["cols"], e["f"], e["rows_pos"], e["rows_neg"], e["rows_any"])
                for e in ctx.toplist()] == \
            [(tuple(e.cols), e.f, e.rows_pos, e.rows_neg, e.rows_any) for e in st.top]
        cols, lens, dead, fit = ctx.population(pop)
        assert [list(c[:n]) for c, n in zip(cols, lens)] == [list(c) for c in st.pop]
        assert dead.astype(bool).tolist() == st.dead
        assert fit.tolist() == [int(f) for f in st.fit]

    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        rep = ctx.run_generations(p, 0)
        st = oebic.initialise(x, op)
        check(ctx, rep, st)
        for _ in range(3):
            rep = ctx.run_generations(p, 1)
            assert oebic.next_generation(x, st, op)
            check(ctx, rep, st)
        if pop == 96:
            rep = ctx.run_generations(p, 16)
            for _ in range(16):
                assert oebic.next_generation(x, st, op)
            check(ctx, rep, st)
        assert (rep.n_fused > 0) == (fuse > 0)
