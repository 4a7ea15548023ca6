"""The generation loop whose evolve launch evaluates every child itself (block-per-slot form, bitmap):
row counts around the steps of a block's threads over a pair row (a step of four words per thread,
the last one partly filled; one row past what the form takes), one to four attempts, exact and
counting tests, both directions and one, ties counting both ways, a tabu stop, graph and eager
replays, and a checkpoint between its generations.  Equal to the oracle."""

import numpy as np
import pytest

from oracle import ebic as oebic
from oracle.params import Params as OParams

pytestmark = pytest.mark.gpu


def _check(ctx, rep, st, pop):
    assert (rep.gens_done, rep.last_hits) == (st.gen, st.hits[-1])
    # (a generation that the tabu-hit limit discards has been evaluated)
    assert rep.n_evaluated == st.n_evaluated or rep.stopped
    assert [(e["cols"], e["f"]) for e in ctx.toplist()] == [(tuple(e.cols), e.f) for e in st.top]
    cols, lens, _, fit = ctx.population(pop)
    assert [list(c[:n]) for c, n in zip(cols, lens)] == [list(c) for c in st.pop]
    assert fit.tolist() == [int(f) for f in st.fit]


@pytest.mark.parametrize("R,A,neg,ns,ratio,max_len", [
    (30, 1, 1, 0, (85, 100), 8), (2000, 1, 1, 1, (1, 2), 20), (16384, 4, 1, 0, (85, 100), 20),
    (16500, 4, 0, 0, (3, 4), 30), (9000, 2, 1, 1, (85, 100), 12), (9000, 3, 0, 1, (1, 1), 30),
    (16384, 1, 1, 0, (85, 100), 10), (16400, 1, 1, 0, (85, 100), 10)])
def test_block_evaluation(R, A, neg, ns, ratio, max_len):
    from paper_2105_01196_gb300 import ebic
    g = np.random.default_rng(R + A)
    x = np.round(g.standard_normal((R, 30)), 1).astype(np.float32)
    pop = 70
    base = dict(neg_trends=neg, ratio_num=ratio[0], ratio_den=ratio[1], non_strict=ns,
                max_len=max_len, init_min_len=2, init_max_len=max_len, pop_size=pop, elite=5,
                n_biclusters=5, max_attempts=A, tabu_hit_limit=0, seed=R)
    st = oebic.run(x, OParams(**base), 3)
    for graph in (1, 0):
        with ebic.Context(0) as ctx:
            ctx.load_matrix(x)
            rep = ctx.run_generations(ebic.Params.make(mode=2, use_graph=graph, **base), 3)
            _check(ctx, rep, st, pop)


def test_many_generations_checkpoint_and_stop():
    """Forty generations (chunks of sixteen and singles), split by a checkpoint into a new context
    and by a call with kernel statistics on (its evaluations in their own launch), and a run that
    the tabu-hit limit ends."""
    from paper_2105_01196_gb300 import ebic
    g = np.random.default_rng(8)
    x = np.round(g.standard_normal((600, 12)), 1).astype(np.float32)
    base = dict(neg_trends=1, ratio_num=85, ratio_den=100, max_len=9, init_min_len=2,
                init_max_len=9, pop_size=90, elite=4, n_biclusters=6, tabu_hit_limit=0, seed=3)
    p = ebic.Params.make(mode=2, **base)
    st = oebic.run(x, OParams(**base), 40)
    with ebic.Context(0) as ctx, ebic.Context(0) as other:
        ctx.load_matrix(x)
        ctx.run_generations(p, 17)
        ctx.profile_enable(True)
        ctx.run_generations(p, 2)
        ctx.profile_enable(False)
        blob = ctx.save_state()
        other.load_matrix(x)
        other.load_state(p, blob)
        for c in (ctx, other):
            _check(c, c.run_generations(p, 21), st, 90)
    base["tabu_hit_limit"] = 30
    st = oebic.run(x, OParams(**base), 40)
    assert st.stopped
    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        rep = ctx.run_generations(ebic.Params.make(mode=2, **base), 40)
        assert rep.stopped
        _check(ctx, rep, st, 90)
