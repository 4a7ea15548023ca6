"""Searches whose evolve launch evaluates every child, with more attempt warps than twelve per SM, where a
block takes several steps over a pair row: four steps of four words per thread (exact) and up to
eight of two (counting), the last one whole, partly filled or of one word; and the same searches
at a ratio that keeps the evaluation launch.  Equal to the oracle."""

import numpy as np
import pytest

from oracle import ebic as oebic
from oracle.params import Params as OParams

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,A,pop,ratio,ns", [
    (33_000, 4, 460, (85, 100), 0), (65_536, 4, 460, (9, 10), 1), (40_100, 4, 460, (1, 1), 0),
    (16_384, 1, 1900, (85, 100), 0), (14_400, 2, 920, (1, 1), 1), (33_000, 4, 460, (4, 5), 0)])
def test_steps_over_a_pair_row(R, A, pop, ratio, ns):
    from paper_2105_01196_gb300 import ebic
    g = np.random.default_rng(R)
    x = g.standard_normal((R, 24)).astype(np.float32)
    x[:, 5] = np.round(x[:, 5])
    x[:, 9] = np.round(x[:, 9])
    base = dict(neg_trends=1, ratio_num=ratio[0], ratio_den=ratio[1], non_strict=ns, max_len=12,
                init_min_len=2, init_max_len=12, pop_size=pop, elite=5, n_biclusters=5,
                max_attempts=A, tabu_hit_limit=0, seed=R)
    st = oebic.run(x, OParams(**base), 2)
    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        p = ebic.Params.make(mode=2, **base)
        ctx.run_generations(p, 0)
        before = ctx.profile_read(ebic.KERNEL_EVAL)["launches"]
        rep = ctx.run_generations(p, 2)
        made = ctx.profile_read(ebic.KERNEL_EVAL)["launches"] - before
        assert made == (2 if ratio == (4, 5) else 0)
        assert (rep.gens_done, rep.last_hits, rep.n_evaluated) == (st.gen, st.hits[-1], st.n_evaluated)
        assert [(e["cols"], e["f"], e["rows_pos"], e["rows_neg"]) for e in ctx.toplist()] == \
            [(tuple(e.cols), e.f, e.rows_pos, e.rows_neg) for e in st.top]
        cols, lens, _, fit = ctx.population(pop)
    assert [list(c[:n]) for c, n in zip(cols, lens)] == [list(c) for c in st.pop]
    assert fit.tolist() == [int(f) for f in st.fit]
