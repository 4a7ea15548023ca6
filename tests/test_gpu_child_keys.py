"""Children's column keys and their random words: columns on both sides of a byte's range up to the
widest matrix, populations of both evolve forms, tournaments of one to five candidates, and
chromosomes that take more words than a warp holds at a time (most draws of a full chromosome's
last columns repeat one it has).  Equal to the oracle, keys included."""

import numpy as np
import pytest

from oracle import ebic as oebic
from oracle.params import Params as OParams

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,pop,init,T", [
    (255, 60, (2, 8), 4), (256, 1400, (2, 6), 3), (257, 60, (2, 8), 1), (65535, 50, (2, 8), 4),
    (64, 40, (60, 64), 4), (64, 1300, (62, 64), 2), (40, 60, (38, 40), 5)])
def test_child_keys_and_words(C, pop, init, T):
    from paper_2105_01196_gb300 import ebic
    g = np.random.default_rng(C + pop)
    x = g.standard_normal((40, C)).astype(np.float32)
    base = dict(neg_trends=1, ratio_num=85, ratio_den=100, max_len=init[1], init_min_len=init[0],
                init_max_len=init[1], pop_size=pop, elite=4, n_biclusters=6, tournament=T,
                tabu_hit_limit=0, seed=C)
    st = oebic.run(x, OParams(**base), 3)
    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        rep = ctx.run_generations(ebic.Params.make(**base), 3)
        assert (rep.gens_done, rep.last_hits) == (st.gen, st.hits[-1])
        assert [(e["cols"], e["f"], e["h"]) for e in ctx.toplist()] == \
            [(tuple(e.cols), e.f, e.h) for e in st.top]
        cols, lens, _, fit = ctx.population(pop)
        assert [list(c[:n]) for c, n in zip(cols, lens)] == [list(c) for c in st.pop]
        assert fit.tolist() == [int(f) for f in st.fit]
