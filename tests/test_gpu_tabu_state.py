"""The tabu list of a run that the tabu-hit limit ended, as its checkpoint holds it: every key of the
generations that were scored and none of the discarded one's, counted once each, whether the loop
evaluates in the evolve launch (its side task then runs beside the scoring that ends the run), in
an evaluation launch, or without the bitmap; equal to the oracle's, graph replays and single
launches alike.  1,100 slots spread the side task over several blocks."""

import struct

import numpy as np
import pytest

from oracle import ebic as oebic
from oracle.params import Params as OParams

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pop,max_len,limit", [(90, 9, 82), (1100, 4, 2240)])
@pytest.mark.parametrize("mode,fuse,graph", [(2, 0, 1), (2, 0, 0), (2, -1, 1), (1, 0, 1)])
def test_stopped_run_keeps_every_tabu_key(pop, max_len, limit, mode, fuse, graph):
    from paper_2105_01196_gb300 import ebic
    g = np.random.default_rng(8)
    x = np.round(g.standard_normal((600, 12)), 1).astype(np.float32)
    base = dict(neg_trends=1, ratio_num=85, ratio_den=100, max_len=max_len, init_min_len=2,
                init_max_len=max_len, pop_size=pop, elite=4, n_biclusters=6, tabu_hit_limit=limit,
                seed=3)
    st = oebic.run(x, OParams(**base), 40)
    assert st.stopped and st.gen > 4
    want = sorted(st.tabu)
    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        rep = ctx.run_generations(ebic.Params.make(mode=mode, fuse_pairs=fuse, use_graph=graph, **base),
                                  40)
        assert (rep.stopped, rep.gens_done) == (1, st.gen)
        blob = ctx.save_state()
    n = struct.unpack_from("<q", blob, 32)[0]          # (the header's key count)
    assert n == len(want)
    assert blob[-8 * n:].view(np.uint64).tolist() == want
