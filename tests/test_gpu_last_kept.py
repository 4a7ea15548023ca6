"""Last-kept counts over 16-bit rank codes (the reference of a direction as a packed maximum or
minimum): from the narrowest matrix of that width to the widest, largest codes included, with
distinct values, many ties and rows of one value.  Equal to the oracle."""

import numpy as np
import pytest

from oracle import counts as ocounts
from oracle.params import Params as OParams
from paper_2105_01196_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [129, 257, 1000, 1024])
@pytest.mark.parametrize("neg,ns", [(1, 0), (1, 1), (0, 0), (0, 1)])
def test_last_kept_wide_codes(C, neg, ns):
    from paper_2105_01196_gb300 import ebic
    g = np.random.default_rng(C)
    x = g.standard_normal((300, C)).astype(np.float32)
    x[100:200] = np.round(x[100:200])
    x[200:210] = 1.5
    x[210] = np.arange(C)
    x[211] = -np.arange(C)
    ci, off = synth.random_population(60, C, 2, 64, C)
    kw = dict(neg_trends=neg, ratio_num=85, ratio_den=100, non_strict=ns, last_kept=1)
    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        got = ctx.eval_population(ci, off, ebic.Params.make(mode=1, **kw))
    p = ebic.Params.make(**kw)
    want = ocounts.eval_population(x, ci, off, OParams(min_rows=p.min_rows, col_cap=p.col_cap,
                                                       **kw))
    for a, b in zip(got, want):
        assert [int(v) for v in a] == [int(v) for v in b]
