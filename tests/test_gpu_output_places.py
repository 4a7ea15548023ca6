"""Device outputs of an evaluation anywhere in a caller's arena: off their boundaries, over one another
(the later one of positive, negative, either, fitness stays) and over the population's own offsets.
The reference is the same call with host outputs (compared with the oracle elsewhere)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("at", [(0, 12_000, 24_000, 40_004), (2, 12_001, 24_003, 40_006),
                                (0, 0, 24_000, 40_000), (0, 12_000, 24_000, 26_000),
                                (80_000, 12_000, 24_000, 40_000), (84_000, 12_000, 24_000, 76_004)])
def test_outputs_anywhere(at):
    import torch
    from paper_2105_01196_gb300 import ebic
    n, C = 2500, 30
    g = np.random.default_rng(7)
    x = g.standard_normal((700, C)).astype(np.float32)
    lens = g.integers(2, 7, size=n)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    ci = np.concatenate([g.choice(C, size=L, replace=False) for L in lens]).astype(np.int32)
    p = ebic.Params.make(neg_trends=1, ratio_num=3, ratio_den=4, mode=1, min_rows=0)
    arena = torch.zeros(100_000, dtype=torch.uint8, device="cuda")
    d_off = arena[80_000:80_000 + 4 * (n + 1)].view(torch.int32)
    d_off.copy_(torch.from_numpy(off))
    d_ci = torch.from_numpy(ci).cuda()
    torch.cuda.synchronize()
    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        want = ctx.eval_population(ci, off, p)
        image = arena.cpu().numpy()
        for o, w in zip(at, want):
            image[o:o + w.nbytes] = w.view(np.uint8)
        ctx.eval_population(d_ci, d_off, p, *[arena[o:] for o in at])
        assert np.array_equal(arena.cpu().numpy(), image)
