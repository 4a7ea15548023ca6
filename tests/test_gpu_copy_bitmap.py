"""The pair words given out where the stored rows are padded: to the device (on a 16-byte boundary and
off it) and to the host, by every way the library has (small bitmaps packed whole, short rows in
pieces through two halves, up to three turns of them, longer rows by strided copies).  Words of every
pair row against the same matrix's comparison, rows past the matrix zero, and nothing written
beside them."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,C", [(4225, 20), (4225, 260), (4225, 610), (8200, 150), (10_000, 40),
                                 (33_333, 70), (4096, 50)])
def test_rows_without_their_padding(R, C):
    import torch
    from paper_2105_01196_gb300 import ebic
    g = torch.Generator(device="cuda").manual_seed(R + C)
    x = torch.randint(0, 50, (R, C), generator=g, device="cuda").float()
    wst = (R + 127) // 128 * 4
    n = C * C * wst
    # the words, column by column: bit j of word w of (a, b) = x[32 w + j, b] > x[32 w + j, a]
    pad = torch.full((wst * 32, C), 0.0, device="cuda")
    pad[:R] = x
    weight = (1 << torch.arange(32, dtype=torch.int64, device="cuda"))[None, :, None]
    want = torch.stack([((pad > pad[:, a:a + 1]).view(wst, 32, C) * weight).sum(1).t()
                        for a in range(C)]).to(torch.int32).view(-1)
    with ebic.Context(0) as ctx:
        ctx.load_matrix(x)
        ctx.build_bitmap()
        for shift in (0, 1, 2):
            out = torch.full((n + 8,), 7, dtype=torch.int32, device="cuda")
            ctx.copy_bitmap(out[shift:shift + n])
            assert torch.equal(out[shift:shift + n], want)
            assert (out[:shift] == 7).all() and (out[shift + n:] == 7).all()
        host = np.full(n + 4, 7, np.uint32)
        for _ in range(2):
            ctx.copy_bitmap(host[:n])
            assert np.array_equal(host[:n], want.cpu().numpy().view(np.uint32))
            assert (host[n:] == 7).all()
        ctx.load_matrix(x.cpu().numpy())              # (the staging buffer is the loads' again)
        ctx.build_bitmap()
        ctx.copy_bitmap(host[:n])
        assert np.array_equal(host[:n], want.cpu().numpy().view(np.uint32))
