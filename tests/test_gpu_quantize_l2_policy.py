"""The first look at inputs beyond L2 reads all but the last tiles with another cache policy: same codes as on either side of the
sizes where that starts and ends, ragged ends, rows off 32-byte boundaries and a subtrahend among them."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_1901_08924_b200 import lpc

pytestmark = pytest.mark.gpu
TILE = 8192


@pytest.mark.parametrize("b", [2, 8])
@pytest.mark.parametrize("sub", [False, True])
@pytest.mark.parametrize("tiles,extra,shift", [(768, 0, 0), (769, 5, 0), (1100, -3, 4), (1600, 0, 1)])
def test_scale_and_codes_around_the_kept_tail(b, sub, tiles, extra, shift):
    # two workers; with N * tiles around 1,536 tiles (48 MB, or 96 MB with the subtrahend) the policy starts
    N, length, seed, k = 2, tiles * TILE + extra, 7, 3
    g = torch.Generator(device="cuda").manual_seed(tiles + b)
    ld = (length + 3) // 4 * 4 + 8
    base, base2 = (torch.randn((N, ld), generator=g, device="cuda") for _ in range(2))
    U, S = base[:, shift:shift + length], base2[:, shift:shift + length]
    ctx = lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, b, lpc.CLIP_STD, 2.0, seed)
    codes, delta, clipped = ctx.quantize_pack(U, k, U_sub=S if sub else None)
    ctx.sync_status()
    V = (U - S if sub else U).cpu().numpy()
    words = codes.cpu().numpy().view(np.uint32)
    W = orc.packed_words(length, b)
    for i in range(N):
        w, dl, cl = orc.quantize_pack(np.ascontiguousarray(V[i]), b, orc.CLIP_STD, 2.0, seed, i, k)
        assert delta[i, 0].item() == dl and int(clipped[i, 0]) == cl
        assert (words[i, :W] == w).all()
    ctx.close()
