"""The first look at inputs beyond L2 reads all but the last tiles with another cache policy: same codes as the oracle's on either side of
the sizes where that starts and ends, ragged ends, several tensors, rows off 32-byte boundaries and a subtrahend among them, and the
library says that the side the case is about has run."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_1901_08924_b200 import lpc

pytestmark = pytest.mark.gpu
TILE = 8192
L2 = torch.cuda.get_device_properties(0).L2_cache_size if torch.cuda.is_available() else 132644864
KEPT, FROM = L2 // 8 * 3 // (4 * TILE), L2 // 8 * 5 // (4 * TILE)  # tiles
N = 2


def _vectors(length, ld, shift, sub, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    base = [torch.randn((N, ld), generator=g, device="cuda") for _ in range(2 if sub else 1)]
    U = [v[:, shift:shift + length] for v in base]
    return U[0], U[1] if sub else None


@pytest.mark.parametrize("b", [2, 8])
@pytest.mark.parametrize("sub", [False, True])
@pytest.mark.parametrize("tiles,extra,shift", [(768, 0, 0), (769, 5, 0), (1100, -3, 4), (1600, 0, 1)])
def test_scale_and_codes_around_the_kept_tail(b, sub, tiles, extra, shift):
    length, seed, k = tiles * TILE + extra, 7, 3
    U, S = _vectors(length, (length + 3) // 4 * 4 + 8, shift, sub, tiles + b)
    ctx = lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, b, lpc.CLIP_STD, 2.0, seed)
    codes, delta, clipped = ctx.quantize_pack(U, k, U_sub=S)
    ctx.sync_status()
    _check(U, S, None, b, lpc.CLIP_STD, 2.0, seed, k, codes, delta, clipped)
    ctx.close()


def _check(U, S, offs, b, clip, value, seed, k, codes, delta, clipped):
    V = (U if S is None else U - S).cpu().numpy()
    words = codes.cpu().numpy().view(np.uint32)
    offs = [0, V.shape[1]] if offs is None else offs
    woff, _ = lpc.packed_layout(V.shape[1], b, offs)
    for i in range(N):
        block = 0
        for s, (lo, hi) in enumerate(zip(offs, offs[1:])):
            w, dl, cl = orc.quantize_pack(np.ascontiguousarray(V[i, lo:hi]), b, clip, value, seed, i, k, block_base=block)
            assert delta[i, s].item() == dl and int(clipped[i, s]) == cl
            assert (words[i, woff[s]:woff[s] + orc.packed_words(hi - lo, b)] == w).all()
            block += (hi - lo + 7) // 8


HALF = FROM // 2  # tiles of each of the two vectors at the line
CLIPS = [(lpc.CLIP_NONE, 1.0), (lpc.CLIP_LAMBDA, 0.5), (lpc.CLIP_STD, 2.0)]  # the first two form no sums


@pytest.mark.parametrize("sub", [False, True])
@pytest.mark.parametrize("rule,tiles,extra,shift,pad,offs,kept", [
    (0, HALF, 0, 0, 0, None, 0),             # the last size that stays in L2 by itself
    (1, HALF, 1, 0, 7, None, KEPT),          # one value more
    (2, HALF + 2, -5, 8, 5, None, KEPT),     # a ragged end, vectors off the allocation's start
    (0, HALF + 2, 0, 4, 0, None, 0),         # 16-byte loads carry no policy
    (1, HALF + 2, 0, 0, 4, None, 0),         # every second row off 32 bytes
    (2, HALF + 2, -3, 1, 2, None, 0),
    (0, HALF + 2, 0, 0, 0, [0, 24, 64, 8 * TILE, 700 * TILE + 8], KEPT),  # tensors of 24, 40 and many values, tiles that end early
    (1, HALF + 2, 0, 0, 0, [0, 24, 68, 700 * TILE + 8], 0),               # one of them off 32 bytes
])
def test_kept_tail_by_size_alignment_and_clip_rule(sub, rule, tiles, extra, shift, pad, offs, kept):
    length, seed, k, b = tiles * TILE + extra, 5, 2, 4
    clip, value = CLIPS[(rule + sub) % 3]
    U, S = _vectors(length, (length + pad + 7) // 8 * 8 + 8 + (4 if pad == 4 else 0), shift, sub, tiles + shift)
    offs = None if offs is None else offs + [length]
    ctx = lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, b, clip, value, seed)
    codes, delta, clipped = ctx.quantize_pack(U, k, U_sub=S, seg_offsets=offs)
    ctx.sync_status()
    assert ctx.query(lpc.INFO_QUANT_LAUNCHES) == 3 and ctx.query(lpc.INFO_QUANT_KEPT_TILES) == kept
    _check(U, S, offs, b, clip, value, seed, k, codes, delta, clipped)
    ctx.close()


@pytest.mark.parametrize("sub,times", [(False, 16), (True, 6)])
def test_no_policy_beyond_what_it_saves(sub, times):
    most = times * L2 // (2 if sub else 1) // (4 * TILE)  # tiles of each input
    # the codes of a vector depend on its row and its values alone: both calls are held against shorter calls on the same rows
    length = (most // N + 1) * TILE
    U, S = _vectors(length, length, 0, sub, 1)
    ctx = lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, 4, lpc.CLIP_LAMBDA, 0.5, 3)
    U[:, 0] = 100.0  # the largest magnitude, and with it the scale, is the same in every call
    if sub:
        S[:, 0] = 0.0
    out = {}
    for tiles, kept in ((most // N, KEPT), (most // N + 1, 0), (FROM // N, 0)):
        V, W = U[:, :tiles * TILE], None if S is None else S[:, :tiles * TILE]
        codes, delta, _ = ctx.quantize_pack(V, 1, U_sub=W)
        ctx.sync_status()
        assert ctx.query(lpc.INFO_QUANT_KEPT_TILES) == kept
        out[tiles] = codes, delta
    (short, d0), (mid, d1), (long, d2) = out[FROM // N], out[most // N], out[most // N + 1]
    assert torch.equal(d0, d1) and torch.equal(d0, d2) and (d0 == 100.0 * 0.5 / 7).all()
    assert torch.equal(short, mid[:, :short.shape[1]]) and torch.equal(mid, long[:, :mid.shape[1]])
    ctx.close()
