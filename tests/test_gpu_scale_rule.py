"""The c * std scale rule on vectors whose sums, lengths and thresholds cover its branches: the threshold is formed in single
precision with an interval around it, and by doubles where that interval does not decide; the scale, its reciprocal (through
the codes) and the counts have to be the oracle's bits either way."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_1901_08924_b200 import lpc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b", [1, 2, 3, 4, 7, 8, 16, 32])
@pytest.mark.parametrize("length", [1, 3, 64, 1000, 4099])
def test_scale_of_many_vectors_bit_exact(b, length):
    # 512 vectors per call: scales over 2^-140 .. 2^120 (second moments underflow and overflow), constant vectors (variance zero
    # or rounding noise), a mean far above the deviation, one outlier, a single value
    rng = np.random.default_rng(1000 * b + length)
    N = 512
    U = rng.standard_normal((N, length)) * np.exp2(rng.uniform(-140, 60, (N, 1)))
    U[1::8] += np.abs(U[1::8]).max(axis=1, keepdims=True) * 1000.0
    U[2::8] = U[2::8, :1]
    U[3::8] *= 0.0
    U[3::8, 0] = rng.standard_normal(U[3::8, 0].shape)
    U[4::8] = rng.standard_normal(U[4::8].shape) * np.exp2(rng.uniform(60, 120, (U[4::8].shape[0], 1)))
    U = U.astype(np.float32)
    for value in (0.5, 2.5, 3.0000002):
        ctx = lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, b, lpc.CLIP_STD, value, 3)
        codes, delta, clipped = ctx.quantize_pack(torch.from_numpy(U).cuda(), 1)
        ctx.status()
        got = delta.cpu().numpy()[:, 0].view(np.uint32)
        W = orc.packed_words(length, b)
        words = codes.cpu().numpy().view(np.uint32)[:, :W]
        for i in range(N):
            w, dl, cl = orc.quantize_pack(U[i], b, orc.CLIP_STD, value, 3, i, 1)
            assert got[i] == np.float32(dl).view(np.uint32), (i, value)
            assert (words[i] == w).all() and int(clipped[i, 0]) == cl, (i, value)
        ctx.close()
