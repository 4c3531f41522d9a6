"""The scale of the one-launch loop, which is formed in single precision with an interval around the threshold and by doubles where
that does not decide: bit for bit the scales of one-step launches, which take the doubles.  Gradients from 2^-100 to 2^100, with
means up to a thousand deviations, with one coordinate that is not zero, constant ones."""
import numpy as np
import pytest
import torch

from paper_1901_08924_b200 import lpc

pytestmark = pytest.mark.gpu


def _same(a, b):
    return torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))


@pytest.mark.parametrize("kind", ["gauss", "mean", "single", "constant"])
@pytest.mark.parametrize("exponent", [-55, -30, -13, 0, 20, 50])
@pytest.mark.parametrize("b,value", [(1, 0.5), (2, 2.5), (3, 3.0000002), (4, 3.0), (8, 2.0), (32, 1.0)])
def test_loop_scales_equal_single_steps(kind, exponent, b, value):
    N, B, d, n, count = 4, 1, 1000, 64, 40
    rng = np.random.default_rng((exponent + 100) * 7 + b)
    X = rng.standard_normal((n, d))
    if kind == "mean":
        X = X + np.exp2(rng.uniform(-4, 10, (n, 1)))
    elif kind == "single":
        X = np.where(np.arange(d) == rng.integers(0, d, (n, 1)), X, 0.0)
    elif kind == "constant":
        X = np.repeat(X[:, :1], d, axis=1)
    # u = (X_a (x - x~)) X_a grows with the square of the rows' scale
    X = torch.from_numpy((X * np.exp2(exponent)).astype(np.float32)).cuda()
    y = torch.from_numpy(rng.standard_normal(n).astype(np.float32)).cuda()
    shift = torch.from_numpy((rng.standard_normal(d) * 0.1).astype(np.float32)).cuda()
    out = []
    for persistent in (0, 1):
        c = lpc.Context(X, y, lpc.LEAST_SQUARES, 0.0, N, B, b, lpc.CLIP_STD, value, 5)
        c.set_option(lpc.OPT_PERSISTENT, persistent)
        c.snapshot_full_grad()
        c.set_iterate(shift)  # away from the snapshot, or the first step's u is zero
        deltas = []
        for k in range(0, count, 2):  # two steps per call: the loop leaves the last step's scales
            c.inner_steps(0.0, k, 2)  # step 0: the iterate stays, every pair of steps sees other rows
            deltas.append(c.get_buffer(lpc.BUF_DELTA).clone())
        c.status()
        assert c.query(lpc.INFO_LOOP_LAUNCHES) == (count // 2 if persistent else 0)
        out.append((torch.stack(deltas), c.get_buffer(lpc.BUF_CODES), c.get_buffer(lpc.BUF_CLIPPED)))
        c.close()
    for a, e in zip(*out):
        assert _same(a, e)


def _definition(bits, S1, S2, length, b, mode, value):
    """Eq. 2 and the c * std threshold with every operation in doubles, rounded once; then float32 operations, as numpy rounds them."""
    M = bits.view(np.float32)
    with np.errstate(all="ignore"):
        if mode == lpc.CLIP_STD:
            mean, ex2 = S1.astype(np.float64) / length, S2.astype(np.float64) / length
            t = np.float64(np.float32(value)) * np.sqrt(np.maximum(ex2 - mean * mean, 0.0))
            T = np.minimum(t, M).astype(np.float32)
        else:
            T = M * np.float32(value) if mode == lpc.CLIP_LAMBDA else M.copy()
        one = np.float32(1.0)
        delta = np.full_like(T, one) if b == 32 else T if b == 1 else T / np.float32(2 ** (b - 1) - 1)
        rdelta = one / delta
        lower = -T if b in (1, 32) else -(T + delta)
        zero = np.zeros_like(T, bool) if b == 32 else (M == 0) | (T == 0) | (delta == 0) | np.isinf(rdelta)
    bad = bits >= 0x7F800000
    out = np.stack([np.where(zero, 0, delta), np.where(zero, 0, rdelta), T, np.where(zero, 0, lower)], axis=1).astype(np.float32)
    out[bad] = [np.nan, 0, 0, 0]
    return out, np.where(bad, 3, zero.astype(np.int32))


@pytest.mark.parametrize("length", [1, 1000, 4096, 11689512])
@pytest.mark.parametrize("b,mode,value", [
    (2, lpc.CLIP_STD, 2.0), (4, lpc.CLIP_STD, 3.0000002), (8, lpc.CLIP_STD, 2.5), (1, lpc.CLIP_STD, 0.1), (32, lpc.CLIP_STD, 1.0),
    (16, lpc.CLIP_STD, 9e5), (3, lpc.CLIP_STD, 1e-7), (3, lpc.CLIP_STD, 1e7), (5, lpc.CLIP_LAMBDA, 0.3), (7, lpc.CLIP_NONE, 1.0)])
def test_loop_scales_equal_the_definition_and_both_branches_decide(length, b, mode, value):
    count = 1 << 19
    rng = np.random.default_rng(b * 100 + length % 97)
    sigma = np.exp2(rng.uniform(-60, 60, count))       # variances over the whole range of floats, so outside the interval's range too
    mean = sigma * rng.choice([-1.0, 1.0], count) * np.exp2(rng.uniform(-8, 6, count))  # to where nothing of the second moment is left
    M = (sigma * rng.uniform(0.05, 8.0, count)).astype(np.float32)
    M[:64], M[64:96] = 0.0, np.float32(1e-44)
    bits = M.view(np.uint32).copy()
    bits[96:128] = rng.choice([0x7F800000, 0x7FC00000, 0x7FFFFFFF], 32)
    with np.errstate(over="ignore"):
        S1, S2 = (length * mean).astype(np.float32), (length * (sigma * sigma + mean * mean)).astype(np.float32)
    scale, flags = lpc.debug_loop_scales(*(torch.from_numpy(a).cuda() for a in (bits.view(np.int32), S1, S2)), length, b, mode, value)
    scale, flags = scale.cpu().numpy(), flags.cpu().numpy()
    want, want_flags = _definition(bits, S1, S2, length, b, mode, value)
    assert (flags & 3 == want_flags).all()
    assert ((scale.view(np.uint32) == want.view(np.uint32)) | (np.isnan(scale) & np.isnan(want))).all()
    doubles = (flags & 4) != 0
    if mode != lpc.CLIP_STD:
        assert not doubles.any()
        return
    with np.errstate(all="ignore"):
        x = S2.astype(np.float64) / length
        v = x - (S1.astype(np.float64) / length) ** 2
    asked = (bits != 0) & (bits < 0x7F800000)
    inside = asked & (v > 0.26 * x) & (v > 1.1e-25) & (v < 0.9e25)  # a margin around the rule's own, rounded tests
    outside = asked & ~((v > 0.24 * x) & (v > 0.9e-25) & (v < 1.1e25))
    assert inside.sum() > count // 4 and outside.sum() > count // 8
    assert doubles[outside].all()
    if 1e-6 <= value <= 1e6:
        # the interval of 2 * 2^-38 takes 2^-14 to 2^-13 of the spacing of floats: 6e-5 to 1.2e-4 of the cases
        assert 2e-5 < doubles[inside].mean() < 3e-4
    else:
        assert doubles[asked].all()
