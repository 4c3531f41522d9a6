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
