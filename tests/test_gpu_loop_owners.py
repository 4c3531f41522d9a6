"""The one-launch loop where each coordinate's update belongs to one CTA: worker counts and widths around the rule that takes it,
slices that the workers do not divide evenly, coordinates that end inside an owner's share, empty slices; bit for bit the
iterates, codes and estimators of one-step launches."""
import numpy as np
import pytest
import torch

from paper_1901_08924_b200 import lpc, synth

pytestmark = pytest.mark.gpu


def _same(a, b):
    return torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))


OWN = {False: (lpc.INFO_LOOP_CLUSTER_SIZE, lpc.INFO_LOOP_OWNED), True: (lpc.INFO_ALPC_LOOP_CLUSTER_SIZE, lpc.INFO_ALPC_LOOP_OWNED)}


@pytest.mark.parametrize("alpc", [False, True])
@pytest.mark.parametrize("n,d,N,B,b,own", [
    (17 * 8, 4096, 17, 3, 4, 1),    # the first count beyond sixteen; shares of 64 coordinates of a slice of 1,024
    (16 * 8, 4096, 16, 3, 4, 0),    # sixteen: every cluster updates its copy
    (31 * 8, 8188, 31, 16, 2, 1),   # 31 shares of 72 in slices of 2,048, the last column inside one; rows that do not fit a step ahead
    (32 * 4, 5000, 32, 2, 8, 1),    # the last CTA of a cluster has few columns
    (24 * 4, 64, 24, 1, 1, 1),      # more workers than groups of eight coordinates
    (33 * 4, 2052, 33, 4, 4, 1),    # slices that are half empty
    (2 * 16, 512, 2, 5, 3, 1),      # widths known at run time: owners from one worker on
    (4 * 16, 256, 1, 5, 3, 1),
    (5 * 16, 1000, 5, 32, 6, 1),
    (16 * 8, 2048, 16, 8, 32, 1),
    (4 * 16, 512, 1, 5, 3, 0),      # more coordinates to an owner than threads
    (4 * 16, 2048, 4, 8, 3, 0),     # but not for three or four in clusters of four CTAs whose rows stay in registers
    (3 * 16, 2048, 3, 8, 16, 0),
    (4 * 16, 2048, 4, 9, 3, 1),
    (5 * 16, 2048, 5, 8, 3, 1),
    (4 * 16, 512, 4, 4, 32, 1),
    (4 * 16, 508, 4, 4, 32, (1, 0)),  # Algorithm 1 / Algorithm 2, whose short vectors of whole floats are updated by everybody
    (64 * 2, 1024, 64, 2, 16, 1),   # the most workers the loop takes
    (32 * 8, 8192, 32, 25, 2, 1),   # the most rows that leave room for the products (8 KB), one more, and too many for the loop
    (32 * 8, 8192, 32, 26, 2, 0),
    (32 * 8, 8192, 32, 27, 2, None),
])
def test_owned_update_equals_single_steps(n, d, N, B, b, own, alpc):
    X, y, _ = synth.linear_problem(n, d, loss="least_squares", sparsity=0.2, noise=0.1, seed=d + N)
    X, y = X.cuda(), y.cuda()
    x0 = torch.from_numpy((np.random.default_rng(3).standard_normal(d) * 0.1).astype(np.float32)).cuda()
    one, many = (lpc.Context(X, y, lpc.LEAST_SQUARES, 1e-5, N, B, b, lpc.CLIP_STD, 2.0, 11) for _ in range(2))
    count = 9
    for c in (one, many):
        c.set_option(lpc.OPT_TAP_U, 1)
        c.set_iterate(x0)
        if alpc:
            c.alpc_begin()
        c.snapshot_full_grad()
    one.set_option(lpc.OPT_PERSISTENT, 0)
    par = (0.4, 0.5, 0.3, 0.2)
    for k in range(2 * count):
        if alpc:
            one.alpc_double_sample_step(*par, k)
        else:
            one.inner_step(0.05, k)
    for k0 in (0, count):  # two launches: the second one's words must not be taken for the first one's
        if alpc:
            many.alpc_double_sample_steps(*par, k0, count)
        else:
            many.inner_steps(0.05, k0, count)
    one.sync_status()
    many.sync_status()
    cluster, owned = (many.query(q) for q in OWN[alpc])
    assert (owned if cluster else None) == (own[alpc] if isinstance(own, tuple) else own)
    assert many.query(lpc.INFO_LOOP_LAUNCHES) == (2 if cluster else 0)
    for w in [lpc.BUF_X, lpc.BUF_CODES, lpc.BUF_DELTA, lpc.BUF_U, lpc.BUF_V, lpc.BUF_CLIPPED] + (
            [lpc.BUF_Y, lpc.BUF_Z, lpc.BUF_YSUM, lpc.BUF_VHAT] if alpc else []):
        assert _same(one.get_buffer(w), many.get_buffer(w)), w
    assert torch.isfinite(many.get_iterate()).all()
    one.close()
    many.close()


@pytest.mark.parametrize("alpc", [False, True])
@pytest.mark.parametrize("n,d,N,b,at", [
    (17 * 8, 1000, 17, 4, 512),   # the last slice ends early; its first coordinate is the infinite one
    (33 * 4, 2052, 33, 4, 2048),  # four columns in a slice of 1,024
    (33 * 4, 2052, 33, 4, 0),     # an empty slice: its threads hold no coordinate, the first one is infinite
    (4 * 16, 64, 4, 3, 0),        # a slice narrower than a pass
    (64 * 2, 996, 64, 16, 512),
])
def test_columns_outside_a_slice_stay_zero_beside_an_infinite_coordinate(n, d, N, b, at, alpc):
    # a logistic margin may be infinite, its derivative is not: gradients, scales and codes stay finite as long as
    # nobody multiplies the infinite coordinate by the zeros that stand for columns that do not exist
    X, y, _ = synth.linear_problem(n, d, loss="logistic", sparsity=0.2, noise=0.1, seed=d + N)
    X[:, at] = X[:, at].abs() + 0.5  # 0 * inf in the column itself would be a NaN of its own
    X, y = X.cuda(), y.cuda()
    x0 = torch.from_numpy((np.random.default_rng(3).standard_normal(d) * 0.1).astype(np.float32)).cuda()
    far = x0.clone()
    far[at] = float("inf")
    one, many = (lpc.Context(X, y, lpc.LOGISTIC, 1e-5, N, 3, b, lpc.CLIP_STD, 2.0, 11) for _ in range(2))
    one.set_option(lpc.OPT_PERSISTENT, 0)
    par, count = (0.4, 0.5, 0.3, 0.2), 4
    for c in (one, many):
        c.set_iterate(x0)
        if alpc:
            c.alpc_begin()
        c.snapshot_full_grad()
        if alpc:
            c.set_buffer(lpc.BUF_Y, far)
            c.set_buffer(lpc.BUF_Z, far)
        else:
            c.set_iterate(far)
        if alpc:
            c.alpc_double_sample_steps(*par, 0, count)
        else:
            c.inner_steps(0.05, 0, count)
        c.sync_status()
    assert many.query(lpc.INFO_LOOP_LAUNCHES) == 1 and many.query(OWN[alpc][1]) == 1
    for w in [lpc.BUF_X, lpc.BUF_CODES, lpc.BUF_DELTA] + ([lpc.BUF_Y, lpc.BUF_Z, lpc.BUF_YSUM] if alpc else []):
        assert _same(one.get_buffer(w), many.get_buffer(w)), w
    delta, x = many.get_buffer(lpc.BUF_DELTA), many.get_iterate()
    assert torch.isfinite(delta).all() and (delta > 0).all()
    assert x[at] == float("inf") and torch.isfinite(x).sum() == d - 1
    one.close()
    many.close()


@pytest.mark.parametrize("alpc", [False, True])
@pytest.mark.parametrize("n,d,N,b", [(17 * 8, 1000, 17, 4), (33 * 4, 2052, 33, 2), (5 * 16, 512, 5, 3), (4 * 16, 1024, 4, 32)])
def test_owned_update_with_gradients_that_are_not_finite(n, d, N, b, alpc):
    # least squares with entries whose products overflow in the rows of one worker: its message is a NaN scale with zero codes (b = 32:
    # its values), which the proximal step takes to 0, and the loop goes on and ends with the status of single steps
    X, y, _ = synth.linear_problem(n, d, loss="least_squares", sparsity=0.2, noise=0.1, seed=d + N)
    rows = n // N
    X[2 * rows:3 * rows, 5] = 1e25
    X, y = X.cuda(), y.cuda()
    x0 = torch.from_numpy((np.random.default_rng(3).standard_normal(d) * 0.1).astype(np.float32)).cuda()
    count, out = 3, []
    for persistent in (0, 1):
        c = lpc.Context(X, y, lpc.LEAST_SQUARES, 1e-5, N, 3, b, lpc.CLIP_STD, 2.0, 11)
        c.set_option(lpc.OPT_PERSISTENT, persistent)
        c.set_iterate(x0)
        if alpc:
            c.alpc_begin()
        for w in (lpc.BUF_MARGINS, lpc.BUF_MU):  # the snapshot's own values stay finite
            c.set_buffer(w, torch.zeros(n if w == lpc.BUF_MARGINS else d, device="cuda"))
        if alpc:
            c.alpc_double_sample_steps(0.4, 0.5, 0.3, 0.2, 0, count)
        else:
            c.inner_steps(0.05, 0, count)
        assert c.status() == lpc.ERR_NONFINITE
        assert c.query(lpc.INFO_LOOP_LAUNCHES) == persistent and (not persistent or c.query(OWN[alpc][1]) == 1)
        out.append([c.get_buffer(w) for w in (lpc.BUF_X, lpc.BUF_DELTA, lpc.BUF_CODES, lpc.BUF_CLIPPED)])
        assert c.status() == lpc.OK  # reported once
        c.close()
    for a, e in zip(*out):
        if a.dtype == torch.float32:  # NaNs, and zeros with the sign of one, need not have the same bits
            assert torch.equal(torch.isnan(a), torch.isnan(e)) and torch.equal(torch.nan_to_num(a, nan=0.0), torch.nan_to_num(e, nan=0.0))
        else:
            assert torch.equal(a, e)
