"""The one-launch loop for large minibatches, whose rows stream: bit for bit what one step at a time gives, for every slice width, full and
ragged slices and groups of rows, clusters of one to eight CTAs, every code width, clip rule and loss, both algorithms, twice in a row."""
import pytest
import torch

from paper_1901_08924_b200 import lpc, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _same(a, b):
    return torch.equal(a.view(torch.int32) if a.dtype == torch.float32 else a, b.view(torch.int32) if b.dtype == torch.float32 else b)


def _problem(n, d, loss, seed):
    X, y, _ = synth.linear_problem(n, d, loss=loss, sparsity=0.2, noise=0.1, seed=seed, device=DEV)
    g = torch.Generator(device=DEV).manual_seed(seed)
    return X, y, 0.1 * torch.randn(d, generator=g, device=DEV)


def _pair(n, d, N, B, b, alpc, loss="logistic", clip=lpc.CLIP_STD, value=2.0, options=(), sigma=0.0, counts=(3, 4), want=None):
    X, y, x0 = _problem(n, d, loss, d + B)
    code = lpc.LOGISTIC if loss == "logistic" else lpc.LEAST_SQUARES
    one, many = (lpc.Context(X, y, code, 1e-4, N, B, b, clip, value, 7) for _ in range(2))
    for c in (one, many):
        for o, v in options:
            c.set_option(o, v)
        if sigma:
            c.set_strong_convexity(sigma)
        c.set_iterate(x0)
        if alpc:
            c.alpc_begin()
        c.snapshot_full_grad()
        if not alpc:
            c.set_iterate(x0 + 0.01)  # away from the snapshot: the first u is not zero
    many.set_buffer(lpc.BUF_MU, one.get_buffer(lpc.BUF_MU))
    par = (0.4, 0.5, 0.3, 0.2) if alpc else (0.05,)
    k = 11
    for count in counts:
        for c in (one, many):
            step, steps = (c.alpc_double_sample_step, c.alpc_double_sample_steps) if alpc else (c.inner_step, c.inner_steps)
            if c is many:
                steps(*par, k, count)
            else:
                for i in range(count):
                    step(*par, k + i)
        k += count
    one.sync_status()
    many.sync_status()
    assert one.query(lpc.INFO_LOOP_LAUNCHES) == 0
    assert many.query(lpc.INFO_LOOP_LAUNCHES) == (len(counts) if want is None else want)
    which = [lpc.BUF_X, lpc.BUF_CODES, lpc.BUF_DELTA, lpc.BUF_CLIPPED, lpc.BUF_BATCH_IDX, lpc.BUF_COEF]
    for w in which + ([lpc.BUF_Y, lpc.BUF_Z, lpc.BUF_YSUM, lpc.BUF_VHAT] if alpc else []):
        p, q = one.get_buffer(w), many.get_buffer(w)
        if not alpc and w in (lpc.BUF_BATCH_IDX, lpc.BUF_COEF):
            p, q = p[:N], q[:N]  # the last row belongs to Algorithm 2's shared batch
        assert _same(p, q), w
    assert one.comm_bits() == many.comm_bits()
    if sigma:
        for c in (one, many):
            c.alpc_end_epoch(sum(counts))
        assert _same(one.get_iterate(), many.get_iterate())
    one.close()
    many.close()


@pytest.mark.parametrize("alpc", [False, True])
@pytest.mark.parametrize("n,d,N,B,b", [
    (512, 64, 4, 100, 4),      # slices of 128, not half full; groups of 32 rows, the last of 4
    (512, 1000, 2, 65, 2),     # 128 x 8, the last slice of 104; three groups
    (512, 1100, 5, 129, 8),    # 256 x 5
    (512, 2044, 8, 96, 1),     # 256 x 8, the last of 252
    (1024, 1028, 17, 200, 3),  # slices of 256 or 512 for 17 workers
    (1024, 700, 33, 256, 4),   # more clusters: wider slices
    (512, 5000, 2, 255, 16),   # 1,024 x 5, the last of 904
    (512, 8192, 8, 77, 4),     # 1,024 x 8
    (256, 8196, 2, 70, 2),     # 2,048 x 5, the last of 4 columns; groups of 4 rows, the last of 2
    (512, 12288, 3, 129, 8),   # 2,048 x 6; a last group of one row
    (256, 16384, 2, 256, 4),   # 2,048 x 8
    (512, 4000, 32, 66, 32),   # full precision
    (512, 300, 1, 256, 5),     # one worker
    (1280, 132, 64, 100, 2),   # many workers
])
def test_loop_equals_single_steps(n, d, N, B, b, alpc):
    _pair(n // N * N, d, N, B, b, alpc)


@pytest.mark.parametrize("alpc", [False, True])
@pytest.mark.parametrize("clip,value", [(lpc.CLIP_NONE, 1.0), (lpc.CLIP_LAMBDA, 0.5)])
@pytest.mark.parametrize("d,b", [(900, 4), (4100, 8), (10000, 3)])
def test_clip_rules_losses_and_options(d, b, clip, value, alpc):
    _pair(512, d, 2, 101, b, alpc, loss="least_squares", clip=clip, value=value,
          options=((lpc.OPT_SAMPLE_GLOBAL, 1), (lpc.OPT_LOOP_COOPERATIVE, 0)), counts=(2, 131))


@pytest.mark.parametrize("n,d,N,B,b", [(512, 9000, 8, 16, 4), (512, 8200, 16, 9, 2), (512, 16384, 2, 32, 8), (1024, 4096, 32, 64, 4)])
@pytest.mark.parametrize("alpc", [False, True])
def test_small_minibatches_of_long_rows(n, d, N, B, b, alpc):
    # rows or clusters that the loop with resident rows has no room for: three groups of rows are enough for this one
    _pair(n, d, N, B, b, alpc)


def test_strongly_convex_weights():
    _pair(512, 1500, 4, 80, 4, True, sigma=0.01)
    _pair(512, 9000, 2, 80, 2, True, sigma=0.01)


def test_paths_that_stay_with_single_launches():
    # taps and profiles need the kernels of a step one by one; so does a cluster size that the caller asks for
    for option in (lpc.OPT_TAP_U, lpc.OPT_PROFILE):
        _pair(512, 1000, 2, 100, 4, False, options=((option, 1),), want=0)
    _pair(512, 1000, 2, 100, 4, False, options=((lpc.OPT_CLUSTER_SIZE, 2),), want=0)
    _pair(1024, 1000, 2, 300, 4, False, want=0)  # more rows than the loop takes


def test_captured_steps_replay():
    # the loop hands words over under tags that a replay would repeat: captured steps are plain launches
    B = 100
    X, y, x0 = _problem(512, 1000, "logistic", 1)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        c, ref = (lpc.Context(X, y, lpc.LOGISTIC, 1e-4, 4, B, 4, lpc.CLIP_STD, 2.0, 7) for _ in range(2))
        for a in (c, ref):
            a.set_iterate(x0)
            a.snapshot_full_grad()
        c.set_buffer(lpc.BUF_MU, ref.get_buffer(lpc.BUF_MU))
        c.inner_steps(0.05, 0, 5)
        ref.inner_steps(0.05, 0, 5)
        c.sync_status()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            c.inner_steps(0.05, 5, 140)
        for _ in range(3):  # every replay goes on from where the last one ended
            graph.replay()
            for k in range(5, 145):
                ref.inner_step(0.05, k)
            assert _same(c.get_iterate(), ref.get_iterate())
        assert c.query(lpc.INFO_LOOP_LAUNCHES) == 1
        c.sync_status()
        c.close()
        ref.close()


def test_non_finite_gradients_are_reported():
    X, y, x0 = _problem(512, 1000, "least_squares", 3)
    X[130:260, 5] = 1e25  # the rows of one worker: their products overflow
    for persistent in (0, 1):
        c = lpc.Context(X, y, lpc.LEAST_SQUARES, 1e-4, 4, 100, 4, lpc.CLIP_STD, 2.0, 7)
        c.set_option(lpc.OPT_PERSISTENT, persistent)
        c.set_iterate(x0)
        c.set_buffer(lpc.BUF_MARGINS, torch.zeros(512, device=DEV))
        c.set_buffer(lpc.BUF_MU, torch.zeros(1000, device=DEV))
        c.inner_steps(0.05, 0, 3)
        assert c.status() == lpc.ERR_NONFINITE and c.status() == lpc.OK
        assert c.query(lpc.INFO_LOOP_LAUNCHES) == persistent
        c.close()


def test_clipped_counts_of_a_step_after_a_loop_with_more_ctas():
    # a loop has more CTAs per worker than a single step: their counts must not stay in the sum
    X, y, x0 = _problem(512, 1000, "logistic", 4)
    c, ref = (lpc.Context(X, y, lpc.LOGISTIC, 1e-4, 4, 100, 4, lpc.CLIP_STD, 1.0, 7) for _ in range(2))
    for a in (c, ref):
        a.set_iterate(x0)
        a.snapshot_full_grad()
        a.set_iterate(x0 + 0.01)
    c.inner_steps(0.0, 0, 3)
    c.inner_step(0.0, 3)
    ref.inner_step(0.0, 3)
    assert c.query(lpc.INFO_LOOP_LAUNCHES) == 1
    assert torch.equal(c.get_buffer(lpc.BUF_CLIPPED), ref.get_buffer(lpc.BUF_CLIPPED)) and c.get_buffer(lpc.BUF_CLIPPED).sum() > 0
    c.close()
    ref.close()
