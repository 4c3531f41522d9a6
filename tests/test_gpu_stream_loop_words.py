"""The streaming loop where the words of a group are fetched in whole accesses, one, two, four or eight of them by code width, sixteen a round:
bit for bit what one step at a time gives, with rounds that are full, ragged and single, and with slices of 512 columns."""
import pytest
import torch

from paper_1901_08924_b200 import lpc, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _pair(n, d, N, B, b, alpc, clip=lpc.CLIP_STD, value=2.0, want_slice=0):
    X, y, _ = synth.linear_problem(n, d, loss="logistic", sparsity=0.2, noise=0.1, seed=d + B, device=DEV)
    g = torch.Generator(device=DEV).manual_seed(d + B)
    x0 = 0.1 * torch.randn(d, generator=g, device=DEV)
    one, many = (lpc.Context(X, y, lpc.LOGISTIC, 1e-4, N, B, b, clip, value, 7) for _ in range(2))
    for c in (one, many):
        c.set_iterate(x0)
        if alpc:
            c.alpc_begin()
        c.snapshot_full_grad()
        if not alpc:
            c.set_iterate(x0 + 0.01)
    many.set_buffer(lpc.BUF_MU, one.get_buffer(lpc.BUF_MU))
    if alpc:
        many.alpc_double_sample_steps(0.4, 0.5, 0.3, 0.2, 3, 4)
    else:
        many.inner_steps(0.05, 3, 4)
    for k in range(3, 7):
        if alpc:
            one.alpc_double_sample_step(0.4, 0.5, 0.3, 0.2, k)
        else:
            one.inner_step(0.05, k)
    one.sync_status()
    many.sync_status()
    assert many.query(lpc.INFO_LOOP_LAUNCHES) == 1
    if want_slice:
        assert many.query(lpc.INFO_ALPC_STREAM_LOOP_SLICE if alpc else lpc.INFO_STREAM_LOOP_SLICE) == want_slice
    for w in [lpc.BUF_X, lpc.BUF_CODES, lpc.BUF_DELTA, lpc.BUF_CLIPPED] + ([lpc.BUF_Y, lpc.BUF_Z, lpc.BUF_YSUM, lpc.BUF_VHAT] if alpc else []):
        assert torch.equal(one.get_buffer(w).view(torch.int32), many.get_buffer(w).view(torch.int32)), w
    one.close()
    many.close()


@pytest.mark.parametrize("alpc", [False, True])
@pytest.mark.parametrize("b", [3, 5, 6, 7, 9, 10, 12, 15, 16, 32])
@pytest.mark.parametrize("N,d", [(1, 140), (3, 500), (17, 132)])
def test_every_width(N, d, b, alpc):
    _pair(510 // N * N, d, N, 70, b, alpc)


# slices of 512 columns, whose groups have sixteen rows in four row parts; the last slice of 4, 512 and 440
@pytest.mark.parametrize("alpc", [False, True])
@pytest.mark.parametrize("b", [1, 2, 4, 8, 3, 6, 9, 32])
@pytest.mark.parametrize("d,N,B", [(2052, 4, 70), (4096, 8, 256), (3000, 16, 77)])
def test_slices_of_512_columns(d, N, B, b, alpc):
    _pair(512, d, N, B, b, alpc, clip=lpc.CLIP_LAMBDA if b == 2 else lpc.CLIP_STD, value=0.5 if b == 2 else 2.0, want_slice=512)


@pytest.mark.parametrize("N,d,B,b,alpc,loops", [
    (16, 8192, 256, 4, False, 1), (64, 2552, 65, 4, True, 1),     # a fixed width always takes the loop
    (16, 8000, 256, 5, False, 0), (32, 8192, 256, 3, False, 0),   # clusters of eight with 128 CTAs; slices of 2,048 columns
    (8, 8192, 256, 3, False, 1), (32, 4000, 66, 32, False, 1),    # 64 CTAs; 128 of them in clusters of four
    (64, 2000, 100, 32, False, 0), (4, 10000, 100, 32, False, 0),
    (3, 10000, 100, 9, False, 1), (3, 10000, 100, 9, True, 0), (3, 10000, 64, 9, True, 1),
    (20, 10000, 100, 9, False, 1), (32, 5000, 33, 32, False, 1),  # single steps need two rounds of clusters; keep their rows resident
    (64, 900, 256, 7, True, 1), (33, 1000, 100, 32, True, 1),     # slices of 512 columns and narrower ones
])
def test_lines_of_the_rule(N, d, B, b, alpc, loops):
    X, y, _ = synth.linear_problem(N * 16, d, loss="logistic", sparsity=0.2, noise=0.1, seed=1, device=DEV)
    c = lpc.Context(X, y, lpc.LOGISTIC, 1e-4, N, B, b, lpc.CLIP_STD, 2.0, 7)
    c.set_iterate(torch.zeros(d, device=DEV))
    if alpc:
        c.alpc_begin()
    c.snapshot_full_grad()
    if alpc:
        c.alpc_double_sample_steps(0.4, 0.5, 0.3, 0.2, 0, 2)
    else:
        c.inner_steps(0.05, 0, 2)
    c.sync_status()
    assert c.query(lpc.INFO_LOOP_LAUNCHES) == loops
    assert (c.query(lpc.INFO_ALPC_STREAM_LOOP_SLICE if alpc else lpc.INFO_STREAM_LOOP_SLICE) > 0) == bool(loops)
    c.close()
