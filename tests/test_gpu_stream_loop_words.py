"""The streaming loop where the words of a group are fetched in whole accesses, one, two, four or eight of them by code width, sixteen a round:
bit for bit what one step at a time gives, with rounds that are full, ragged and single, and with slices of 512 columns."""
import pytest
import torch

from paper_1901_08924_b200 import lpc, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _pair(n, d, N, B, b, alpc, clip=lpc.CLIP_STD, value=2.0):
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
    for w in [lpc.BUF_X, lpc.BUF_CODES, lpc.BUF_DELTA, lpc.BUF_CLIPPED] + ([lpc.BUF_Y, lpc.BUF_Z, lpc.BUF_YSUM, lpc.BUF_VHAT] if alpc else []):
        assert torch.equal(one.get_buffer(w).view(torch.int32), many.get_buffer(w).view(torch.int32)), w
    one.close()
    many.close()


@pytest.mark.parametrize("alpc", [False, True])
@pytest.mark.parametrize("b", [3, 5, 6, 7, 9, 10, 12, 15, 16, 32])
@pytest.mark.parametrize("N,d", [(1, 140), (3, 500), (17, 132)])
def test_every_width(N, d, b, alpc):
    _pair(510 // N * N, d, N, 70, b, alpc)


# by the plan's arithmetic on 148 SMs: slices of 512 columns, whose groups have sixteen rows in four row parts; the last slice of 4, 512 and 440
@pytest.mark.parametrize("alpc", [False, True])
@pytest.mark.parametrize("b", [1, 2, 4, 8, 3, 6, 9, 32])
@pytest.mark.parametrize("d,N,B", [(2052, 4, 70), (4096, 8, 256), (3000, 16, 77)])
def test_slices_of_512_columns(d, N, B, b, alpc):
    assert lpc.debug_stream_loop_slices(d, N, B, alpc, 231424, 148, 256)[0] == 0
    assert lpc.debug_stream_loop_slices(d, N, B, alpc, 231424, 148, 512)[0] == (d + 511) // 512
    _pair(512, d, N, B, b, alpc, clip=lpc.CLIP_LAMBDA if b == 2 else lpc.CLIP_STD, value=0.5 if b == 2 else 2.0)
