"""CPU-only checks of the streaming loop's launch plan: whatever the shape, its slices stay inside the exchange buffers."""
import itertools

import pytest

SMEM, SMS = 231424, 148  # a B200's


@pytest.fixture(scope="module")
def lpc():
    from paper_1901_08924_b200 import build, lpc as binding
    build.build()
    return binding


def test_slices_stay_inside_the_exchange_buffers(lpc):
    # narrow slices need more than 64 rows, so few rows of a short vector lead to slices wider than the vector; the CTAs of a worker write
    # words for every column of their slices
    taken = 0
    dims = [4, 64, 124, 128, 132, 256, 260, 512, 516, 1000, 1024, 1028, 2044, 2048, 2052, 4096, 8192, 8196, 16384]
    for d, N, B, alpc in itertools.product(dims, (1, 2, 16, 33, 64), (9, 10, 16, 17, 32, 33, 40, 50, 64, 65, 100, 256), (0, 1)):
        for SL in (128, 256, 512, 1024, 2048):
            ctas, room = lpc.debug_stream_loop_slices(d, N, B, alpc, SMEM, SMS, SL)
            assert room >= max(d, 128) and room & (room - 1) == 0
            if ctas:
                taken += 1
                assert (ctas - 1) * SL < d <= ctas * SL <= room, (d, N, B, alpc, SL)
    assert taken > 1000


def test_arguments(lpc):
    assert lpc.debug_stream_loop_slices(128, 2, 256, 0, SMEM, SMS, 128) == (1, 128)
    assert lpc.debug_stream_loop_slices(4096, 16, 256, 0, SMEM, SMS, 512) == (8, 4096)
    assert lpc.debug_stream_loop_slices(1000, 64, 16, 0, SMEM, SMS, 2048) == (0, 1024)
    assert lpc.debug_stream_loop_slices(128, 2, 256, 0, 0, SMS, 128)[0] == 0       # no shared memory
    assert lpc.debug_stream_loop_slices(16384, 19, 256, 0, SMEM, SMS, 2048)[0] == 0  # 152 CTAs
    for bad in (64, 192, 4096):
        with pytest.raises(lpc.LpcError):
            lpc.debug_stream_loop_slices(128, 2, 256, 0, SMEM, SMS, bad)
