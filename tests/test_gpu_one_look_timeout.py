"""What a wait that runs out leaves behind in the quantizer's one look at many tensors: the call ends and reports it, whether tiles had been
described by then or not, and the calls after it are right, their counts of clipped values among them."""
import pytest
import torch

from paper_1901_08924_b200 import lpc

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("b,clip,value", [(4, lpc.CLIP_STD, 1.0), (6, lpc.CLIP_LAMBDA, 0.5)])
def test_calls_after_a_wait_that_ran_out(b, clip, value):
    N, length = 16, 2400000  # 293 tiles of a worker in eight tensors; about 32 of them per CTA
    offs = [0, 8192, 8200, 300000, 600004, 900000, 1500000, 2000000, length]
    g = torch.Generator(device=DEV).manual_seed(b)
    U, S = (torch.randn((N, length), generator=g, device=DEV) for _ in range(2))
    ctx, ref = (lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, b, clip, value, 3) for _ in range(2))
    ref.set_option(lpc.OPT_ONE_LAUNCH_QUANTIZE, 0)
    want = ref.quantize_pack(U, 7, U_sub=S, seg_offsets=offs)
    ref.sync_status()
    assert want[2].sum() > 0
    for tiles in (0, 1, 3, 9, 20, 1 << 20):  # the last one is never reached
        ctx.debug_one_look_stop(tiles)
        ctx.quantize_pack(U, 5, U_sub=S, seg_offsets=offs)
        assert ctx.status() == (lpc.OK if tiles > 100 else lpc.ERR_TIMEOUT) and ctx.status() == lpc.OK
        for _ in range(2):
            got = ctx.quantize_pack(U, 7, U_sub=S, seg_offsets=offs)
            assert ctx.status() == lpc.OK and ctx.query(lpc.INFO_QUANT_LAUNCHES) == 1
            for p, q in zip(got, want):
                assert torch.equal(p.view(torch.int32), q.view(torch.int32)), tiles
    with pytest.raises(lpc.LpcError):
        ctx.debug_one_look_stop(-1)
    ctx.close()
    ref.close()
