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


@pytest.mark.parametrize("b,clip,value", [(4, lpc.CLIP_STD, 1.0), (3, lpc.CLIP_LAMBDA, 0.5), (8, lpc.CLIP_STD, 3.0)])
def test_tiles_that_never_come_are_looked_at_by_those_who_need_them(b, clip, value):
    # the first CTA does nothing: the scales of all messages that it has a tile of need that tile's maximum and sums from somebody else.  With one tile
    # more per worker than there are CTAs its tiles walk down from the end, through second tiles of short tensors with ragged ends
    tile, sms, N = 8192, torch.cuda.get_device_properties(0).multi_processor_count, 32
    ends = [8188, 12, 4100, 4, 1064, 8192, 8, 8184, 516, 5]
    sizes = [(sms + 1 - 2 * len(ends)) * tile] + [tile + e for e in ends]
    offs = [sum(sizes[:i]) for i in range(len(sizes) + 1)]
    tiles = [-(-s // tile) for s in sizes]
    first = [sum(tiles[:i]) for i in range(len(tiles))]
    assert sum(tiles) == sms + 1
    g = torch.Generator(device=DEV).manual_seed(b)
    ld = (offs[-1] + 3) // 4 * 4
    U, S = (torch.randn((N, ld), generator=g, device=DEV)[:, :offs[-1]] for _ in range(2))
    ctx, ref = (lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, b, clip, value, 3) for _ in range(2))
    ref.set_option(lpc.OPT_ONE_LAUNCH_QUANTIZE, 0)
    want = ref.quantize_pack(U, 7, U_sub=S, seg_offsets=offs)[1]
    ref.sync_status()
    ctx.debug_one_look_stop(0)
    got = ctx.quantize_pack(U, 7, U_sub=S, seg_offsets=offs, delta_out=torch.full((N, len(sizes)), -1.0, device=DEV))[1]
    assert ctx.query(lpc.INFO_QUANT_LAUNCHES) == 1 and ctx.status() == lpc.ERR_TIMEOUT
    ragged = 0
    for i in range(N):
        for s, t0 in enumerate(first):
            mine = [t for t in range(tiles[s]) if (i * sum(tiles) + t0 + t) % sms == 0]
            if mine and mine[0] > 0:  # whoever has a message's first tile reports its scale
                ragged += s > 0
                assert got[i, s].item() == want[i, s].item(), (i, s)
    assert ragged >= 8
    ctx.close()
    ref.close()
