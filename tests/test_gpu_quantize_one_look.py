"""Many tensors with a subtrahend in one launch that reads both inputs once: bit for bit what the three launches give, and the oracle's for
sampled workers, on either side of the lines of the rule, with ragged, tiny, empty and all-zero tensors, every clip rule and kind of width,
twice in a row, in a replayed graph, beside another kernel that holds part of the chip, and with values that are not finite."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_1901_08924_b200 import lpc, synth

pytestmark = pytest.mark.gpu
TILE, DEV = 8192, "cuda"
PROPS = torch.cuda.get_device_properties(0) if torch.cuda.is_available() else None
SMS, L2 = (PROPS.multi_processor_count, PROPS.L2_cache_size) if PROPS else (148, 132644864)
FROM = L2 // 4 * 3 // 4  # values of each input
# whole tiles, an empty tensor, short ones and ragged ends; three of them all zero
ODD = [0, 4, 4, 1000, 1064, 2 * TILE, 2 * TILE + 12, 100 * TILE, 100 * TILE + TILE - 4, 300 * TILE, 2500000]


def _inputs(N, length, offs, seed, pad=0):
    g = torch.Generator(device=DEV).manual_seed(seed)
    ld = (length + 3) // 4 * 4 + pad
    U, S = (torch.randn((N, ld), generator=g, device=DEV)[:, :length] for _ in range(2))
    if offs is not None:
        for s in (2, 5, 8):
            if s + 1 < len(offs):
                U[1, offs[s]:offs[s + 1]] = S[1, offs[s]:offs[s + 1]]
    return U, S


def _call(N, b, clip, value, seed, k, U, S, offs, one, want):
    ctx = lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, b, clip, value, seed)
    ctx.set_option(lpc.OPT_ONE_LAUNCH_QUANTIZE, one)
    for kk in (k + 1, k):  # nothing of one call leaks into the next
        out = ctx.quantize_pack(U, kk, U_sub=S, seg_offsets=offs)
    ctx.sync_status()
    assert ctx.query(lpc.INFO_QUANT_LAUNCHES) == want
    out = [t.clone() for t in out]
    ctx.close()
    return out


def _same(a, b):
    assert all(torch.equal(x.view(torch.int32), y.view(torch.int32)) for x, y in zip(a, b))


def _against_oracle(out, U, S, offs, b, clip, value, seed, k, workers):
    codes, delta, clipped = out
    length = U.shape[1]
    offs = [0, length] if offs is None else offs
    woff, _ = lpc.packed_layout(length, b, offs)
    for i in workers:
        u, words, block = (U[i] - S[i]).cpu().numpy(), codes[i].cpu().numpy().view(np.uint32), 0
        for s, (lo, hi) in enumerate(zip(offs, offs[1:])):
            if hi > lo:
                w, dl, cl = orc.quantize_pack(np.ascontiguousarray(u[lo:hi]), b, clip, value, seed, i, k, block_base=block)
                assert (words[woff[s]:woff[s] + orc.packed_words(hi - lo, b)] == w).all(), (i, s)
                assert delta[i, s].item() == dl and int(clipped[i, s]) == cl, (i, s)
            else:
                assert delta[i, s].item() == 0 and int(clipped[i, s]) == 0
            block += (hi - lo + 7) // 8


@pytest.mark.parametrize("b,clip,value", [(1, 2, 1.5), (2, 1, 0.5), (3, 0, 1.0), (4, 2, 2.0), (5, 1, 0.25), (8, 2, 3.0), (9, 0, 1.0),
                                          (12, 2, 2.0), (16, 2, 1.0)])
def test_odd_tensors_every_width_and_clip_rule(b, clip, value):
    N, seed, k = 16, 11, 5
    U, S = _inputs(N, ODD[-1], ODD, b, pad=4)
    got = _call(N, b, clip, value, seed, k, U, S, ODD, 1, 1)
    _same(got, _call(N, b, clip, value, seed, k, U, S, ODD, 0, 3))
    _against_oracle(got, U, S, ODD, b, clip, value, seed, k, (1, N - 1))


@pytest.mark.parametrize("N,length,offs,shift,launches", [
    (12, FROM // 12 // 4 * 4, None, 0, 3),                          # the last size that is left to three launches
    (12, FROM // 12 // 4 * 4 + 4, None, 0, 1),
    (12, FROM // 12 // 4 * 4 + 7, None, 0, 1),                      # a ragged end of three values
    (13, 2 * SMS * TILE, None, 0, 1),                               # the longest message
    (13, 2 * SMS * TILE + 1, None, 0, 3),
    (13, 2 * SMS * TILE, None, 1, 3),                               # off 16-byte boundaries
    (13, 2 * SMS * TILE, [0, 6, 2 * SMS * TILE], 0, 3),             # a tensor off them
    (13, 2 * SMS * TILE, [0, 8, 2 * SMS * TILE], 0, 1),
    (16, 300 * 12000, list(range(0, 300 * 12000 + 1, 12000)), 0, 3),  # tiles three quarters full
    (16, 150 * 15000, list(range(0, 150 * 15000 + 1, 15000)), 0, 1),  # and full to 92 %
])
def test_lines_of_the_rule(N, length, offs, shift, launches):
    b, seed, k = 4, 3, 9
    U, S = _inputs(N, length + shift, None, N, pad=4)
    U, S = U[:, shift:], S[:, shift:]
    got = _call(N, b, lpc.CLIP_STD, 2.0, seed, k, U, S, offs, 1, launches)
    _same(got, _call(N, b, lpc.CLIP_STD, 2.0, seed, k, U, S, offs, 0, 3))


def test_many_small_tensors_of_few_workers_and_one_worker():
    # one or two workers: consecutive tiles of a CTA often belong to the same tensor
    for N, count in ((1, 130), (2, 70)):
        ln = 26 * TILE - 8
        offs = [i * ln for i in range(count + 1)]
        U, S = _inputs(N, offs[-1], None, 5)
        got = _call(N, 2, lpc.CLIP_STD, 2.5, 1, 2, U, S, offs, 1, 1)
        _same(got, _call(N, 2, lpc.CLIP_STD, 2.5, 1, 2, U, S, offs, 0, 3))


def test_replayed_graph_and_status():
    N, b, offs = 8, 4, synth.segment_offsets(synth.resnet18_shapes())
    U, S = _inputs(N, offs[-1], None, 2)
    ctx = lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, b, lpc.CLIP_STD, 2.5, 4)
    ref = [t.clone() for t in ctx.quantize_pack(U, 3, U_sub=S, seg_offsets=offs)]
    ctx.sync_status()
    ctx.close()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, b, lpc.CLIP_STD, 2.5, 4)
        out = ctx.quantize_pack(U, 1, U_sub=S, seg_offsets=offs)  # the scratch is made here
        ctx.sync_status()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            ctx.quantize_pack(U, 3, U_sub=S, seg_offsets=offs, codes_out=out[0], delta_out=out[1], clipped_out=out[2])
        for _ in range(3):
            for t in out:
                t.fill_(-1)
            V = U.clone()
            U.mul_(1.5)  # other values in between: nothing of a replay may be taken for the next one's
            graph.replay()
            U.copy_(V)
            graph.replay()
        ctx.sync_status()
        _same(out, ref)
        for bad in (float("nan"), float("inf")):
            V = U.clone()
            V[3, offs[20] + 5] = bad
            codes, delta, _ = ctx.quantize_pack(V, 3, U_sub=S, seg_offsets=offs)
            assert ctx.status() == lpc.ERR_NONFINITE and ctx.status() == lpc.OK
            assert torch.isnan(delta[3, 20]) and torch.isnan(delta).sum() == 1
            keep = torch.ones_like(delta, dtype=torch.bool)
            keep[3, 20] = False
            assert torch.equal(delta[keep], ref[1][keep])
        ctx.close()


def test_beside_a_kernel_that_holds_part_of_the_chip():
    # a training loop on another stream takes 64 SMs and their shared memory for some milliseconds: the launch's other CTAs cannot start
    # before it ends, and those that run look at the missing tiles themselves
    n, d, m = 16 * 512, 4096, 1500
    X, y, _ = synth.linear_problem(n, d, loss="least_squares", seed=1, device=DEV)
    N, offs = 16, list(range(0, 2000001, 250000))
    U, S = _inputs(N, offs[-1], None, 6)
    ref = _call(N, 4, lpc.CLIP_STD, 2.0, 1, 2, U, S, offs, 0, 3)
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(one):
        loop = lpc.Context(X, y, lpc.LEAST_SQUARES, 1e-4, 16, 8, 4, lpc.CLIP_STD, 3.0, 0)
        loop.snapshot_full_grad()
        loop.inner_steps(1e-3, 0, 16)
        loop.sync_status()
    with torch.cuda.stream(two):
        ctx = lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, 4, lpc.CLIP_STD, 2.0, 1)
        out = ctx.quantize_pack(U, 1, U_sub=S, seg_offsets=offs)
        ctx.sync_status()
    with torch.cuda.stream(one):
        loop.inner_steps(1e-3, 16, m)
    with torch.cuda.stream(two):
        ctx.quantize_pack(U, 2, U_sub=S, seg_offsets=offs, codes_out=out[0], delta_out=out[1], clipped_out=out[2])
        ctx.sync_status()
        assert ctx.query(lpc.INFO_QUANT_LAUNCHES) == 1
        _same(out, ref)
        ctx.close()
    with torch.cuda.stream(one):
        loop.sync_status()
        loop.close()
