"""Counts and replays beside the one-launch loops: the clipped counts are those of the last step whatever ran before it, and captured
steps can be replayed."""
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


def test_clipped_counts_of_a_step_after_a_loop_with_more_ctas():
    # a loop has more CTAs per worker than a single step: their counts must not stay in the sum
    X, y, x0 = _problem(512, 1000, "logistic", 4)
    for B in (4, 8):
        c, ref = (lpc.Context(X, y, lpc.LOGISTIC, 1e-4, 4, B, 4, lpc.CLIP_STD, 1.0, 7) for _ in range(2))
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


@pytest.mark.parametrize("B", [1, 8])
def test_captured_steps_replay(B):
    # both loops hand words over under tags that a replay would repeat: captured steps are plain launches
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
