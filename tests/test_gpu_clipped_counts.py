"""The clipped counts are those of the last step that ran, whatever was captured, replayed or run before it with another number of CTAs per
worker: a loop of eight CTAs, single steps of one, a replayed graph of them."""
import pytest
import torch

from paper_1901_08924_b200 import lpc, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _contexts(B):
    X, y, _ = synth.linear_problem(512, 1000, loss="logistic", sparsity=0.2, noise=0.1, seed=4, device=DEV)
    g = torch.Generator(device=DEV).manual_seed(4)
    x0 = 0.1 * torch.randn(1000, generator=g, device=DEV)
    both = [lpc.Context(X, y, lpc.LOGISTIC, 1e-4, 4, B, 4, lpc.CLIP_STD, 1.0, 7) for _ in range(2)]
    for a in both:
        a.set_iterate(x0)
        a.snapshot_full_grad()
        a.set_iterate(x0 + 0.01)
    return both


@pytest.mark.parametrize("B", [8, 100])  # the loops with resident and with streaming rows; a step size of zero keeps the point
def test_counts_follow_what_ran(B):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        c, ref = _contexts(B)

        def want(k):
            ref.inner_step(0.0, k)
            out = ref.get_buffer(lpc.BUF_CLIPPED)
            assert out.sum() > 0
            return out

        c.inner_step(0.0, 0)
        c.inner_steps(0.0, 0, 3)
        assert torch.equal(c.get_buffer(lpc.BUF_CLIPPED), want(2))
        graph = torch.cuda.CUDAGraph()
        c.sync_status()
        with torch.cuda.graph(graph, stream=stream):
            c.inner_steps(0.0, 10, 3)
        assert torch.equal(c.get_buffer(lpc.BUF_CLIPPED), want(2))    # captured, not run
        graph.replay()
        assert torch.equal(c.get_buffer(lpc.BUF_CLIPPED), want(12))
        c.inner_steps(0.0, 20, 3)
        assert torch.equal(c.get_buffer(lpc.BUF_CLIPPED), want(22))
        graph.replay()                                                # a step with fewer CTAs than the loop before it
        assert torch.equal(c.get_buffer(lpc.BUF_CLIPPED), want(12))
        assert c.query(lpc.INFO_LOOP_LAUNCHES) == 2
        c.set_option(lpc.OPT_PERSISTENT, 0)
        c.inner_steps(0.0, 30, 140)                                   # the library's own graph and steps behind it
        assert torch.equal(c.get_buffer(lpc.BUF_CLIPPED), want(169))
        c.sync_status()
        ref.sync_status()
        c.close()
        ref.close()
