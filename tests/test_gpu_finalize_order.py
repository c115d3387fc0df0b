"""A result taken right after a graph of accumulate calls has been replayed on the default stream, with no
synchronisation in between, holds the replayed rows: the context's own stream is the one it was captured on."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")


@pytest.mark.parametrize("mode", [G.STATS_FP64, G.STATS_EXACT])
@pytest.mark.parametrize("call", ["raw", "finalize", "warm"])
def test_results_wait_for_a_replayed_graph(mode, call):
    p, n, passes = 8, 2_000_000, 8
    dtype, name = (torch.float64, G.STATS_F64) if mode == G.STATS_FP64 else (torch.int16, G.STATS_I16)
    cols = [torch.randint(0, 100, (n,), device="cuda").to(dtype) for _ in range(p)]
    with G.stats_init(G.Config([name] * p, mode)) as ctx:
        G.stats_accumulate(ctx, cols, n)  # allocations, pivot
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        G.stats_reset(ctx)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            for _ in range(passes):
                G.stats_accumulate(ctx, cols, n, stream)
        torch.cuda.synchronize()
        graph.replay()
        if call == "raw":
            raw = G.stats_raw(ctx)
            assert raw.n == passes * n
            assert np.array_equal(raw.s, [passes * float(c.double().sum()) for c in cols])
        else:
            an = G.stats_finalize(ctx) if call == "finalize" else G.stats_finalize_warm(ctx)
            assert np.abs(an.mean * n - [float(c.double().sum()) for c in cols]).max() <= 1e-6
        assert G.stats_raw(ctx).n == passes * n
