"""STATS_FP64 of up to 12 columns: the first call's scratch serves every later one, so a larger call can be
captured into a graph after a small one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")


@pytest.mark.parametrize("p", [1, 9, 12])
@pytest.mark.parametrize("mode", [G.STATS_FP64, G.STATS_FP64_SHIFTED])
def test_larger_call_after_a_small_one_is_captured(p, mode):
    few, many = 100, 1_200_003
    g = torch.Generator(device="cuda")
    g.manual_seed(p)
    cols = [torch.randn(many, generator=g, device="cuda", dtype=torch.float64) for _ in range(p)]
    with G.stats_init(G.Config([G.STATS_F64] * p, mode)) as ctx, G.stats_init(G.Config([G.STATS_F64] * p, mode)) as ref:
        for c in (ctx, ref):
            G.stats_accumulate(c, [x[:few] for x in cols], few)
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            G.stats_accumulate(ctx, cols, many, stream)
        for _ in range(2):
            graph.replay()
            G.stats_accumulate(ref, cols, many)
        torch.cuda.synchronize()
        a, b = G.stats_raw(ctx), G.stats_raw(ref)
        assert a.n == b.n == few + 2 * many
        assert np.array_equal(a.s, b.s) and np.array_equal(a.S, b.S)
