"""attn_combine_kernel with more than 8 splits a head (few heads, long caches):
split counts at the edges of its batches of 16 and of its 32 lanes, the largest
(64), and splits of more than one tile, against the oracle with the tolerance
of test_gpu_attention.py.  One-tile splits: L in tiles of 128, few heads."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2509_26436_gb300 import inputs  # noqa: E402
from test_gpu_attention import Q, _case  # noqa: E402,F401


@pytest.mark.parametrize("gs", [8, 64])
@pytest.mark.parametrize("BH,tiles", [(1, 9), (2, 15), (1, 16), (3, 17), (2, 31), (1, 32), (2, 33), (1, 48), (1, 63),
                                      (2, 64), (1, 65), (1, 130)])
def test_more_than_8_splits(Q, gs, BH, tiles):  # noqa: F811
    L = tiles * 128 - 5
    _case(Q, BH, L + 3, L, gs, seed=8300 + tiles)


@pytest.mark.parametrize("out", ["float16", "bfloat16"])
def test_more_than_8_splits_16_bit_outputs(Q, out):  # noqa: F811
    _case(Q, 2, 3000, 2900, 16, seed=8400, out=out)


def test_merging_64_splits_costs_less_than_the_step(Q):  # noqa: F811
    """3 heads in 64 one-tile splits against 8 (merged in a cluster): the
    tiles run side by side, so what differs is the merge, a launch and at most
    as long as the step itself.  4.2-fold when every thread
    fetched the splits past the eighth one after the other."""
    def step_us(L):
        q, k, v = (Q.quantize(torch.from_numpy(x).cuda(), group_s=8) for x in inputs.attention_inputs(3, L, 8500))
        ws = torch.empty(Q.attention_workspace_size(3, L), dtype=torch.uint8, device="cuda")
        o = torch.empty(3, 128, dtype=torch.float16, device="cuda")
        stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            Q.attention_decode(q, k, v, L, L, 128 ** -0.5, out=o, workspace=ws)
            torch.cuda.synchronize()
            with torch.cuda.graph(graph, stream=stream):
                for _ in range(20):
                    Q.attention_decode(q, k, v, L, L, 128 ** -0.5, out=o, workspace=ws)
            best = float("inf")
            for _ in range(9):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                graph.replay()
                b.record(stream)
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b) * 50)
        return best

    # the step and a merge as long, one launch each: 2-fold, and half a step of slack
    assert step_us(64 * 128 - 95) < 2.5 * step_us(8 * 128 - 7)
