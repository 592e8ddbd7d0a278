"""The merge inside a cluster at its larger sizes (6 to 8 splits, the portable
limit) against the oracle and, bit for bit, against the combine kernel with as
many splits.  Which form ran, and with how many splits, is read off the
workspace: the cluster form leaves it as it was, the combine form keeps its
partial results there (132 floats a head and split, the last two unused)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_2509_26436_gb300 import inputs  # noqa: E402
from test_gpu_attention import Q, _check  # noqa: E402,F401


def _run(Q, xs, heads, L, gs, out):  # noqa: F811
    q, k, v = (Q.quantize(torch.from_numpy(x[:n]).cuda(), group_s=gs)
               for x, n in zip(xs, (heads, heads * L, heads * L)))
    ws = torch.full((Q.attention_workspace_size(heads, L),), 0xA5, dtype=torch.uint8, device="cuda")
    o = Q.attention_decode(q, k, v, L, L, 128 ** -0.5, out_dtype=getattr(torch, out), workspace=ws)
    assert Q.device_status() == 0
    written = torch.nonzero(ws != 0xA5)
    splits = 0 if written.numel() == 0 else -(-(int(written.max()) + 1) // (heads * 132 * 4))
    return o, splits  # 0: merged in a cluster


@pytest.mark.parametrize("gs", [8, 16, 64])
@pytest.mark.parametrize("tiles", [6, 7, 8])
def test_cluster_merge_agrees(Q, gs, tiles):  # noqa: F811
    L, few = tiles * 128 - 37, 5
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # just more CTAs than are resident, at 5 and at 6 a SM: still `tiles` splits a head
    many = [n * sms // tiles + 1 for n in (5, 6)]
    xs = inputs.attention_inputs(max(many), L, 8600 + tiles)
    want, combined = _run(Q, xs, few, L, gs, "float32")
    assert not combined
    enc = [O.encode(x[:n], 64, gs) for x, n in zip(xs, (few, few * L, few * L))]
    _check(want.cpu().numpy(), *enc, L, L, 128 ** -0.5, "float32")
    others = [_run(Q, xs, n, L, gs, "float32") for n in many]
    assert tiles in [n for _, n in others], "no call reached the combine kernel with as many splits"
    for o, n in others:
        if n == tiles:
            assert torch.equal(o[:few], want)


def test_nine_splits_take_the_combine_kernel(Q):  # noqa: F811
    L = 9 * 128
    xs = inputs.attention_inputs(2, L, 8700)
    o, combined = _run(Q, xs, 2, L, 16, "float32")
    assert combined == 9
    _check(o.cpu().numpy(), *(O.encode(x, 64, 16) for x in xs), L, L, 128 ** -0.5, "float32")


def test_cluster_step_in_a_graph(Q):  # noqa: F811
    """Cache append, query encoding and an 8-split step, captured once and
    replayed on new inputs in the same buffers."""
    BH, L = 3, 8 * 128
    xs = [torch.from_numpy(x).cuda() for x in inputs.attention_inputs(BH, L, 8800)]
    q, k, v = (Q.quantize(x, group_s=16) for x in xs)
    new = torch.zeros(BH, 1, 128, dtype=torch.float16, device="cuda")
    ws = torch.empty(Q.attention_workspace_size(BH, L), dtype=torch.uint8, device="cuda")
    o = torch.empty(BH, 128, dtype=torch.float32, device="cuda")

    def step():
        Q.quantize(xs[0], out=q)
        Q.kv_append(new, k, L, L - 1)
        Q.attention_decode(q, k, v, L, L, 128 ** -0.5, out=o, workspace=ws)

    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        step()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            step()
    torch.cuda.synchronize()
    for seed in (1, 2):
        g = torch.Generator(device="cuda").manual_seed(seed)
        xs[0].copy_(torch.randn(BH, 128, generator=g, device="cuda"))
        new.copy_(torch.randn(BH, 1, 128, generator=g, device="cuda"))
        o.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        got = o.clone()
        step()
        assert torch.equal(o, got) and Q.device_status() == 0
