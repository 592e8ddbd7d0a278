"""The two ways the attention step merges its splits: inside the kernel (the
splits of a head are one cluster, when all CTAs are resident at once) and by
the combine kernel.  With L in `tiles` tiles of 128 tokens, `few` heads take
`tiles` splits in a cluster; `many` heads take as many splits (fill = ceil(760
or 912 resident CTAs / many) = tiles) but more CTAs than fit at once, so the
combine kernel merges them.  Both use the same arithmetic in the same order:
the heads they share agree bit for bit."""
import pytest

from paper_2509_26436_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gs", [8, 16, 32, 64])
@pytest.mark.parametrize("tiles,few,many", [(2, 7, 600), (3, 101, 340), (4, 150, 250), (5, 152, 186)])
@pytest.mark.parametrize("out", ["float16", "bfloat16", "float32"])
def test_merges_agree(gs, tiles, few, many, out):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_26436_gb300 as Q

    L = tiles * 128 - 37
    q, k, v = (torch.from_numpy(x).cuda() for x in inputs.attention_inputs(many, L, 8200 + tiles))

    def run(heads):
        enc = [Q.quantize(x[:n].contiguous(), group_s=gs) for x, n in ((q, heads), (k, heads * L), (v, heads * L))]
        return Q.attention_decode(*enc, L, L, 128 ** -0.5, out_dtype=getattr(torch, out))

    assert torch.equal(run(few), run(many)[:few])
    assert Q.device_status() == 0
