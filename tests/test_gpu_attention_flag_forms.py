"""The FLAG forms of the attention step's operands (one byte or 4 bits per
subgroup), each on its own: the caches may differ, and the query may differ
from both.  The form changes how a FLAG is stored, not its value, so every
combination gives the same output, bit for bit, as byte FLAGs throughout.
Sizes: one token, a full tile, one past it, several tiles per split."""
import itertools

import pytest

from paper_2509_26436_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gs", [8, 16, 32, 64])
@pytest.mark.parametrize("BH,L_max,L", [(3, 2, 1), (2, 128, 128), (5, 140, 129), (2, 1500, 1411)])
def test_flag_forms_agree(gs, BH, L_max, L):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_26436_gb300 as Q

    xs = [torch.from_numpy(x).cuda() for x in inputs.attention_inputs(BH, L_max, 8100 + L)]
    enc = {fb: [Q.quantize(x, group_s=gs, flag_bits=fb) for x in xs] for fb in (8, 4)}
    want = Q.attention_decode(*enc[8], L_max, L, 128 ** -0.5, out_dtype=torch.float32)
    for fq, fk, fv in itertools.product((8, 4), repeat=3):
        got = Q.attention_decode(enc[fq][0], enc[fk][1], enc[fv][2], L_max, L, 128 ** -0.5, out_dtype=torch.float32)
        assert torch.equal(got, want), (fq, fk, fv)
    assert Q.device_status() == 0
