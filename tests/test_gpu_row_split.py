"""Cut tiles of the tcgen05 GEMM with scales per row (group_q = K).

The int32 sums of a tile's parts add up exactly, so a cut changes no result:
the outputs are compared bit for bit with those of the same call with a
partials dump, which runs whole tiles, and (sampled rows) with the oracle.
Shapes: every form of the cut (equal parts, ranges over fewer tiles than SMs,
two waves, tail of a last wave), ragged M and N, group counts that leave a
remainder of the four-stage accumulation, and shapes that are not cut.
"""
import numpy as np
import pytest

import oracle as O
from paper_2509_26436_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    import paper_2509_26436_gb300 as Q
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    return Q


# M, N, K, launches at 152 SMs
SHAPES = [(2048, 1280, 11520, 3),    # 80 tiles, ranges of 95 groups
          (1999, 1272, 11584, 3),    # the same, ragged, 181 groups
          (2560, 3072, 8192, 3),     # 240 tiles, two waves
          (2560, 3072, 5120, 2),     # the same, too few groups to pay
          (1790, 3064, 3072, 3),     # 168 tiles, tail of 16 in 4 parts
          (1000, 1304, 4160, 3),     # 48 tiles in 3 parts, 65 groups
          (1, 8, 12288, 3),          # one tile in 4 parts
          (256, 320, 1152, 2),       # too few groups to pay
          (130, 264, 64, 2)]


@pytest.mark.parametrize("M,N,K,launches", SHAPES)
@pytest.mark.parametrize("out_dtype", ["float16", "bfloat16", "float32"])
def test_per_row_cut_tiles(Q, M, N, K, launches, out_dtype):
    dt = getattr(torch, out_dtype)
    xa = inputs.laplace_activations(M, K, seed=M + K)
    xw = inputs.gaussian_weights(N, K, seed=N + K)
    bias = torch.from_numpy(np.random.default_rng(3).normal(0, 0.1, N).astype(np.float16)).cuda()
    a = Q.quantize(torch.from_numpy(xa).cuda(), group_s=16, group_q=K)
    w = Q.encode_weights(torch.from_numpy(xw).cuda(), group_s=16, group_q=K)
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert Q.linear_launch_count(M, N, K, Q.Params(K, 16)) == launches
    y = Q.linear(a, w, bias, out_dtype=dt)
    whole, part = Q.linear(a, w, bias, out_dtype=dt, partials_group=0)
    assert Q.device_status() == 0
    assert torch.equal(y, whole)
    if out_dtype == "float32":
        rows = np.unique(np.linspace(0, M - 1, 4).astype(int))
        va, vw = O.decode_values(O.encode(xa[rows], K, 16)), O.decode_values(O.encode(xw, K, 16))
        P = O.group_partials(va, vw, K)[0]
        assert np.array_equal(part[torch.from_numpy(rows).cuda()].cpu().numpy().astype(np.int64), P)
