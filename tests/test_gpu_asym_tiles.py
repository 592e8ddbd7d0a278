"""Asymmetric tcgen05 GEMM with more than two tiles per CTA: the record warp's
hand-over, the 4-stage operand ring, the 8 scale slots and a warp's output block
go on from one tile to the next.  Ragged rows and columns; one, two, three and
five groups (below, at and past the three groups of record copies in flight,
not multiples of the ring).  fp32 outputs equal ALGO_SIMT's bit for bit,
two-byte outputs the fp32 result rounded once, sampled rows the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2509_26436_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prepared", [False, True])
@pytest.mark.parametrize("with_bias", [False, True])
@pytest.mark.parametrize("M,N,K", [(2600, 4104, 320), (5191, 2056, 64), (5191, 2056, 128), (5191, 2056, 192)])
def test_more_tiles_than_ctas(M, N, K, with_bias, prepared):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_26436_gb300 as Q

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert -(-M // 128) * -(-N // 256) > 2 * sms
    xa = (inputs.laplace_activations(M, K, seed=M + K) + 0.03).astype(np.float16)
    xw = (inputs.gaussian_weights(N, K, seed=N + K) - 0.004).astype(np.float16)
    kw = dict(group_s=16, mode=Q.ASYMMETRIC)
    a = Q.quantize(torch.from_numpy(xa).cuda(), **kw)
    w = Q.encode_weights(torch.from_numpy(xw).cuda(), **kw)
    bias = torch.linspace(-1, 1, N, device="cuda").half() if with_bias else None
    wp = Q.prepare_weights(w) if prepared else None
    y = {dt: Q.linear(a, w, bias, out_dtype=dt, w_prepared=wp) for dt in (torch.float32, torch.float16, torch.bfloat16)}
    ref = Q.linear(a, w, bias, out_dtype=torch.float32, algo=Q.ALGO_SIMT)
    assert Q.device_status() == 0
    for dt, got in y.items():
        assert torch.equal(got, ref.to(dt)), dt
    rows = np.unique(np.linspace(0, M - 1, 6).astype(int))
    exact, rabs = O.linear(O.encode(xa[rows], 64, 16, mode=1), O.encode(xw, 64, 16, mode=1),
                           None if bias is None else bias.cpu().numpy(), with_abs=True)
    # as tests/test_gpu_linear.py: fp32 output, (G + 4) roundings of the absolute sum
    tol = 1e-5 * np.abs(exact) + (K // 64 + 4) * 2.0 ** -24 * rabs + 2.0 ** -24
    got = y[torch.float32][torch.from_numpy(rows).cuda()].cpu().numpy().astype(np.float64)
    assert (np.abs(got - exact) <= tol).all()
