"""Zero-point terms of the asymmetric tcgen05 GEMM.

The tensor core adds z_w (64 z_a - A_g) - z_a W_g to each group's sum from
fp16 records; all of it is integer and below 2^23, so the fp32 outputs equal
those of the CUDA-core kernel bit for bit.  One-sided groups take the zero
points to their ends (-128, 127) and the group sums to their largest values;
shapes: tile edges, ragged rows and columns, one group, more groups than
pipeline stages.
"""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    import paper_2509_26436_gb300 as Q
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    return Q


def _one_sided(rows, K, seed):
    """Groups of 64: all positive, all negative, constant, mixed, zero."""
    rng = np.random.default_rng(seed)
    x = rng.uniform(0.1, 8, (rows, K // 64, 64))
    kind = rng.integers(0, 5, (rows, K // 64, 1))
    x = np.where(kind == 1, -x, x)
    x = np.where(kind == 2, 7.5, x)
    x = np.where(kind == 3, x * rng.choice([-1, 1], x.shape), x)
    return np.where(kind == 4, 0, x).reshape(rows, K).astype(np.float16)


@pytest.mark.parametrize("M,N,K", [(128, 256, 64), (127, 264, 640), (129, 248, 1152), (1, 8, 192), (300, 520, 2368)])
@pytest.mark.parametrize("gs,flag_bits", [(8, 8), (16, 4), (64, 8)])
def test_asymmetric_zero_point_ends(Q, M, N, K, gs, flag_bits):
    xa, xw = _one_sided(M, K, M + K), _one_sided(N, K, N + K)
    kw = dict(group_s=gs, mode=Q.ASYMMETRIC, flag_bits=flag_bits)
    a = Q.quantize(torch.from_numpy(xa).cuda(), **kw)
    w = Q.encode_weights(torch.from_numpy(xw).cuda(), **kw)
    assert int(w.zeros.min()) == -128 and int(w.zeros.max()) >= 126
    bias = torch.linspace(-1, 1, N, device="cuda").half()
    y = Q.linear(a, w, bias, out_dtype=torch.float32)
    ref = Q.linear(a, w, bias, out_dtype=torch.float32, algo=Q.ALGO_SIMT)
    dump, part = Q.linear(a, w, bias, out_dtype=torch.float32, partials_group=K // 64 - 1)
    assert Q.device_status() == 0
    assert torch.equal(y, ref) and torch.equal(dump, ref)
    ea, ew = O.encode(xa, 64, gs, mode=1), O.encode(xw, 64, gs, mode=1)
    exact, rabs = O.linear(ea, ew, bias.cpu().numpy(), with_abs=True)
    # as tests/test_gpu_linear.py: fp32 output, (G + 4) roundings of the absolute sum
    tol = 1e-5 * np.abs(exact) + (K // 64 + 4) * 2.0 ** -24 * rabs + 2.0 ** -24
    assert (np.abs(y.cpu().numpy().astype(np.float64) - exact) <= tol).all()
