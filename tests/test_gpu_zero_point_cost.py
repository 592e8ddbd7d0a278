"""Zero points in the two CUDA-core GEMMs: two multiply-adds per output and
group beside the group's 64 products (SIMT) or its dot products and shifts
(SHIFT), so an asymmetric layer takes at most a quarter more than a symmetric
one (it had taken 1.38 and 1.47 times as long).  All three algorithms
give the same fp32 outputs, at ragged sizes and every subgroup size."""
import pytest

from paper_2509_26436_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_26436_gb300 as Q
    return Q


def _operands(Q, M, N, K, gs, mode):
    xa = inputs.laplace_activations(M, K, seed=M + K) + 0.05
    xw = inputs.gaussian_weights(N, K, seed=N + K)
    return [Q.quantize(torch.from_numpy(x.astype("float16")).cuda(), group_s=gs, mode=mode) for x in (xa, xw)]


@pytest.mark.parametrize("algo", ["ALGO_SIMT", "ALGO_SHIFT"])
def test_zero_points_cost_at_most_a_quarter(Q, algo):
    def gemm_us(mode):
        a, w = _operands(Q, 2001, 1600, 1152, 32, mode)
        ts = []
        for _ in range(12):
            ev = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            Q.linear(a, w, algo=getattr(Q, algo), gemm_events=ev)
            torch.cuda.synchronize()
            ts.append(ev[0].elapsed_time(ev[1]) * 1e3)
        return sorted(ts)[6]

    assert gemm_us(Q.ASYMMETRIC) < 1.25 * gemm_us(Q.SYMMETRIC)


@pytest.mark.parametrize("gs", [8, 16, 32, 64])
@pytest.mark.parametrize("M,N,K", [(1, 8, 64), (63, 72, 128), (65, 56, 192), (130, 264, 640)])
def test_algorithms_agree(Q, gs, M, N, K):
    a, w = _operands(Q, M, N, K, gs, Q.ASYMMETRIC)
    bias = torch.linspace(-1, 1, N, device="cuda").half()
    y = [Q.linear(a, w, bias, out_dtype=torch.float32, algo=al) for al in (Q.ALGO_TCGEN05, Q.ALGO_SIMT, Q.ALGO_SHIFT)]
    assert Q.device_status() == 0
    assert torch.equal(y[0], y[1]) and torch.equal(y[1], y[2])
