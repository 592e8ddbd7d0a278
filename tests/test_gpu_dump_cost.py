"""A call with a partials dump runs the group loop of every call and reads one
group a second time: its GEMM takes less than twice the GEMM without a dump
(it writes 4 bytes more per output, about a quarter of the GEMM's time here, and
re-reads 1 group of 18).  It had taken 2.5-5 times as long in a loop of its
own.  The dump also stays exact at the edges of tiles and with more tiles
than SMs: partials against the oracle, outputs against the call without it."""
import numpy as np
import pytest

import oracle as O
from paper_2509_26436_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_26436_gb300 as Q
    return Q


def _operands(Q, M, N, K, mode):
    xa = inputs.laplace_activations(M, K, seed=M + K)
    xw = inputs.gaussian_weights(N, K, seed=N + K)
    kw = dict(group_s=16, mode=mode)
    return xa, xw, Q.quantize(torch.from_numpy(xa).cuda(), **kw), Q.encode_weights(torch.from_numpy(xw).cuda(), **kw)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("out", ["float16", "float32"])
def test_dump_costs_less_than_the_gemm(Q, mode, out):
    M, N, K = 4001, 3456, 1152  # 448 whole tiles
    _, _, a, w = _operands(Q, M, N, K, mode)

    def gemm_us(**kw):
        ts = []
        for _ in range(12):
            ev = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            Q.linear(a, w, out_dtype=getattr(torch, out), gemm_events=ev, **kw)
            torch.cuda.synchronize()
            ts.append(ev[0].elapsed_time(ev[1]) * 1e3)
        return sorted(ts)[6]

    assert gemm_us(partials_group=3) < 2 * gemm_us()


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("M,N,K,g", [(1, 8, 64, 0), (129, 264, 192, 0), (127, 248, 192, 2), (2500, 2312, 320, 4),
                                     (2500, 2312, 320, 0)])
def test_dump_is_exact(Q, mode, M, N, K, g):
    xa, xw, a, w = _operands(Q, M, N, K, mode)
    y, part = Q.linear(a, w, out_dtype=torch.float32, partials_group=g)
    ref = Q.linear(a, w, out_dtype=torch.float32, algo=Q.ALGO_SIMT)
    assert Q.device_status() == 0
    assert torch.equal(y, ref)
    rows = np.unique(np.linspace(0, M - 1, 200).astype(int))
    va = O.decode_values(O.encode(xa[rows], 64, 16, mode=mode))[:, 64 * g:64 * g + 64]
    vw = O.decode_values(O.encode(xw, 64, 16, mode=mode))[:, 64 * g:64 * g + 64]
    assert np.array_equal(part[torch.from_numpy(rows).cuda()].cpu().numpy().astype(np.int64), O.group_partials(va, vw, 64)[0])
