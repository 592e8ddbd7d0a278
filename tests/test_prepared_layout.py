"""The layout of prepared weights belongs to the library's version: a stored
buffer of another layout has the same size and passes every check, so the
version has to change with the layout.  This test restates the layout of
version 1.8 and holds the two together: whoever changes one changes the other."""
import numpy as np
import pytest

from paper_2509_26436_gb300 import _native as N
from paper_2509_26436_gb300 import build as B

VERSION = (1 << 16) | 8


def test_version_of_this_layout():
    B.build()
    assert N.load().quartz_version() == VERSION


def _align256(n):
    return -(-n // 256) * 256


@pytest.mark.gpu
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("rows,K", [(8, 64), (264, 192)])
def test_layout(mode, rows, K):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_26436_gb300 as Q

    x = np.random.default_rng(rows + mode).normal(0.3, 1, (rows, K)).astype(np.float16)
    w = Q.encode_weights(torch.from_numpy(x).cuda(), group_s=16, mode=mode)
    buf = Q.prepare_weights(w).cpu().numpy()
    G, pad = K // 64, -(-rows // 256) * 256
    at = _align256(-(-rows // 16) * 16 * K)
    side = buf[at:at + (3 if mode else 1) * G * pad * 4]
    assert len(buf) == at + _align256(len(side))
    scales = side[:G * pad * 4].view(np.float32).reshape(G, pad)
    assert np.array_equal(scales[:, :rows], w.scales.cpu().numpy().astype(np.float32).T)
    assert not scales[:, rows:].any()
    if not mode:
        return
    recs = side[G * pad * 4:].view(np.float16).reshape(G, pad, 4)
    r = np.arange(pad)
    recs = recs[:, (r & ~15) | ((r & 3) << 2) | ((r >> 2) & 3)]  # row r lies at its 4 x 4 transposed place
    z, s = w.zeros.cpu().numpy().T, w.gsum.cpu().numpy().T
    lo = np.fmod(s, 16)
    assert np.array_equal(recs[:, :rows], np.stack([z, z, s - lo, lo], axis=-1))
    assert not recs[:, rows:].any()
