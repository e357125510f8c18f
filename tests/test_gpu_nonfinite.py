"""An infinity in one 32-coordinate group of a token reaches only what the support
connects to that group: every other group of the token's outputs, every other
token, and every dC entry of other groups are, bit for bit, those of the same call
with that group set to zero."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2608_26430_gb300 import framefb as ffb
from paper_2608_26430_gb300 import workloads as wl
from paper_2608_26430_gb300.batch import AdapterBatch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
ALL = ffb.OP_FORWARD | ffb.OP_BACKWARD_DX | ffb.OP_GRAD_COEFF


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_26430_gb300.build import build
    build()
    ffb.lib()


def group(c, d):
    """32-coordinate group of frame column c (paper order) of a k = 16 frame of dimension d."""
    return (c % (d // 16)) // 2


# columns of 4 entries (one thread each), of 10 (halves of 5), of more than 16
# (compacted buffers, halves of 9)
@pytest.mark.parametrize("dtype,n,m,nnz", [("f32", 4096, 4096, 1000), ("f32", 4096, 4096, 2560), ("f32", 4096, 4096, 4608),
                                           ("bf16", 1024, 9216, 4608)])
@pytest.mark.parametrize("g", [0, 5])
def test_infinities_stay_in_their_group(dtype, n, m, nnz, g):
    N, t = 7, 3
    w = wl.Workload("inf", (wl.MatSpec("w", n, m),), N=N, nnz=nnz, dtype=dtype, c_std=0.02)
    b = AdapterBatch(w, DEV, ops=ALL)
    buf, ws = b.bufs[0], b.workspace(ALL)
    row, col = b.supports[b.keys[0]]
    out = []
    for val in (0.0, float("inf")):
        buf.X[t, 32 * g:32 * g + 32] = 0
        buf.dY[t, 32 * g:32 * g + 32] = 0
        buf.X[t, 32 * g + 3] = val
        buf.dY[t, 32 * g + 5] = val
        buf.Y.zero_()
        buf.dX.zero_()
        b.run(ALL, ws)
        torch.cuda.synchronize()
        out.append([x.float().cpu().numpy().copy() for x in (buf.Y, buf.dX, buf.dC)])
    (y0, x0, c0), (y1, x1, c1) = out
    gr, gc = group(row, m), group(col, n)
    others = np.arange(N) != t
    assert np.array_equal(y0[others], y1[others]) and np.array_equal(x0[others], x1[others])
    for got, want, hit in ((y1, y0, set(gr[gc == g])), (x1, x0, set(gc[gr == g]))):
        apart = np.array([i for i in range(want.shape[1] // 32) if i not in hit])
        assert apart.size and hit
        a, e = got[t].reshape(-1, 32)[apart], want[t].reshape(-1, 32)[apart]
        assert np.array_equal(a, e), apart[~np.isfinite(a).all(axis=1)]
        assert not np.isfinite(got[t].reshape(-1, 32)[sorted(hit)]).all()
    apart = (gr != g) & (gc != g)
    assert np.array_equal(c1[apart], c0[apart])
