"""GPU parity of the row-transform kernel (rho = 2 frames: one DFT of size
d / 2 per token, as fast Fourier transforms on chip) against the fp64 oracle.

Every DFT size the kernel has passes for, mixed sizes, token counts around a
token pair and a unit, every op mask, plan columns cut in halves, runs split
between columns, padded rows, an empty support.

Y and dX are held to the bf16 bar of the other GPU tests.  dC is fp32: each
transform has at most 11 butterfly levels of fp32 operations and its twiddle
powers, under 16 roundings of 2^-24 along a path, two transforms meet in a
product, so 1e-5 relative (Frobenius) bounds it.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2608_26430_gb300 import framefb as ffb
from paper_2608_26430_gb300 import workloads as wl
from paper_2608_26430_gb300.batch import AdapterBatch
from tests.oracle_side import Expect, assert_bf16, host64

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


def rho2(mats, N, nnz, **kw):
    dims = sorted({d for nm in mats for d in nm})
    return wl.Workload("rho2", tuple(wl.MatSpec(f"w{i}", n, m) for i, (n, m) in enumerate(mats)), N=N, nnz=nnz,
                       dtype="bf16", c_std=0.02, frames=tuple((d, d // 2, 2) for d in dims), **kw)


def check(b, ops):
    assert ffb.framefb_kernel_names(b.mats, ops, b.dtype_code) == [f"row_kernel<{ops}>"]
    ws = b.workspace(ops)
    b.run(ops, ws)
    torch.cuda.synchronize()
    for j, buf in enumerate(b.bufs):
        e = Expect(b, j)
        X, dY = host64(buf.X), host64(buf.dY)
        if ops & ffb.OP_FORWARD:
            assert_bf16(host64(buf.Y), e.y(X, np.zeros((b.N, buf.spec.m))), what=f"Y[{j}]")
        if ops & ffb.OP_BACKWARD_DX:
            assert_bf16(host64(buf.dX), e.dx(dY, np.zeros((b.N, buf.spec.n))), what=f"dX[{j}]")
        if ops & ffb.OP_GRAD_COEFF:
            ref = e.dc(X, dY)
            assert np.linalg.norm(host64(buf.dC) - ref) <= 1e-5 * np.linalg.norm(ref), f"dC[{j}]"


@pytest.mark.parametrize("mats,N,nnz", [
    ([(256, 256)], 1, 60), ([(256, 256)] * 3, 37, 300), ([(512, 512)], 2, 300), ([(512, 512)], 611, 2000),
    ([(768, 768)] * 2, 513, 1000), ([(768, 768)], 600, 4096), ([(1024, 1024)], 3, 1500), ([(2048, 2048)], 45, 4000),
    ([(3072, 3072)], 19, 1100), ([(4096, 4096)], 33, 4096),
    ([(768, 1024), (1024, 768), (1024, 1024)], 515, 1000), ([(4096, 1024), (1024, 4096)], 7, 2500),
    ([(768, 3072), (3072, 768)], 520, 2000), ([(256, 4096), (512, 2048), (4096, 4096), (256, 256)], 21, 900)])
def test_sizes(mats, N, nnz):
    check(AdapterBatch(rho2(mats, N, nnz), DEV, ops=ALL), ALL)


@pytest.mark.parametrize("mats,N,nnz", [([(1024, 1024)], 301, 900), ([(4096, 4096)], 10, 3000),
                                        ([(512, 4096)], 13, 1500), ([(768, 768)], 514, 1000)])
@pytest.mark.parametrize("ops", [ffb.OP_FORWARD, ffb.OP_BACKWARD_DX, ffb.OP_GRAD_COEFF,
                                 ffb.OP_BACKWARD_DX | ffb.OP_GRAD_COEFF])
def test_every_mode(ops, mats, N, nnz):
    check(AdapterBatch(rho2(mats, N, nnz), DEV, ops=ops), ops)


@pytest.mark.parametrize("d,N,nnz", [(1024, 90, 1000), (1024, 90, 4096), (4096, 21, 4096), (512, 33, 3000)])
def test_split_runs(d, N, nnz):
    """Zipf rows: runs longer than a plan column are split (overflow slots and
    fix-ups), and the halves of a column pass open runs on."""
    b = AdapterBatch(rho2([(d, d)], N, nnz, support_mode=wl.ZIPF_ROWS), DEV, ops=ALL)
    h = np.frombuffer(b.plans[(d, d)].image()[:128].tobytes(), dtype=np.int32)
    assert h[12] > 0  # fix-ups
    check(b, ALL)


def test_entry_points_agree_and_accumulate():
    w = rho2([(1024, 1024), (4096, 1024)], 61, 2000)
    a = AdapterBatch(w, DEV, ops=ALL)
    ws = a.workspace(ALL)
    a.run(ALL, ws)
    s = AdapterBatch(w, DEV, ops=ALL)
    ffb.framefb_forward(s.mats, s.dtype_code, ws)
    ffb.framefb_backward_dx(s.mats, s.dtype_code, ws)
    ffb.framefb_grad_coeff(s.mats, s.dtype_code, ws)
    torch.cuda.synchronize()
    for x, y in zip(a.bufs, s.bufs):
        assert torch.equal(x.Y, y.Y) and torch.equal(x.dX, y.dX) and torch.equal(x.dC, y.dC)
    once = [(x.Y.float(), x.dX.float()) for x in a.bufs]
    a.run(ALL, ws)
    torch.cuda.synchronize()
    for x, (y1, x1) in zip(a.bufs, once):  # one bf16 rounding of twice the delta
        torch.testing.assert_close(x.Y.float(), 2 * y1, rtol=2 ** -7, atol=1e-6)
        torch.testing.assert_close(x.dX.float(), 2 * x1, rtol=2 ** -7, atol=1e-6)


def test_padded_rows_and_empty_support():
    N, n, m, pad = 29, 1024, 512, 24
    src = AdapterBatch(rho2([(n, m)], N, 700), DEV, ops=ALL)
    bb, key = src.bufs[0], src.keys[0]

    def padded(t, d):
        p = torch.full((N, d + pad), 7.0, device=DEV, dtype=torch.bfloat16)
        p[:, :d] = 0 if t is None else t
        return p

    Xp, dYp, Yp, dXp = padded(bb.X, n), padded(bb.dY, m), padded(None, m), padded(None, n)
    dC = torch.zeros(700, device=DEV)
    mat = ffb.make_mat(src.dev_frames[n], src.dev_frames[m], src.plans[key], src.plan_dev[key], bb.c_val, bb.scale, N,
                       X=Xp, dX=dXp, dY=dYp, Y=Yp, dC=dC, ldx=n + pad, ldy=m + pad)
    assert ffb.framefb_kernel_names([mat], ALL, ffb.FRAMEFB_BF16) == ["row_kernel<7>"]
    ffb.framefb_run([mat], ALL, ffb.FRAMEFB_BF16, ffb.workspace([mat], ALL, DEV))
    src.run(ALL, src.workspace(ALL))
    torch.cuda.synchronize()
    assert torch.equal(Yp[:, :m], bb.Y) and torch.equal(dXp[:, :n], bb.dX) and torch.equal(dC, bb.dC)
    assert bool((Yp[:, m:] == 7).all()) and bool((dXp[:, n:] == 7).all())
    e = AdapterBatch(rho2([(n, m)], N, 0), DEV, ops=ALL, y_init="random")
    Y0, X0 = e.bufs[0].Y.clone(), e.bufs[0].dX.clone()
    e.run(ALL, e.workspace(ALL))
    torch.cuda.synchronize()
    assert torch.equal(e.bufs[0].Y, Y0) and torch.equal(e.bufs[0].dX, X0)


def test_workspace_covers_fewer_tokens():
    """One workspace serves calls of fewer tokens, whichever path takes them."""
    sizes = [ffb.framefb_workspace_size(AdapterBatch(rho2([(768, 768)], N, 1000), DEV, ops=ALL).mats, ALL)
             for N in (1, 511, 512, 900)]
    assert sizes == sorted(sizes)


def test_more_matrices_than_a_launch_holds():
    w = rho2([(256, 256)] * 100, 5, 100)
    b = AdapterBatch(w, DEV, ops=ALL)
    check(b, ALL)
    assert ffb.framefb_wait_timeouts() == 0
