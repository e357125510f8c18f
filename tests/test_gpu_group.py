"""GPU parity of the group-transform kernel (structured frames on the CUDA
cores) against the fp64 oracle: fp32 activations, and the bf16 shapes with a
side of more than 128 groups (compacted buffers).

fp32 is held to the fp32 bar of the other GPU tests (1e-5 of the largest
reference value), bf16 outputs to the bf16 bar; dC of the bf16 shapes is summed
in fp32 from exact inputs, 1e-5 relative (Frobenius).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2608_26430_gb300 import framefb as ffb
from paper_2608_26430_gb300 import workloads as wl
from paper_2608_26430_gb300.batch import AdapterBatch
from tests.oracle_side import Expect, assert_bf16, assert_f32, host64

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


def load(mats, N, nnz, dtype="f32", **kw):
    return wl.Workload("group", tuple(wl.MatSpec(f"w{i}", n, m) for i, (n, m) in enumerate(mats)), N=N, nnz=nnz,
                       dtype=dtype, c_std=0.02, **kw)


def check(b, ops):
    assert ffb.framefb_kernel_names(b.mats, ops, b.dtype_code) == [f"fft_tile_kernel<{ops}>"]
    b.run(ops, b.workspace(ops))
    torch.cuda.synchronize()
    f32 = b.dtype_code == ffb.FRAMEFB_F32
    close = assert_f32 if f32 else assert_bf16
    for j, buf in enumerate(b.bufs):
        e = Expect(b, j)
        X, dY = host64(buf.X), host64(buf.dY)
        if ops & ffb.OP_FORWARD:
            close(host64(buf.Y), e.y(X, np.zeros((b.N, buf.spec.m))), what=f"Y[{j}]")
        if ops & ffb.OP_BACKWARD_DX:
            close(host64(buf.dX), e.dx(dY, np.zeros((b.N, buf.spec.n))), what=f"dX[{j}]")
        if ops & ffb.OP_GRAD_COEFF:
            ref = e.dc(X, dY)
            if f32:
                assert_f32(host64(buf.dC), ref, what=f"dC[{j}]")
            else:
                assert np.linalg.norm(host64(buf.dC) - ref) <= 1e-5 * np.linalg.norm(ref), f"dC[{j}]"


# columns of 1, 4, 8 (two CTAs per SM), 16 (one) and 32 entries (compacted
# buffers); group counts that are no multiple of 8; matrices of several costs
# in one launch; fewer tokens than a pair, odd counts
@pytest.mark.parametrize("mats,N,nnz", [
    ([(256, 256)], 1, 100), ([(256, 256)] * 5, 8, 1000), ([(96, 160)], 37, 300), ([(768, 768)] * 3, 611, 1000),
    ([(768, 768)], 45, 2000), ([(1024, 768)], 33, 4000), ([(3072, 768), (768, 3072)], 21, 2000),
    ([(4096, 4096)], 19, 4096), ([(512, 512)], 27, 6000), ([(4096, 256), (256, 256), (256, 2048)], 77, 500),
    ([(32, 64)], 5, 40)])
def test_fp32(mats, N, nnz):
    check(AdapterBatch(load(mats, N, nnz), DEV, ops=ALL), ALL)


@pytest.mark.parametrize("d,N,nnz", [(768, 35, 1000), (768, 35, 3000)])
def test_fp32_split_runs(d, N, nnz):
    b = AdapterBatch(load([(d, d)], N, nnz, support_mode=wl.ZIPF_ROWS), DEV, ops=ALL)
    assert np.frombuffer(b.plans[(d, d)].image()[:128].tobytes(), dtype=np.int32)[12] > 0  # fix-ups
    check(b, ALL)


@pytest.mark.parametrize("ops", [ffb.OP_FORWARD, ffb.OP_BACKWARD_DX, ffb.OP_GRAD_COEFF,
                                 ffb.OP_BACKWARD_DX | ffb.OP_GRAD_COEFF])
@pytest.mark.parametrize("dtype,mats,N,nnz", [("f32", [(768, 1024)], 23, 1500), ("bf16", [(256, 4608)], 5, 4300)])
def test_every_mode(ops, dtype, mats, N, nnz):
    kw = {} if dtype == "f32" else {"support_mode": wl.ZIPF_ROWS}
    check(AdapterBatch(load(mats, N, nnz, dtype, **kw), DEV, ops=ops), ops)


@pytest.mark.parametrize("mats,N", [([(4608, 256), (256, 4608)], 131)])
def test_bf16_wide_sides(mats, N):
    check(AdapterBatch(load(mats, N, 4300, "bf16", support_mode=wl.ZIPF_ROWS), DEV, ops=ALL), ALL)


def test_workspace_covers_fewer_tokens():
    """One workspace serves calls of fewer tokens, whichever path takes them."""
    sizes = [ffb.framefb_workspace_size(AdapterBatch(load([(4608, 256)], N, 4300, "bf16", support_mode=wl.ZIPF_ROWS), DEV,
                                                     ops=ALL).mats, ALL) for N in (3, 127, 128, 400)]
    assert sizes == sorted(sizes)


def test_entry_points_agree():
    w = load([(768, 768), (1024, 768)], 50, 1500)
    a, s = AdapterBatch(w, DEV, ops=ALL), AdapterBatch(w, DEV, ops=ALL)
    ws = a.workspace(ALL)
    a.run(ALL, ws)
    ffb.framefb_forward(s.mats, s.dtype_code, ws)
    ffb.framefb_backward_dx(s.mats, s.dtype_code, ws)
    ffb.framefb_grad_coeff(s.mats, s.dtype_code, ws)
    torch.cuda.synchronize()
    for x, y in zip(a.bufs, s.bufs):
        assert torch.equal(x.Y, y.Y) and torch.equal(x.dX, y.dX) and torch.equal(x.dC, y.dC)


@pytest.mark.parametrize("dtype,pad,off", [("f32", 4, 0), ("f32", 8, 4), ("bf16", 16, 8)])
def test_rows_on_16_byte_boundaries(dtype, pad, off):
    """Rows that start on 16- but not 32-byte boundaries, padding untouched."""
    N, n, m, nnz = (9, 256, 768, 700) if dtype == "f32" else (3, 256, 4608, 4300)
    src = AdapterBatch(load([(n, m)], N, nnz, dtype, **({} if dtype == "f32" else {"support_mode": wl.ZIPF_ROWS})), DEV,
                       ops=ALL)
    bb, key = src.bufs[0], src.keys[0]

    def padded(t, d):
        p = torch.full((N * (d + pad) + off,), 3.0, device=DEV, dtype=src.dtype)
        v = p[off:].view(N, d + pad)
        v[:, :d] = 0 if t is None else t
        return v

    Xp, dYp, Yp, dXp = padded(bb.X, n), padded(bb.dY, m), padded(None, m), padded(None, n)
    dC = torch.zeros(nnz, device=DEV)
    mat = ffb.make_mat(src.dev_frames[n], src.dev_frames[m], src.plans[key], src.plan_dev[key], bb.c_val, bb.scale, N,
                       X=Xp, dX=dXp, dY=dYp, Y=Yp, dC=dC, ldx=n + pad, ldy=m + pad)
    assert ffb.framefb_kernel_names([mat], ALL, src.dtype_code) == ["fft_tile_kernel<7>"]
    ffb.framefb_run([mat], ALL, src.dtype_code, ffb.workspace([mat], ALL, DEV))
    src.run(ALL, src.workspace(ALL))
    torch.cuda.synchronize()
    assert torch.equal(Yp[:, :m], bb.Y) and torch.equal(dXp[:, :n], bb.dX) and torch.equal(dC, bb.dC)
    assert bool((Yp[:, m:] == 3).all()) and bool((dXp[:, n:] == 3).all())
