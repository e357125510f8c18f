"""Which kernels a call runs on, and what it needs, at the lines between the
routes of structured plans (checked against the fp64 oracle: bf16 bar for Y and
dX, 1e-5 relative for fp32)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2608_26430_gb300 import framefb as ffb
from paper_2608_26430_gb300 import workloads as wl
from paper_2608_26430_gb300.batch import AdapterBatch
from tests.oracle_side import Expect, assert_bf16, assert_f32, host64

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
F, ALL = ffb.OP_FORWARD, ffb.OP_FORWARD | ffb.OP_BACKWARD_DX | ffb.OP_GRAD_COEFF


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_26430_gb300.build import build
    build()
    ffb.lib()


def load(mats, N, nnz, dtype="bf16", **kw):
    return wl.Workload("routes", tuple(wl.MatSpec(f"w{i}", n, m) for i, (n, m) in enumerate(mats)), N=N, nnz=nnz,
                       dtype=dtype, c_std=0.02, **kw)


def names(b, ops):
    return ffb.framefb_kernel_names(b.mats, ops, b.dtype_code)


# sides of up to 256 groups, at most 16 entries per column: whole on the fused
# tcgen05 kernels at any token count, a forward pass without a workspace
@pytest.mark.parametrize("shape", [(8192, 1024), (1024, 8192), (8192, 8192)])
@pytest.mark.parametrize("N", [5, 131])
def test_wide_sides_of_the_fused_kernels(shape, N):
    b = AdapterBatch(load([shape], N, 900), DEV, ops=ALL)
    assert names(b, F) == ["tc_tile_kernel<1>"]
    assert ffb.framefb_workspace_size(b.mats, F) == 0
    ffb.framefb_forward(b.mats, b.dtype_code, None)
    e, buf = Expect(b, 0), b.bufs[0]
    X = host64(buf.X)
    torch.cuda.synchronize()
    assert_bf16(host64(buf.Y), e.y(X, np.zeros((N, shape[1]))), what="Y")
    buf.Y.zero_()
    vals = torch.stack([buf.c_val, 2 * buf.c_val])
    m = ffb.framefb_mat.from_buffer_copy(b.mats[0])
    m.c_val = vals.data_ptr()
    ffb.framefb_forward_tenants([m], b.dtype_code, [0, 2, N], [1, 0], 2)
    torch.cuda.synchronize()
    want = e.y(X, np.zeros((N, shape[1])))
    want[:2] *= 2
    assert_bf16(host64(buf.Y), want, what="Y of tenants")


@pytest.mark.parametrize("ops", [F, ffb.OP_GRAD_COEFF])
def test_parts_of_short_columns_without_dx(ops):
    b = AdapterBatch(load([(1024, 9216)], 37, 700), DEV, ops=ops)
    assert names(b, ops) == [f"tc2_tile_kernel<{ops}>"]
    b.run(ops, b.workspace(ops))
    torch.cuda.synchronize()
    e, buf = Expect(b, 0), b.bufs[0]
    if ops == F:
        assert_bf16(host64(buf.Y), e.y(host64(buf.X), np.zeros((37, 9216))), what="Y")
    else:
        assert_bf16(host64(buf.dC), e.dc(host64(buf.X), host64(buf.dY)), what="dC")


@pytest.mark.parametrize("shape,N", [((1024, 4608), 45), ((4608, 1024), 200)])
def test_without_parts_wide_plans_run_as_contractions(shape, N, monkeypatch):
    monkeypatch.setenv("FRAMEFB_PARTS", "0")
    b = AdapterBatch(load([shape], N, 4300, support_mode=wl.ZIPF_ROWS), DEV, ops=ALL)
    assert "dense_gemm_kernel<bf16_hilo><grouped>" in names(b, ALL)
    assert all(k.startswith(("dense_", "group_block_kernel")) for k in names(b, ALL))
    b.run(ALL, b.workspace(ALL))
    torch.cuda.synchronize()
    e, buf = Expect(b, 0), b.bufs[0]
    X, dY = host64(buf.X), host64(buf.dY)
    assert_bf16(host64(buf.Y), e.y(X, np.zeros((N, shape[1]))), what="Y")
    assert_bf16(host64(buf.dX), e.dx(dY, np.zeros((N, shape[0]))), what="dX")
    assert_bf16(host64(buf.dC), e.dc(X, dY), what="dC")


# more than 32 entries per column, or the switch: the one-phase FFT kernel under
# its own name
@pytest.mark.parametrize("mats,N,nnz,kernel", [([(256, 256)], 37, 9000, ""), ([(768, 256), (256, 768)], 21, 9000, ""),
                                               ([(256, 256)] * 3, 9, 200, "tile"), ([(1024, 768)], 33, 4000, "tile")])
def test_fp32_one_phase_kernel(mats, N, nnz, kernel, monkeypatch):
    monkeypatch.setenv("FRAMEFB_KERNEL", kernel)
    b = AdapterBatch(load(mats, N, nnz, "f32"), DEV, ops=ALL)
    for ops in (F, ffb.OP_BACKWARD_DX, ffb.OP_GRAD_COEFF, ffb.OP_BACKWARD_DX | ffb.OP_GRAD_COEFF, ALL):
        assert names(b, ops) == [f"fft_phase_kernel<{ops}>"]
        for x in b.bufs:
            x.Y.zero_()
            x.dX.zero_()
            x.dC.fill_(float("nan"))
        b.run(ops, b.workspace(ops))
        torch.cuda.synchronize()
        for j, x in enumerate(b.bufs):
            e, X, dY = Expect(b, j), host64(x.X), host64(x.dY)
            if ops & F:
                assert_f32(host64(x.Y), e.y(X, np.zeros((N, x.spec.m))), what=f"Y[{j}]")
            if ops & ffb.OP_BACKWARD_DX:
                assert_f32(host64(x.dX), e.dx(dY, np.zeros((N, x.spec.n))), what=f"dX[{j}]")
            if ops & ffb.OP_GRAD_COEFF:
                assert_f32(host64(x.dC), e.dc(X, dY), what=f"dC[{j}]")
    monkeypatch.setenv("FRAMEFB_KERNEL", "")
    if nnz <= 8192:
        assert names(b, ALL) == ["fft_tile_kernel<7>"]


# fp32 plans in compacted buffers: wide sides with short columns stay on the
# one-phase kernel; long columns leave it where both gradients are asked for, or
# (8192 features and more in all) for a forward pass, or for many tokens
@pytest.mark.parametrize("shape,N,nnz,fused,forward,dx", [((8448, 64), 5, 300, "phase", "phase", "phase"),
                                                          ((256, 256), 9, 6000, "tile", "phase", "phase"),
                                                          ((4096, 4096), 5, 4608, "tile", "tile", "phase"),
                                                          ((4096, 4096), 800, 4608, "tile", "tile", "tile")])
def test_fp32_compacted_buffers(shape, N, nnz, fused, forward, dx):
    b = AdapterBatch(load([shape], N, nnz, "f32"), DEV, ops=ALL)
    for ops, kernel in ((ALL, fused), (F, forward), (ffb.OP_BACKWARD_DX, dx)):
        assert names(b, ops) == [f"fft_{kernel}_kernel<{ops}>"]
    if max(shape) > 256:
        return
    e, x = Expect(b, 0), b.bufs[0]
    X, dY = host64(x.X), host64(x.dY)
    b.run(F)
    b.run(ffb.OP_BACKWARD_DX)
    torch.cuda.synchronize()
    assert_f32(host64(x.Y), e.y(X, np.zeros((N, shape[1]))), what="Y")
    assert_f32(host64(x.dX), e.dx(dY, np.zeros((N, shape[0]))), what="dX")


def test_one_workspace_serves_fewer_tokens_of_wide_plans():
    """Wide bf16 plans run as contractions below 128 tokens (unpadded rows) or on the
    warp-MMA kernel (padded rows), fp32 ones with long columns on the one-phase kernel
    below 768: the workspace of more tokens serves them."""
    for dtype, shape, pad, Ns in (("bf16", (4608, 64), 0, (1, 64, 127, 128, 300)), ("bf16", (4608, 64), 16, (1, 64, 127, 128, 300)),
                                  ("f32", (4096, 4096), 0, (1, 100, 767, 768))):
        kw = {"support_mode": wl.ZIPF_ROWS} if dtype == "bf16" else {}
        b = AdapterBatch(load([shape], max(Ns), 4300 if dtype == "bf16" else 4608, dtype, **kw), DEV, ops=ALL)
        sizes = []
        for N in Ns:
            c = ffb.framefb_mat.from_buffer_copy(b.mats[0])
            c.N, c.ldx, c.ldy = N, c.ldx + pad, c.ldy + pad
            sizes.append(ffb.framefb_workspace_size([c], ALL if dtype == "bf16" else ffb.OP_GRAD_COEFF))
        assert sizes == sorted(sizes), (dtype, shape, pad, sizes)


def test_contractions_over_more_than_a_chunk_of_tokens():
    """T-block frames have no transform kernel: more tokens than the contraction path
    holds at a time (8192), dC summed over both chunks."""
    w = wl.WORKLOADS["tblock_tff"]
    N = 8192 + 77
    b = AdapterBatch(w, DEV, N=N, indices=[0, 1], ops=ALL)
    assert "dense_gemm_kernel<bf16_hilo>" in names(b, ALL) and not any(k.startswith("row") for k in names(b, ALL))
    b.run(ALL, b.workspace(ALL))
    torch.cuda.synchronize()
    for j, x in enumerate(b.bufs):
        e, X, dY = Expect(b, j), host64(x.X), host64(x.dY)
        assert_bf16(host64(x.Y), e.y(X, np.zeros((N, x.spec.m))), what=f"Y[{j}]")
        assert_bf16(host64(x.dX), e.dx(dY, np.zeros((N, x.spec.n))), what=f"dX[{j}]")
        assert_bf16(host64(x.dC), e.dc(X, dY), what=f"dC[{j}]")
