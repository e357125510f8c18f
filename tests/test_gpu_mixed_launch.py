"""One launch of the group kernel over matrices of unlike cost, over plans of their
own, with fewer units than CTAs, and more matrices than one launch holds: results against the fp64 oracle (fp32 bar), and a
workspace that serves every smaller token count."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2608_26430_gb300 import framefb as ffb
from paper_2608_26430_gb300 import workloads as wl
from paper_2608_26430_gb300.batch import AdapterBatch
from tests.oracle_side import Expect, assert_f32, host64

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
ALL = ffb.OP_FORWARD | ffb.OP_BACKWARD_DX | ffb.OP_GRAD_COEFF
MIXED = [(1024, 1024)] + [(256, 256)] * 5
UNLIKE = [(256, 256), (4096, 256), (256, 256), (256, 2048)]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_26430_gb300.build import build
    build()
    ffb.lib()


def load(mats, N, nnz, **kw):
    return AdapterBatch(wl.Workload("mixed", tuple(wl.MatSpec(f"w{i}", n, m) for i, (n, m) in enumerate(mats)), N=N,
                                    nnz=nnz, dtype="f32", c_std=0.02, **kw), DEV, ops=ALL)


def first(b, N):
    out = []
    for m in b.mats:
        c = ffb.framefb_mat.from_buffer_copy(m)
        c.N = N
        out.append(c)
    return out


@pytest.mark.parametrize("mats,nnz", [(MIXED, 1000), (UNLIKE, 500)])
def test_one_workspace_serves_fewer_tokens(mats, nnz):
    b = load(mats, 700, nnz)
    sizes = [ffb.framefb_workspace_size(first(b, N), ALL) for N in range(1, 701)]
    assert sizes == sorted(sizes)
    for N in (150, 202, 203, 204, 405, 406, 407):
        ws = torch.empty(sizes[N], dtype=torch.uint8, device=DEV)  # of N + 1 tokens
        ffb.framefb_run(first(b, N), ALL, b.dtype_code, ws)
    torch.cuda.synchronize()


@pytest.mark.parametrize("mats,nnz,N,kw", [(MIXED, 1000, 203, {}), (UNLIKE, 500, 1, {}), (UNLIKE, 500, 64, {}),
                                           (UNLIKE, 500, 333, {}), ([(256, 256)] * 20, 128, 9, {"per_layer_support": True}),
                                           ([(512, 256)] * 9, 3000, 5, {"per_layer_support": True}),
                                           ([(64, 96)] * 163, 40, 3, {})])
def test_parity(mats, nnz, N, kw):
    b = load(mats, N, nnz, **kw)
    b.run(ALL, b.workspace(ALL))
    torch.cuda.synchronize()
    for j, x in enumerate(b.bufs):
        e, X, dY = Expect(b, j), host64(x.X), host64(x.dY)
        assert_f32(host64(x.Y), e.y(X, np.zeros((N, x.spec.m))), what=f"Y[{j}]")
        assert_f32(host64(x.dX), e.dx(dY, np.zeros((N, x.spec.n))), what=f"dX[{j}]")
        assert_f32(host64(x.dC), e.dc(X, dY), what=f"dC[{j}]")


def test_dc_sums_are_as_accurate_as_the_one_phase_kernels(monkeypatch):
    """dC over many tokens per CTA: no further from fp64 than the one-phase kernel's on
    the same inputs, over the entries of all matrices (both kernels sum in fp32; what
    differs is the number of roundings along a sum)."""
    err = {}
    for kernel in ("", "tile"):
        monkeypatch.setenv("FRAMEFB_KERNEL", kernel)
        b = load([(768, 768)] * 8, 2048, 1000)
        b.run(ffb.OP_GRAD_COEFF, b.workspace(ffb.OP_GRAD_COEFF))
        torch.cuda.synchronize()
        num = den = 0.0
        for j, x in enumerate(b.bufs):
            ref = Expect(b, j).dc(host64(x.X), host64(x.dY))
            num += np.sum((host64(x.dC) - ref) ** 2)
            den += np.sum(ref ** 2)
        err[kernel] = np.sqrt(num / den)
    assert err[""] <= err["tile"], err


def test_many_big_plans_fit_the_static_workspace():
    w = wl.Workload("big", tuple(wl.MatSpec(f"w{i}", 256, 4608) for i in range(110)), N=40, nnz=8192, dtype="bf16",
                    c_std=0.02, support_mode=wl.ZIPF_ROWS)
    b, ref = (AdapterBatch(w, DEV, ops=ALL, alias_inputs=True) for _ in range(2))
    assert ffb.framefb_kernel_names(b.mats, ALL, b.dtype_code) == ["fft_tile_kernel<7>"]
    ffb.framefb_run_static_ws(b.mats, ALL, b.dtype_code)
    ref.run(ALL, ref.workspace(ALL))
    torch.cuda.synchronize()
    for x, y in zip(b.bufs, ref.bufs):
        assert torch.equal(x.Y, y.Y) and torch.equal(x.dX, y.dX) and torch.equal(x.dC, y.dC)
