"""Calls queued back to back without a synchronisation: every kernel waits for
what the stream holds ahead of it, so the results are those of calls with the
device idle in between, bit for bit.  Eagerly and under capture, after copies,
memsets and work of another stream, on one shared workspace.
"""
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


# (dtype, matrices, tokens, entries, rho = 2): group, packed, two-token and row
# kernels, with grids of a few CTAs and of every SM
SHAPES = [("f32", [(256, 256)], 8, 128, False), ("f32", [(768, 768)] * 4, 700, 1000, False),
          ("bf16", [(256, 256)], 33, 200, False), ("bf16", [(768, 768)] * 6, 1500, 1000, False),
          ("bf16", [(4096, 4096)], 37, 4096, False), ("bf16", [(1024, 1024)] * 2, 301, 900, True),
          # one kernel in two launches, the second with less shared memory
          ("bf16", [(768, 768), (1024, 256)], 77, 600, False)]


def build_batch(shape):
    dtype, mats, N, nnz, rho2 = shape
    dims = sorted({d for nm in mats for d in nm})
    kw = {"frames": tuple((d, d // 2, 2) for d in dims)} if rho2 else {}
    w = wl.Workload("chain", tuple(wl.MatSpec(f"w{i}", n, m) for i, (n, m) in enumerate(mats)), N=N, nnz=nnz,
                    dtype=dtype, c_std=0.02, **kw)
    return AdapterBatch(w, DEV, ops=ALL, y_init="random")


def program(b, c, src, mom, ws, sync):
    """Copies in, two steps, an optimiser update, a second step from its values."""
    for j, buf in enumerate(b.bufs):
        for name in ("X", "dY", "Y", "dX"):
            getattr(buf, name).copy_(src[j][name])
    c.copy_(src[-1]["c"])
    mom.zero_()
    sync()
    b.run(ALL, ws)
    sync()
    for buf in b.bufs:
        ffb.framefb_adamw(buf.c_val, buf.dC, mom[0, :buf.dC.numel()], mom[1, :buf.dC.numel()], 1, 1e-3)
        sync()
    b.run(ALL, ws)
    sync()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("how", ["eager", "graph"])
def test_back_to_back(shape, how):
    b = build_batch(shape)
    c = torch.stack([buf.c_val for buf in b.bufs])
    vals = [{n: getattr(buf, n).clone() for n in ("X", "dY", "Y", "dX")} for buf in b.bufs]
    src = vals + [{"c": c.clone()}]
    keep = [buf.c_val for buf in b.bufs]
    mom = torch.zeros(2, b.bufs[0].dC.numel(), device=DEV)
    ws = b.workspace(ALL)

    class Values:  # the coefficient values back to their start
        def copy_(self, x):
            for k, v in zip(keep, x):
                k.copy_(v)

    def outputs():
        torch.cuda.synchronize()
        return [t.clone() for buf in b.bufs for t in (buf.Y, buf.dX, buf.dC, buf.c_val)]

    program(b, Values(), src, mom, ws, torch.cuda.synchronize)
    want = outputs()
    if how == "eager":
        for _ in range(20):
            program(b, Values(), src, mom, ws, lambda: None)
            assert all(torch.equal(x, y) for x, y in zip(outputs(), want))
        return
    st, side = torch.cuda.Stream(), torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    spare = torch.empty(1 << 20, device=DEV)
    with torch.cuda.graph(g, stream=st):
        side.wait_stream(st)
        with torch.cuda.stream(side):
            spare.zero_()
        program(b, Values(), src, mom, ws, lambda: None)
        st.wait_stream(side)
        b.run(ffb.OP_FORWARD, ws)  # the first launch after a join
    b.run(ffb.OP_FORWARD, ws)
    want = outputs()
    for _ in range(5):
        g.replay()
        g.replay()
        assert all(torch.equal(x, y) for x, y in zip(outputs(), want))
