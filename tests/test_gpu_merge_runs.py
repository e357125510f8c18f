"""Merge where an out group's entries do not fit the stage of a CTA, or its tenants'
values do not: runs of blocks, batches of tenants, every split of the grid, against
the fp64 oracle (fp32: 1e-5 of the largest delta; bf16: the bf16 bar)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import adapter
from paper_2608_26430_gb300 import framefb as ffb
from paper_2608_26430_gb300 import workloads as wl
from tests.oracle_side import assert_bf16, frame, host64, oracle_support

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_26430_gb300.build import build
    build()
    ffb.lib()


# every position of C; one out group with most entries (Zipf rows, as in a LLaMA-3
# plan); more than a stage in every group; more out groups than resident CTAs; no
# entries; one and odd numbers of tenants
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n,m,nnz,mode,T", [
    (64, 64, 4096, wl.UNIFORM, 5), (1024, 256, 8192, wl.ZIPF_ROWS, 7), (2048, 768, 9000, wl.ZIPF_ROWS, 1),
    (256, 96, 12000, wl.UNIFORM, 3), (64, 9760, 3000, wl.UNIFORM, 2), (768, 32, 20000, wl.UNIFORM, 9),
    (288, 64, 0, wl.UNIFORM, 3), (96, 64, 700, wl.UNIFORM, 131)])
def test_runs_and_batches(n, m, nnz, mode, T, dtype):
    fin, fout = ffb.Frame(n, 16, n // 16), ffb.Frame(m, 16, m // 16)
    row, col, _, _ = ffb.framefb_support_build(m, n, nnz, 3, mode, 1.1, 16)
    orow, ocol, _, _ = oracle_support(m, n, nnz, 3, mode, 1.1, 16)
    assert np.array_equal(row, orow) and np.array_equal(col, ocol)
    plan = ffb.Plan(fin, fout, row, col)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    W0 = wl.normal((m, n), 5, 0.02, dt, DEV)
    cv = wl.normal((T, max(nnz, 1)), 6, 0.02, torch.float32, DEV)
    Wout = torch.full((T, m, n), float("nan"), device=DEV, dtype=dt)
    ffb.framefb_merge(W0, fin.to_device(DEV), fout.to_device(DEV), plan, plan.to_device(DEV), cv, T, 0.7, Wout)
    torch.cuda.synchronize()
    w0, got = host64(W0), host64(Wout)
    for t in sorted({0, T // 2, T - 1}):
        C = adapter.dense_C(m, n, row, col, host64(cv[t])[:nnz])
        ref = adapter.merge(w0, [C], frame(n, 16), frame(m, 16), 0.7)[0]
        if dtype == "f32":
            # W0 + delta rounds once to 2^-24 of the sum
            assert np.max(np.abs(got[t] - ref)) <= 1e-5 * np.max(np.abs(ref - w0)) + 2.0 ** -23 * np.max(np.abs(ref))
        else:
            assert_bf16(got[t], ref, what=f"W_{t}")
