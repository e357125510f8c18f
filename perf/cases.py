"""Workloads that the framework's time is measured on.

Each case is one call of a user's program through the public entry points
(``paper_2608_26430_gb300.framefb``), on inputs that sit on the GPU, with the
frames, plans, workspace and descriptors that such a program keeps between
calls.  Shapes, token counts and support sizes are those of the repository's
workloads (``paper_2608_26430_gb300/workloads.py``) or other sizes of the same
ranges.

A case is a dict of plain values:
  kind      "step"     framefb_run over a set of matrices (ops: "fused" =
                       forward + dX + dC in one pass, "forward", "backward" =
                       dX + dC), followed by one AdamW step on all coefficient
                       values where adamw is set
            "tenants"  mixed-tenant serving forward (framefb_forward_tenants)
            "merge"    multi-tenant merge (framefb_merge)
  mats      "n x m x count" items separated by commas (in x out features)
  tokens    rows of every activation
  nnz       support size of every shape
  rho       0: frames of k = 16 subspaces (rho = d / 16); 2: rho = 2 frames
            (k = d / 2), the regime of the paper's own experiments
  zipf      rows of the support drawn from Zipf(1.1) instead of uniformly
  dtype     "bf16" or "f32" activations
  tenants   tenants of the serving and merge kinds
"""
import functools
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_2608_26430_gb300 import framefb as ffb

DEV = "cuda:0"
ALPHA = 200.0  # s = alpha / sqrt(m n)
OPS = {"forward": ffb.OP_FORWARD, "backward": ffb.OP_BACKWARD_DX | ffb.OP_GRAD_COEFF,
       "fused": ffb.OP_FORWARD | ffb.OP_BACKWARD_DX | ffb.OP_GRAD_COEFF}
ADAMW = {"lr": 1e-3, "beta1": 0.9, "beta2": 0.999, "eps": 1e-8, "weight_decay": 0.01}
FIRST_STEP = 100  # the optimiser is met in the middle of a training run


def _case(name, kind, mats, tokens, nnz, ops="fused", rho=0, zipf=False, dtype="bf16", tenants=0, adamw=False):
    c = {"name": name, "kind": kind, "mats": mats, "tokens": tokens, "nnz": nnz, "ops": ops, "rho": rho, "zipf": zipf,
         "dtype": dtype, "tenants": tenants, "adamw": adamw}
    return c


def listed():
    return [
        # the smallest call: one small fp32 layer at a handful of tokens, where launches and host time count
        _case("fp32_256_step", "step", "256x256x1", 8, 128, dtype="f32"),
        # a decode step of a served model: the q, k, v projections of one layer, one token of each of 33 sequences
        _case("llama2_decode_forward", "step", "4096x4096x3", 33, 4096, ops="forward"),
        # fine-tuning in fp32 (no mixed precision): the q and v adapters of four RoBERTa-base layers, 16 x 128 tokens
        _case("roberta_fp32_step", "step", "768x768x8", 2048, 1000, dtype="f32"),
        # RoBERTa-base q/v fine-tuning, all 12 layers in one batched call, 32 x 128 tokens
        _case("roberta_qv_step", "step", "768x768x24", 4096, 1000),
        # ViT-B/16 fine-tuning, all adapters of 12 blocks, 64 images x 197 tokens (a ragged count)
        _case("vit_b16_step", "step", "768x768x48,768x3072x12,3072x768x12", 12608, 2000),
        # serving the same model for 64 tenants, one image each, without merging
        _case("vit_b16_tenants_forward", "tenants", "768x768x48,768x3072x12,3072x768x12", 12608, 2000, ops="forward",
              tenants=64),
        # building the merged weights of 64 tenants of one projection
        _case("vit_b16_merge", "merge", "768x768x1", 0, 2000, tenants=64),
        # LLaMA-2-7B q/k/v/o training, one layer, 4 x 2048 tokens, forward and backward in one pass
        _case("llama2_layer_step", "step", "4096x4096x4", 8192, 4096),
        # the same layer as an autograd backward calls it, one ragged sequence, followed by the optimiser step
        _case("llama2_layer_backward_adamw", "step", "4096x4096x4", 2039, 4096, ops="backward", adamw=True),
        # a whole LLaMA-3-8B layer (grouped-query attention and MLP) with a heavy-tailed support, 16384 tokens
        _case("llama3_layer_step", "step", "4096x4096x2,4096x1024x2,4096x14336x2,14336x4096x1", 16384, 8192, zipf=True),
        # the paper's frame regime (rho = 2) at LLaMA-2 and RoBERTa-base shapes
        _case("llama2_rho2_step", "step", "4096x4096x4", 8192, 4096, rho=2),
        _case("roberta_rho2_step", "step", "768x768x24", 4096, 1000, rho=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: model families with their widths, any token count."""
    family = rng.choice(["small", "vit", "llama", "llama3", "rho2", "fp32", "tenants", "merge", "backward", "decode"])
    c = _case("", "step", "", 0, 0)
    del c["name"]
    if family in ("small", "vit"):
        d = rng.choice([256, 512, 768, 1024])
        wide = rng.choice([d, 3072]) if family == "vit" else d
        c.update(mats=f"{d}x{d}x{rng.randint(1, 24)}" + (f",{d}x{wide}x{rng.randint(1, 6)}" if wide != d else ""),
                 tokens=_log_int(rng, 1, 12608), nnz=_log_int(rng, 128, 2000), ops=rng.choice(["fused", "forward"]))
    elif family in ("llama", "backward", "decode"):
        c.update(mats=f"4096x{rng.choice([4096, 1024])}x{rng.randint(1, 4)}",
                 tokens=_log_int(rng, 1, 64) if family == "decode" else _log_int(rng, 64, 8192),
                 nnz=_log_int(rng, 1000, 4096),
                 ops={"llama": rng.choice(["fused", "forward"]), "backward": "backward", "decode": "forward"}[family],
                 adamw=family == "backward")
    elif family == "llama3":
        c.update(mats=rng.choice(["4096x14336x2", "14336x4096x1", "4096x1024x2", "4096x4096x1,4096x14336x1"]),
                 tokens=_log_int(rng, 64, 8192), nnz=8192, zipf=True, ops=rng.choice(["fused", "backward", "forward"]))
    elif family == "rho2":
        d = rng.choice([768, 1024, 4096])
        c.update(mats=f"{d}x{rng.choice([d, 1024])}x{rng.randint(1, 4)}", tokens=_log_int(rng, 16, 8192),
                 nnz=_log_int(rng, 500, 4096), rho=2, ops=rng.choice(["fused", "forward", "backward"]))
    elif family == "fp32":
        d = rng.choice([256, 768, 1024, 3072])
        c.update(mats=f"{d}x{rng.choice([d, 768])}x{rng.randint(1, 4)}", tokens=_log_int(rng, 1, 4096),
                 nnz=_log_int(rng, 128, 2000), dtype="f32", ops=rng.choice(["fused", "forward", "backward"]))
    elif family == "tenants":
        d = rng.choice([768, 1024, 4096])
        c.update(kind="tenants", mats=f"{d}x{d}x{rng.randint(1, 12)}", tokens=_log_int(rng, 64, 8192),
                 nnz=_log_int(rng, 500, 2000), ops="forward", tenants=rng.randint(2, 64))
    else:
        d = rng.choice([256, 768, 1024])
        c.update(kind="merge", mats=f"{d}x{rng.choice([d, 768])}x1", nnz=_log_int(rng, 128, 2000), ops="forward",
                 tenants=rng.randint(1, 64), dtype=rng.choice(["bf16", "f32"]))
    return c


# ---------------------------------------------------------------------------
# what a program keeps: frames, supports and plans, one per shape
# ---------------------------------------------------------------------------
def _k_of(case, d):
    return d // 2 if case["rho"] == 2 else 16


def _shapes(case):
    """[(n, m, count)] of the case's matrices."""
    return [tuple(int(x) for x in item.split("x")) for item in case["mats"].split(",")]


@functools.lru_cache(maxsize=None)
def _support(rows, cols, nnz, zipf):
    """nnz distinct positions of a rows x cols matrix, sorted row-major."""
    rng = np.random.default_rng(1)
    got = np.empty(0, np.int64)
    p = np.arange(1, rows + 1, dtype=np.float64) ** -1.1
    while got.size < nnz:
        r = rng.choice(rows, nnz, p=p / p.sum()) if zipf else rng.integers(0, rows, nnz)
        got = np.unique(np.concatenate([got, r.astype(np.int64) * cols + rng.integers(0, cols, nnz)]))
    got = np.sort(rng.permutation(got)[:nnz])
    return (got // cols).astype(np.int32), (got % cols).astype(np.int32)


@functools.lru_cache(maxsize=None)
def _frame(d, k):
    f = ffb.Frame(d, k, d // k)
    return f, f.to_device(DEV)


@functools.lru_cache(maxsize=None)
def _plan(n, kn, m, km, nnz, zipf):
    p = ffb.Plan(_frame(n, kn)[0], _frame(m, km)[0], *_support(m, n, nnz, zipf))
    return p, p.to_device(DEV)


def _plans(case):
    """The plan of every shape, built side by side as a program does at start-up."""
    for n, m, _ in _shapes(case):
        _frame(n, _k_of(case, n)), _frame(m, _k_of(case, m))
    keys = [(n, _k_of(case, n), m, _k_of(case, m), case["nnz"], case["zipf"]) for n, m, _ in _shapes(case)]
    with ThreadPoolExecutor(max_workers=len(keys)) as ex:
        return list(ex.map(lambda a: _plan(*a), keys))


# ---------------------------------------------------------------------------
# inputs, from the seed alone
# ---------------------------------------------------------------------------
def _type(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


def _inputs(case, seed):
    """Activations N(0, 1), coefficient values N(0, 0.02^2), and outputs that
    hold a small frozen part before the call, one batch of tensors per shape;
    segment lengths of the serving kind."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    t, N, nnz, T = _type(case), case["tokens"], case["nnz"], case["tenants"]

    def normal(*shape, std=1.0, dtype=t):
        return torch.randn(*shape, generator=g, device=DEV, dtype=dtype).mul_(std)

    f32 = torch.float32
    out = {"shape": []}
    total = sum(c for _, _, c in _shapes(case))
    if case["kind"] == "merge":
        n, m, _ = _shapes(case)[0]
        return {"W0": normal(m, n, std=0.02), "C": normal(T, nnz, std=0.02, dtype=f32)}
    if case["kind"] == "tenants":
        out["C"] = normal(total, T, nnz, std=0.02, dtype=f32)
        if N % T == 0:  # requests of one length, one per tenant
            cuts, who = [N // T * i for i in range(T + 1)], list(range(T))
        else:           # ragged requests
            r = np.random.default_rng(int(seed))
            cuts = [0] + sorted(r.integers(0, N, min(N, T) - 1).tolist()) + [N]
            who = r.integers(0, T, len(cuts) - 1).tolist()
        out["segments"] = (cuts, who)
    else:
        out["C"] = normal(total, nnz, std=0.02, dtype=f32)
    fwd, bwd = bool(OPS[case["ops"]] & ffb.OP_FORWARD), bool(OPS[case["ops"]] & ffb.OP_BACKWARD_DX)
    for n, m, c in _shapes(case):
        s = {"X": normal(c, N, n)}
        if bwd:
            s["dY"], s["dX"] = normal(c, N, m), normal(c, N, n, std=1e-3)
        if fwd:
            s["Y"] = normal(c, N, m, std=1e-3)
        out["shape"].append(s)
    if case["adamw"]:
        out["m"] = normal(total, nnz, std=1e-2, dtype=f32)
        out["v"] = normal(total, nnz, std=1e-2, dtype=f32).square_()
    return out


def _scale(n, m):
    return ALPHA / math.sqrt(m * n)


def prepare(case, seed):
    plans = _plans(case)
    s = _inputs(case, seed)
    s.update(case=case, dtype=ffb.FRAMEFB_F32 if case["dtype"] == "f32" else ffb.FRAMEFB_BF16, ops=OPS[case["ops"]])
    if case["kind"] == "merge":
        n, m, _ = _shapes(case)[0]
        s["Wout"] = torch.empty(case["tenants"], m, n, device=DEV, dtype=_type(case))
        s["fin"], s["fout"] = _frame(n, _k_of(case, n))[1], _frame(m, _k_of(case, m))[1]
        s["plan"] = plans[0]
        s["scale"] = _scale(n, m)
        return s
    if s["ops"] & ffb.OP_GRAD_COEFF:
        s["dC"] = torch.empty(s["C"].shape, device=DEV, dtype=torch.float32)
    mats, j = [], 0
    for (n, m, c), (plan, dev), t in zip(_shapes(case), plans, s["shape"]):
        for i in range(c):
            one = {k: t[k][i] for k in t}
            if "dC" in s:
                one["dC"] = s["dC"][j]
            mats.append(ffb.make_mat(_frame(n, _k_of(case, n))[1], _frame(m, _k_of(case, m))[1], plan, dev, s["C"][j],
                                     _scale(n, m), case["tokens"], ldx=n, ldy=m, **one))
            j += 1
    s["mats"] = mats
    s["ws"] = ffb.workspace(mats, s["ops"], DEV) if case["kind"] == "step" else None
    s["step"] = FIRST_STEP
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "merge":
        plan, dev = s["plan"]
        ffb.framefb_merge(s["W0"], s["fin"], s["fout"], plan, dev, s["C"], case["tenants"], s["scale"], s["Wout"])
        return {"W": s["Wout"]}
    if case["kind"] == "tenants":
        cuts, who = s["segments"]
        ffb.framefb_forward_tenants(s["mats"], s["dtype"], cuts, who, case["tenants"])
    else:
        ffb.framefb_run(s["mats"], s["ops"], s["dtype"], s["ws"])
    out = {}
    for i, t in enumerate(s["shape"]):
        out.update({f"{k}{i}": t[k] for k in ("Y", "dX") if k in t})
    if "dC" in s:
        out["dC"] = s["dC"]
    if case["adamw"]:
        ffb.framefb_adamw(s["C"], s["dC"], s["m"], s["v"], s["step"], **ADAMW)
        s["step"] += 1
        out.update(C=s["C"], m=s["m"], v=s["v"])
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    esz = 4 if case["dtype"] == "f32" else 2
    ops, N, nnz = OPS[case["ops"]], case["tokens"], case["nnz"]
    F, D, C = bool(ops & 1), bool(ops & 2), bool(ops & 4)
    total = sum(c for _, _, c in _shapes(case))

    def dft(d):  # one frame transform of one row: d / (2 k) complex DFTs of size k
        return d / 2 * 5 * math.log2(_k_of(case, d))

    if case["kind"] == "merge":
        n, m, _ = _shapes(case)[0]
        T = case["tenants"]
        # per tenant: the sparse C times the 32-wide blocks of both frames
        return {"bytes": esz * m * n * (1 + T) + 4 * nnz * (T + 2), "flops": T * (2.0 * 32 * 32 * nnz + 2.0 * m * n)}
    nbytes = flops = 0.0
    for n, m, c in _shapes(case):
        row = (n if F or C else 0) + (m if D or C else 0) + (2 * m if F else 0) + (2 * n if D else 0)
        nbytes += c * (N * row * esz + 8 * nnz + 4 * nnz * (max(1, case["tenants"]) if F or D else 0) + (4 * nnz if C else 0))
        t = (dft(n) if F or C else 0) + (dft(m) if D or C else 0) + (dft(m) if F else 0) + (dft(n) if D else 0)
        flops += c * N * (t + 2.0 * nnz * (F + D + C) + 2.0 * (m * F + n * D))
    if case["adamw"]:
        nbytes += 24.0 * total * nnz
        flops += 14.0 * total * nnz
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, from the definitions: the columns of a k * rho = d frame
# are the inverse DFT_k basis of each run of k complex coordinates, column
# i * rho + 2 r + s holding frequency i of run r, real (s = 0) or imaginary part
# ---------------------------------------------------------------------------
def _analysis(x, d, k):
    z = torch.fft.ifft(torch.view_as_complex(x.reshape(x.shape[0], d // (2 * k), k, 2)), norm="ortho", dim=-1)
    return torch.view_as_real(z.transpose(1, 2).contiguous()).reshape(x.shape[0], d)


def _synthesis(v, d, k):
    z = torch.view_as_complex(v.reshape(v.shape[0], k, d // (2 * k), 2)).transpose(1, 2)
    return torch.view_as_real(torch.fft.fft(z, norm="ortho", dim=-1).contiguous()).reshape(v.shape[0], d)


def _spmm(v, cols_in, cols_out, c, width):
    z = torch.zeros(v.shape[0], width, device=v.device, dtype=torch.float64)
    return z.index_add_(1, cols_out, v[:, cols_in] * c)


def exact(case, seed):
    s = _inputs(case, seed)
    ops = OPS[case["ops"]]
    C = s["C"].double()
    support = [tuple(torch.from_numpy(x.astype(np.int64)).to(DEV) for x in _support(m, n, case["nnz"], case["zipf"]))
               for n, m, _ in _shapes(case)]
    if case["kind"] == "merge":
        (n, m, _), (row, col) = _shapes(case)[0], support[0]
        W = torch.empty(case["tenants"], m, n, device=DEV, dtype=torch.float64)
        for t in range(case["tenants"]):
            M = torch.zeros(m, n, device=DEV, dtype=torch.float64)
            M[row, col] = C[t]
            # Phi_out C Phi_in^T: the synthesis of the rows' transform, then of the columns'
            M = _synthesis(_synthesis(M, n, 16).T.contiguous(), m, 16).T
            W[t] = s["W0"].double() + _scale(n, m) * M
        return {"W": W}
    out, j, N = {}, 0, case["tokens"]
    dC = torch.zeros(C.shape[0], case["nnz"], device=DEV, dtype=torch.float64)
    step = 2048
    for i, ((n, m, c), (row, col), t) in enumerate(zip(_shapes(case), support, s["shape"])):
        kn, km, sc = _k_of(case, n), _k_of(case, m), _scale(n, m)
        Y = torch.empty(c, N, m, device=DEV, dtype=torch.float64) if "Y" in t else None
        dX = torch.empty(c, N, n, device=DEV, dtype=torch.float64) if "dX" in t else None
        for b in range(c):
            cuts, who = s.get("segments", ([0, N], [None]))
            for t0, t1, w in zip(cuts[:-1], cuts[1:], who):
                cv = C[j] if w is None else C[j, w]
                for a in range(t0, t1, step):
                    e = min(t1, a + step)
                    V = _analysis(t["X"][b, a:e].double(), n, kn)
                    if Y is not None:
                        Y[b, a:e] = t["Y"][b, a:e].double() + sc * _synthesis(_spmm(V, col, row, cv, m), m, km)
                    if dX is not None:
                        U = _analysis(t["dY"][b, a:e].double(), m, km)
                        dX[b, a:e] = t["dX"][b, a:e].double() + sc * _synthesis(_spmm(U, row, col, cv, n), n, kn)
                        dC[j] += sc * (U[:, row] * V[:, col]).sum(0)
            j += 1
        out.update({f"{k}{i}": x for k, x in (("Y", Y), ("dX", dX)) if x is not None})
    if ops & ffb.OP_GRAD_COEFF:
        out["dC"] = dC
    if case["adamw"]:
        h = ADAMW
        p = C * (1 - h["lr"] * h["weight_decay"])
        mm = h["beta1"] * s["m"].double() + (1 - h["beta1"]) * dC
        vv = h["beta2"] * s["v"].double() + (1 - h["beta2"]) * dC * dC
        p = p - h["lr"] * (mm / (1 - h["beta1"] ** FIRST_STEP)) / ((vv / (1 - h["beta2"] ** FIRST_STEP)).sqrt() + h["eps"])
        out.update(C=p, m=mm, v=vv)
    return out
