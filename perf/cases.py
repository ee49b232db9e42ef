"""What this library is used for, as cases that can be timed.

Every case goes through the public C-ABI binding the way a user's program
calls it: arrays on the device, a workspace the library keeps (NULL), a plan
where a solver would keep one.  The matrix families are those of the
repository's workloads and selector set (27-point stencils, R-MAT graphs with
one injected long row, uniform random rows, bands, short rows with a few very
long ones, dense diagonal blocks, mixed batches), generated on the GPU.
"""
import math

import numpy as np
import torch

from paper_1504_06474_gb300 import selector
from paper_1504_06474_gb300 import ssspmv as C

DEV = "cuda"


def listed():
    return [
        # a small matrix in a tight loop: latency of one call
        {"name": "uniform4096_f64", "op": "csr", "prec": "f64", "family": "uniform", "m": 4096,
         "lo": 0, "hi": 32, "empty": 0.05},
        # the headline product: a large regular discretisation, one-shot call
        {"name": "stencil160_f64", "op": "csr", "prec": "f64", "family": "stencil", "nx": 160,
         "ny": 160, "nz": 160},
        # a power-law graph: half the rows empty, one row of 10^6 entries
        {"name": "rmat22_f64", "op": "csr", "prec": "f64", "family": "rmat", "scale": 22, "ef": 16,
         "inject": 1_000_000},
        # short rows with a few dense ones (constraints, hubs)
        {"name": "longrows_f64", "op": "csr", "prec": "f64", "family": "longrows", "m": 1_500_001,
         "nlong": 3, "longlen": 500_000},
        # single precision, an odd grid
        {"name": "stencil_f32", "op": "csr", "prec": "f32", "family": "stencil", "nx": 101,
         "ny": 97, "nz": 103},
        # single precision on a power-law graph
        {"name": "rmat20_f32", "op": "csr", "prec": "f32", "family": "rmat", "scale": 20, "ef": 16,
         "inject": 250_000},
        # stored values in bfloat16, x and y in single precision
        {"name": "stencil_bf16", "op": "csr", "prec": "bf16", "family": "stencil", "nx": 120,
         "ny": 125, "nz": 131},
        # an iterative solver's product: the plan is kept
        {"name": "banded_plan_f64", "op": "plan", "prec": "f64", "family": "banded", "m": 300_001,
         "k": 31},
        # a solver's update y = alpha A x + beta y on a mid-sized matrix
        {"name": "uniform_axpby_f64", "op": "axpby", "prec": "f64", "family": "uniform",
         "m": 120_007, "lo": 0, "hi": 40, "empty": 0.0},
        # many matrices of mixed families in one call
        {"name": "batch96_f32", "op": "batch", "count": 96, "recipe": 3, "m_lo": 1000,
         "m_hi": 200_000},
        # choosing a kernel for a new matrix: row statistics and the network
        {"name": "select_2m", "op": "select", "family": "rmat", "scale": 21, "ef": 8, "inject": 0},
        # one training step of the selector's network on its training set
        {"name": "train_2000", "op": "train", "B": 2000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_matrix(rng, families=("uniform", "stencil", "rmat", "longrows", "banded", "blockdiag")):
    nnz = _log(rng, 60_000, 100_000_000)
    f = rng.choice(families)
    if f == "stencil":
        s = (nnz / 27) ** (1 / 3)
        nx, ny = (max(3, int(s * rng.uniform(0.7, 1.4))) for _ in range(2))
        return {"family": f, "nx": nx, "ny": ny, "nz": max(3, int(nnz / 27 / (nx * ny)))}
    if f == "rmat":
        ef, nnz = rng.randint(4, 16), min(nnz, 60_000_000)
        scale = max(10, int(math.log2(nnz / ef)))
        return {"family": f, "scale": scale, "ef": ef,
                "inject": rng.choice((0, 1 << (scale - 2)))}
    if f == "longrows":
        m = max(64, int(nnz / 6))
        return {"family": f, "m": m, "nlong": rng.randint(1, 8),
                "longlen": min(m, int(nnz / 24), 2_000_000)}
    if f == "banded":
        k = rng.randint(1, 64)
        return {"family": f, "m": max(2 * k, nnz // (2 * k + 1)), "k": k}
    if f == "blockdiag":
        b = rng.randint(32, 256)
        return {"family": f, "m": max(64, int(nnz / (0.7 * b + 8))), "bmax": b}
    lo, hi = rng.choice(((0, rng.randint(2, 40)), (4, 40)))
    return {"family": f, "m": max(64, int(nnz / (0.5 * (lo + hi)))), "lo": lo, "hi": hi,
            "empty": rng.choice((0.0, 0.05))}


def draw(rng):
    op = rng.choice(("csr",) * 8 + ("plan", "plan", "axpby", "axpby", "batch", "shard", "select",
                                    "train"))
    if op == "batch":
        return {"op": op, "count": _log(rng, 8, 96), "recipe": rng.randint(1, 1_000_000),
                "m_lo": 1000, "m_hi": _log(rng, 20_000, 180_000)}
    if op == "train":
        return {"op": op, "B": _log(rng, 64, 4000)}
    c = {"op": op}
    if op == "select":
        return {**c, **_draw_matrix(rng)}
    c["prec"] = "f64" if op in ("axpby", "shard") else rng.choice(("f64", "f64", "f32", "bf16"))
    c.update(_draw_matrix(rng))
    if op == "csr" and c["prec"] == "f64":
        # the automatic choice in most programs; the selector's other classes
        # (the row-parallel one where rows have about the same length)
        even = c["family"] not in ("rmat", "longrows")
        c["variant"] = rng.choice((0,) * 6 + ((1, 2, 3) if even else (1, 2)))
    return c


# ---------------------------------------------------------------------------
# matrices on the GPU

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _sym(n, g, dtype=torch.float64):
    return torch.rand(n, generator=g, device=DEV, dtype=dtype) * 2 - 1


def _row_ptr(lens):
    rp = torch.zeros(lens.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(lens, 0, out=rp[1:])
    return rp


def _uniform_cols(lens, n, g):
    """Columns uniform in [0, n), sorted in every row."""
    rows = torch.repeat_interleave(torch.arange(lens.numel(), device=DEV), lens)
    key = rows * (1 << 32) + torch.randint(0, n, (rows.numel(),), generator=g, device=DEV)
    return (torch.sort(key).values & 0xFFFFFFFF).to(torch.int32)


def _range_cols(first, lens, rp):
    """Row r holds the columns first[r] .. first[r] + lens[r] - 1."""
    shift = torch.repeat_interleave(first - rp[:-1], lens)
    return (torch.arange(shift.numel(), device=DEV) + shift).to(torch.int32)


def _rmat_edges(scale, count, g):
    """Distinct (row, column) keys of an R-MAT graph (0.57, 0.19, 0.19, 0.05)."""
    row = torch.zeros(count, dtype=torch.int64, device=DEV)
    col = torch.zeros_like(row)
    for _ in range(scale):
        u = torch.rand(count, generator=g, device=DEV)
        row = (row << 1) | (u >= 0.76)
        col = (col << 1) | (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    return torch.unique((row << 32) | col)


def _structure(case, g):
    """(m, n, row_ptr int64, col int32) of a case's matrix."""
    f = case["family"]
    if f == "stencil":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        m = nx * ny * nz
        i = torch.arange(m, device=DEV, dtype=torch.int32)
        x, y, z = i % nx, (i // nx) % ny, i // (nx * ny)
        keep = torch.empty((m, 27), dtype=torch.bool, device=DEV)
        cols = torch.empty((m, 27), dtype=torch.int32, device=DEV)
        j = 0
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    keep[:, j] = ((z + dz >= 0) & (z + dz < nz) & (y + dy >= 0) & (y + dy < ny)
                                  & (x + dx >= 0) & (x + dx < nx))
                    cols[:, j] = i + (dz * ny + dy) * nx + dx
                    j += 1
        return m, m, _row_ptr(keep.sum(1)), cols[keep]
    if f == "rmat":
        m = 1 << case["scale"]
        key = _rmat_edges(case["scale"], case["ef"] * m, g)
        if case["inject"]:
            r = int(torch.randint(0, m, (1,), generator=g, device=DEV))
            c = torch.randperm(m, generator=g, device=DEV)[: case["inject"]]
            key = torch.cat([key[(key >> 32) < r], (r << 32) + torch.sort(c).values,
                             key[(key >> 32) > r]])
        return m, m, _row_ptr(torch.bincount(key >> 32, minlength=m)), \
            (key & 0xFFFFFFFF).to(torch.int32)
    m = case["m"]
    if f == "banded":
        r = torch.arange(m, device=DEV)
        first = (r - case["k"]).clamp(min=0)
        lens = (r + case["k"]).clamp(max=m - 1) - first + 1
        rp = _row_ptr(lens)
        return m, m, rp, _range_cols(first, lens, rp)
    if f == "blockdiag":
        sizes = torch.randint(32, case["bmax"] + 1, (m // 32 + 1,), generator=g, device=DEV)
        ends = torch.cumsum(sizes, 0).clamp(max=m)
        starts = torch.cat([ends.new_zeros(1), ends[:-1]])
        first = torch.repeat_interleave(starts, ends - starts)
        lens = torch.repeat_interleave(ends - starts, ends - starts)
        rp = _row_ptr(lens)
        return m, m, rp, _range_cols(first, lens, rp)
    if f == "longrows":
        lens = torch.randint(1, 9, (m,), generator=g, device=DEV)
        lens[torch.randperm(m, generator=g, device=DEV)[: case["nlong"]]] = case["longlen"]
    else:
        lens = torch.randint(case["lo"], case["hi"] + 1, (m,), generator=g, device=DEV)
        if case["empty"]:
            lens[torch.randperm(m, generator=g, device=DEV)[: int(case["empty"] * m)]] = 0
    return m, m, _row_ptr(lens), _uniform_cols(lens, m, g)


def _values(case, m, rp, col, g):
    """Matrix values: the stencil's are diagonally dominant, the others U[-1, 1)."""
    if case["family"] != "stencil":
        return _sym(col.numel(), g)
    val = -1.0 + 0.01 * _sym(col.numel(), g)
    rows = torch.repeat_interleave(torch.arange(m, device=DEV, dtype=torch.int32), rp.diff())
    val[rows == col] = 26.0
    return val


def _inputs(case, seed):
    g = _gen(seed)
    m, n, rp, col = _structure(case, g)
    val = _values(case, m, rp, col, g)
    x, y = _sym(n, g), _sym(m, g)
    p = case.get("prec", "f64")
    if p != "f64":
        val = val.to(torch.float32 if p == "f32" else torch.bfloat16)
        x, y = x.float(), y.float()
    return {"m": m, "n": n, "nnz": col.numel(), "rp": rp.to(torch.int32), "col": col, "val": val,
            "x": x, "y": y}


def _batch_specs(case):
    """(family, m, parameter) per matrix: banded (half-bandwidth 8..64), uniform
    rows of 4..40 entries, R-MAT (edge factor 8) clipped to m rows."""
    rng = np.random.Generator(np.random.PCG64(case["recipe"]))
    out = []
    for _ in range(case["count"]):
        f = ("banded", "uniform", "rmat")[int(rng.integers(0, 3))]
        m = int(round(math.exp(rng.uniform(math.log(case["m_lo"]), math.log(case["m_hi"])))))
        out.append((f, m, int(rng.integers(8, 65))))
    return out


def _batch_inputs(case, seed):
    g = _gen(seed)
    specs = _batch_specs(case)
    ys = torch.empty(sum(m for _, m, _ in specs), dtype=torch.float32, device=DEV)
    mats, at = [], 0
    for f, m, k in specs:
        if f == "rmat":
            scale = max(1, math.ceil(math.log2(m)))
            key = _rmat_edges(scale, 8 << scale, g)
            key = key[((key >> 32) < m) & ((key & 0xFFFFFFFF) < m)]
            rp = _row_ptr(torch.bincount(key >> 32, minlength=m))
            col = (key & 0xFFFFFFFF).to(torch.int32)
        else:
            _, _, rp, col = _structure({"family": f, "m": m, "k": k, "lo": 4, "hi": 40,
                                        "empty": 0.0}, g)
        mats.append({"m": m, "n": m, "nnz": col.numel(), "rp": rp.to(torch.int32), "col": col,
                     "val": _sym(col.numel(), g, torch.float32),
                     "x": _sym(m, g, torch.float32),
                     "y": ys[at:at + m]})
        at += m
    return mats, ys


# the selector's network: 16 features -> 64 -> 64 -> the kernel classes
F, H1, H2, K = selector.F, selector.H1, selector.H2, selector.K
ADAM = {"lr": 3e-3, "b1": 0.9, "b2": 0.999, "eps": 1e-8, "wd": 1e-4}
STEP = 100  # a step in the middle of a training run


def _train_inputs(case, seed):
    g = _gen(seed)
    B = case["B"]
    shapes = ((H1, F), (H1,), (H2, H1), (H2,), (K, H2), (K,))
    p = torch.cat([torch.randn(int(np.prod(s)), generator=g, device=DEV)
                   * (math.sqrt(2.0 / s[-1]) if len(s) == 2 else 0.1) for s in shapes])
    X = torch.rand((B, F), generator=g, device=DEV)
    T = 4.0 + 6.0 * torch.rand((B, K), generator=g, device=DEV)
    m1 = 1e-2 * torch.randn(p.numel(), generator=g, device=DEV)
    m2 = 1e-4 * (0.5 + torch.rand(p.numel(), generator=g, device=DEV))
    return {"B": B, "p": p, "X": X, "T": T, "m1": m1, "m2": m2, "shapes": shapes}


# ---------------------------------------------------------------------------

class _Plan:
    """A plan handle that goes when its owner does."""

    def __init__(self, A, val_bytes):
        self.handle = C.ssspmv_plan_create(A["m"], A["n"], A["nnz"], A["rp"], val_bytes)

    def __del__(self):
        C.ssspmv_plan_destroy(self.handle)


ALPHA, BETA = 0.75, 0.5


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        mats, ys = _batch_inputs(case, seed)
        raw = C.batch_descriptors([(A["m"], A["n"], A["nnz"], A["rp"], A["col"], A["val"], A["x"],
                                    A["y"]) for A in mats])
        total = sum(A["nnz"] for A in mats)
        ws = torch.empty(C.ssspmv_batched_workspace_bytes(len(mats), total), dtype=torch.uint8,
                         device=DEV)
        return {"op": op, "mats": mats, "ys": ys, "total": total, "ws": ws,
                "desc": torch.frombuffer(bytearray(raw), dtype=torch.uint8).to(DEV)}
    if op == "train":
        s = _train_inputs(case, seed)
        n = C.ssspmv_mlp_param_count(F, H1, H2, K)
        return {**s, "op": op, "n": n, "step": STEP,
                "scratch": torch.empty(C.ssspmv_mlp_scratch_floats(s["B"], F, H1, H2, K),
                                       device=DEV),
                "grad": torch.empty(n, device=DEV), "loss": torch.empty(1, device=DEV)}
    s = {**_inputs(case, seed), "op": op}
    if op == "select":
        return {"op": op, "m": s["m"], "n": s["n"], "nnz": s["nnz"], "rp": s["rp"],
                "params": torch.as_tensor(selector.load_default(), device=DEV),
                "feat": torch.empty(F, device=DEV),
                "fscratch": torch.empty(C.ssspmv_features_scratch_bytes(), dtype=torch.uint8,
                                        device=DEV),
                "scratch": torch.empty(C.ssspmv_mlp_scratch_floats(1, F, H1, H2, K), device=DEV),
                "cls": torch.empty(1, dtype=torch.int32, device=DEV)}
    s["prec"] = case["prec"]
    s["opts"] = C.make_opts(variant=case["variant"]) if case.get("variant") else None
    if op in ("plan", "axpby"):
        s["plan"] = _Plan(s, s["val"].element_size())
    elif op == "shard":
        # the middle one of three shards of the product
        nt = C.ssspmv_plan_shape(s["m"], s["nnz"])["ntiles"]
        s["t0"], s["t1"] = nt // 3, 2 * nt // 3
        s["r0"], s["r1"] = C.ssspmv_range_bounds(s["m"], s["nnz"], s["rp"], s["t0"], s["t1"])
        s["ws"] = torch.empty(C.ssspmv_range_workspace_bytes(s["m"], s["nnz"], s["t0"], s["t1"],
                                                             s["r0"], s["r1"]),
                              dtype=torch.uint8, device=DEV)
        s["seam"] = torch.zeros(C.SEAM_BYTES, dtype=torch.uint8, device=DEV)
    return s


def run(s):
    op = s["op"]
    if op == "csr":
        call = {"f64": C.ssspmv_csr_f64, "f32": C.ssspmv_csr_f32,
                "bf16": C.ssspmv_csr_bf16f32}[s["prec"]]
        C.check(call(s["m"], s["n"], s["nnz"], s["rp"], s["col"], s["val"], s["x"], s["y"],
                     opts=s["opts"]), "csr")
        return s["y"]
    if op == "plan":
        C.check(C.ssspmv_plan_execute(s["plan"].handle, s["col"], s["val"], s["x"], s["y"]),
                "plan_execute")
        return s["y"]
    if op == "axpby":
        C.check(C.ssspmv_plan_execute_axpby(s["plan"].handle, s["col"], s["val"], s["x"], s["y"],
                                            ALPHA, BETA), "plan_execute_axpby")
        return s["y"]
    if op == "batch":
        C.check(C.ssspmv_csr_batched_f32(len(s["mats"]), s["desc"], s["total"],
                                         workspace=s["ws"]), "batched")
        return s["ys"]
    if op == "shard":
        C.check(C.ssspmv_csr_f64_range(s["m"], s["n"], s["nnz"], s["rp"], s["col"], s["val"],
                                       s["x"], s["y"], s["t0"], s["t1"], s["r0"], s["r1"],
                                       s["seam"], workspace=s["ws"]), "range")
        return [s["y"][s["r0"]:min(s["r1"] + 1, s["m"])], s["seam"][16:].view(torch.float64)]
    if op == "select":
        C.check(C.ssspmv_features(s["m"], s["n"], s["nnz"], s["rp"], s["feat"], s["fscratch"]),
                "features")
        C.check(C.ssspmv_mlp_select(s["params"], s["feat"], 1, F, H1, H2, K, s["scratch"],
                                    s["cls"]), "select")
        return [s["feat"], s["cls"]]
    C.check(C.ssspmv_mlp_backward(s["p"], s["X"], s["T"], s["B"], F, H1, H2, K, s["scratch"],
                                  s["grad"], s["loss"]), "backward")
    C.check(C.ssspmv_mlp_adam(s["p"], s["grad"], s["m1"], s["m2"], s["n"], ADAM["lr"], ADAM["b1"],
                              ADAM["b2"], ADAM["eps"], ADAM["wd"], s["step"]), "adam")
    s["step"] += 1
    return [s["p"], s["m1"], s["m2"], s["grad"], s["loss"]]


# ---------------------------------------------------------------------------

def _below(m, scale):
    """P(a row of an R-MAT graph over 2^scale rows is below m)."""
    p, pre = 0.0, 1.0
    for b in range(scale, -1, -1):
        bit = (m >> b) & 1
        if b == scale:
            if bit:
                return 1.0
            continue
        if bit:
            p += pre * 0.76
            pre *= 0.24
        else:
            pre *= 0.76
    return p


def _size(case):
    """(m, n, nnz) of a case, random ones by expectation."""
    f = case["family"]
    if f == "stencil":
        m = case["nx"] * case["ny"] * case["nz"]
        return m, m, math.prod(3 * case[d] - 2 for d in ("nx", "ny", "nz"))
    if f == "rmat":
        m = 1 << case["scale"]
        return m, m, int(0.97 * case["ef"] * m) + case["inject"]
    m = case["m"]
    if f == "banded":
        return m, m, m * (2 * case["k"] + 1) - case["k"] * (case["k"] + 1)
    if f == "blockdiag":
        s1 = (32 + case["bmax"]) / 2
        s2 = sum(b * b for b in range(32, case["bmax"] + 1)) / (case["bmax"] - 31)
        return m, m, int(m * s2 / s1)
    if f == "longrows":
        return m, m, int(4.5 * m) + case["nlong"] * case["longlen"]
    return m, m, int(m * 0.5 * (case["lo"] + case["hi"]) * (1 - case["empty"]))


def work(case):
    op = case["op"]
    if op == "train":
        B = case["B"]
        n = H1 * F + H1 + H2 * H1 + H2 + K * H2 + K
        macs = B * (F * H1 + H1 * H2 + H2 * K)
        # forward, weight gradients and input gradients (not into X)
        return {"bytes": 4 * (B * (F + K) + 7 * n), "flops": 2 * (3 * macs - B * F * H1)}
    if op == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for f, m, k in _batch_specs(case):
            if f == "rmat":
                scale = max(1, math.ceil(math.log2(m)))
                nnz = 0.9 * (8 << scale) * _below(m, scale) ** 2
            else:
                nnz = _size({"family": f, "m": m, "k": k, "lo": 4, "hi": 40, "empty": 0.0})[2]
            total["bytes"] += 8 * nnz + 12 * m
            total["flops"] += 2 * nnz
        return total
    m, n, nnz = _size(case)
    if op == "select":
        return {"bytes": 4 * m, "flops": 2 * (F * H1 + H1 * H2 + H2 * K)}
    vb = {"f64": 8, "f32": 4, "bf16": 2}[case["prec"]]
    xb = 8 if vb == 8 else 4
    if op == "shard":
        m, nnz = m / 3, nnz / 3
    return {"bytes": nnz * (vb + 4) + 4 * (m + 1) + xb * ((2 if op == "axpby" else 1) * m + n),
            "flops": 2 * nnz}


def _product(A):
    """A x in 64 bits, row by row."""
    prod = A["val"].double() * A["x"].double()[A["col"].long()]
    return torch.segment_reduce(prod, "sum", offsets=A["rp"].long(), initial=0.0)


def _exact_train(s):
    p, X, T = s["p"].double().requires_grad_(), s["X"].double(), s["T"].double()
    parts, at = [], 0
    for sh in s["shapes"]:
        n = int(np.prod(sh))
        parts.append(p[at:at + n].view(sh))
        at += n
    W1, b1, W2, b2, W3, b3 = parts
    h = torch.relu(torch.relu(X @ W1.T + b1) @ W2.T + b2)
    loss = ((h @ W3.T + b3 - T) ** 2).mean()
    grad, = torch.autograd.grad(loss, p)
    p = p.detach()
    g = grad + ADAM["wd"] * p
    m1 = ADAM["b1"] * s["m1"].double() + (1 - ADAM["b1"]) * g
    m2 = ADAM["b2"] * s["m2"].double() + (1 - ADAM["b2"]) * g * g
    step = (m1 / (1 - ADAM["b1"] ** STEP)) / ((m2 / (1 - ADAM["b2"] ** STEP)).sqrt() + ADAM["eps"])
    return [p - ADAM["lr"] * step, m1, m2, grad, loss.detach().reshape(1)]


def _exact_features(A):
    lens = A["rp"].long().diff()
    m, nnz = A["m"], A["nnz"]
    mean = nnz / m
    a, b = lens[:-1], lens[1:]
    bins = torch.zeros_like(lens)
    for k in range(31):
        bins += lens >= (1 << k)
    cum = torch.cumsum(torch.bincount(bins.clamp(max=31), minlength=32), 0)
    pct = [float((cum < q * m).sum()) / 16 for q in (0.5, 0.9, 0.99)]
    var = float((lens.double() ** 2).sum()) / m - mean * mean

    def share(mask, of=None):
        return float(mask.sum()) / m if of is None else float(of[mask].sum()) / max(nnz, 1)

    return torch.tensor([
        math.log2(m + 1) / 24, math.log2(nnz + 1) / 32, math.log2(mean + 1) / 8,
        math.sqrt(max(var, 0.0)) / (mean + 1), math.log2(int(lens.max()) + 1) / 24,
        share(lens == 0), share(lens <= 4), share(lens.double() >= 2 * mean),
        share(lens > 1024, lens), *pct,
        share((b > 2 * a + 1) | (a > 2 * b + 1)), math.log2(480 / (mean + 1e-9) + 1) / 16,
        share((a == 0) & (b == 0)), share(lens.double() >= 32 * mean, lens)], dtype=torch.float64)


def exact(case, seed):
    op = case["op"]
    if op == "train":
        return _exact_train(_train_inputs(case, seed))
    if op == "batch":
        return torch.cat([_product(A) for A in _batch_inputs(case, seed)[0]])
    A = _inputs(case, seed)
    if op == "select":
        return [_exact_features(A), None]
    if op == "shard":
        return None  # the cut rows hold partial sums
    y = _product(A)
    return ALPHA * y + BETA * A["y"] if op == "axpby" else y
