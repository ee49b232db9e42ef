"""The automatic choice (no options: products by blocks of rows) at the sizes
where it can go wrong: group and copy edges, ragged ends of the arrays, every
number of lanes per row, groups too uneven for a lane per row, groups too
large to stage, rows cut into pieces, empty rows everywhere.  Small integers,
so every sum is exact in any order and y must equal the oracle's row loop;
one structure of each kind also with real values against 1e-13 * sum|a x|."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1504_06474_gb300 import _build
    _build.build()
    return torch.device("cuda:0")


def _lens(kind, m, rng):
    if kind.startswith("const"):
        return np.full(m, int(kind[5:]))
    if kind.startswith("upto"):
        return rng.integers(0, int(kind[4:]) + 1, size=m)
    if kind == "empty":
        return np.zeros(m, np.int64)
    lens = rng.integers(0, 9, size=m) * (rng.random(m) < 0.5)
    if kind == "uneven":      # a few rows of hundreds among short ones
        lens[rng.random(m) < 0.05] = 300
    elif kind == "oversized":  # groups past the staging buffer, rows short of a piece
        lens[rng.random(m) < 0.03] = 1500
        lens[m // 2: m // 2 + 20] = 1100
    elif kind == "pieces":    # rows of one to many pieces, at their edges
        at = rng.choice(m, size=min(m, 8), replace=False)
        lens[at] = np.array([2047, 2048, 2049, 4096, 4097, 12000, 20000, 70001])[: at.size]
    else:                     # "power": row lengths falling by powers
        lens = np.minimum((2.0 / (rng.random(m) + 1e-4)).astype(np.int64), 9000)
        lens[rng.random(m) < 0.4] = 0
    return lens


KINDS = ["const1", "const8", "const16", "const27", "const28", "const31", "const60", "const64",
         "const120", "const250", "const500", "const1100", "upto4", "upto12", "upto40", "upto200",
         "empty", "uneven", "oversized", "pieces", "power"]


def _matrix(kind, m, n, seed, integers=True):
    rng = np.random.default_rng(seed)
    rp = np.zeros(m + 1, np.int64)
    np.cumsum(_lens(kind, m, rng), out=rp[1:])
    nnz = int(rp[-1])
    col = rng.integers(0, n, size=nnz).astype(np.int32)
    if integers:
        val = rng.integers(-6, 7, size=nnz).astype(float)
        x = rng.integers(-6, 7, size=n).astype(float)
    else:
        val, x = rng.uniform(-1, 1, nnz), rng.uniform(-1, 1, n)
    return rp.astype(np.int32), col, val, x


def _device(dev, arrays):
    return [torch.as_tensor(a, device=dev) for a in arrays]


@pytest.mark.parametrize("kind", KINDS)
def test_f64_equals_the_row_loop(dev, kind):
    from paper_1504_06474_gb300 import ssspmv as C
    for m in (1, 31, 33, 1000, 9001) + ((800_003,) if kind in ("upto4", "empty", "power") else ()):
        if kind == "const1100" and m > 1000:
            continue
        rp, col, val, x = _matrix(kind, m, 517, seed=m)
        nnz, want = int(rp[-1]), oracle.spmv(rp, col, val, x)
        rpd, cd, vd, xd = _device(dev, (rp, col, val, x))
        # the library's workspace, a caller's (full of ones), and a plan, twice each
        ws = torch.full((C.ssspmv_workspace_bytes(m, nnz, 8, None),), 255, dtype=torch.uint8,
                        device=dev)
        plan = C.ssspmv_plan_create(m, 517, nnz, rpd, 8)
        try:
            for call in range(6):
                y = torch.full((m,), float("nan"), dtype=torch.float64, device=dev)
                if call < 4:
                    rc = C.ssspmv_csr_f64(m, 517, nnz, rpd, cd, vd, xd, y,
                                          workspace=None if call < 2 else ws)
                else:
                    rc = C.ssspmv_plan_execute(plan, cd, vd, xd, y)
                C.check(rc, "call %d" % call)
                assert np.array_equal(y.cpu().numpy(), want), (kind, m, call)
            assert C.ssspmv_device_status(ws) == 0
            # y = 2 A x - 3 y
            C.check(C.ssspmv_plan_execute_axpby(plan, cd, vd, xd, y, 2.0, -3.0), "axpby")
            assert np.array_equal(y.cpu().numpy(), -want), (kind, m)
        finally:
            C.ssspmv_plan_destroy(plan)


@pytest.mark.parametrize("kind", ["upto40", "const64", "uneven", "oversized", "pieces", "power"])
def test_f64_rounding(dev, kind):
    from paper_1504_06474_gb300 import ssspmv as C
    m, n = 20_011, 4001
    rp, col, val, x = _matrix(kind, m, n, seed=5, integers=False)
    rpd, cd, vd, xd = _device(dev, (rp, col, val, x))
    y = torch.full((m,), float("nan"), dtype=torch.float64, device=dev)
    C.check(C.ssspmv_csr_f64(m, n, int(rp[-1]), rpd, cd, vd, xd, y), "csr")
    yref, s = oracle.spmv_dot2(rp, col, val, x)
    assert np.all(np.abs(y.cpu().numpy() - yref) <= 1e-13 * s)


@pytest.mark.parametrize("m", [8191, 8192, 8193, 8400])
def test_units_by_turns_and_by_ticket(dev, m):
    """One row per unit, on both sides of where a grid-wide ticket hands them
    out, several calls in one workspace (the ticket starts from zero again)."""
    from paper_1504_06474_gb300 import ssspmv as C
    rp, col, val, x = _matrix("const440", m, 997, seed=m)
    nnz, want = int(rp[-1]), oracle.spmv(rp, col, val, x)
    rpd, cd, vd, xd = _device(dev, (rp, col, val, x))
    for _ in range(3):
        y = torch.full((m,), -1.0, dtype=torch.float64, device=dev)
        C.check(C.ssspmv_csr_f64(m, 997, nnz, rpd, cd, vd, xd, y), "csr")
        np.testing.assert_array_equal(y.cpu().numpy(), want)


@pytest.mark.parametrize("prec", ["f32", "bf16"])
@pytest.mark.parametrize("kind", KINDS)
def test_reduced_precision_equals_the_row_loop(dev, kind, prec):
    # every product and sum is an integer below 2^24: exact in FP32 too
    from paper_1504_06474_gb300 import ssspmv as C
    for m in (33, 1000, 9001):
        if kind == "const1100" and m > 1000:
            continue
        rp, col, val, x = _matrix(kind, m, 517, seed=m + 1)
        nnz, want = int(rp[-1]), oracle.spmv(rp, col, val, x)
        vt = torch.float32 if prec == "f32" else torch.bfloat16
        rpd, cd = _device(dev, (rp, col))
        vd = torch.as_tensor(val, device=dev).to(vt)
        xd = torch.as_tensor(x, device=dev).float()
        fn = C.ssspmv_csr_f32 if prec == "f32" else C.ssspmv_csr_bf16f32
        if prec == "bf16":
            vd = vd.view(torch.int16)
        y = torch.full((m,), float("nan"), dtype=torch.float32, device=dev)
        C.check(fn(m, 517, nnz, rpd, cd, vd, xd, y), prec)
        assert np.array_equal(y.cpu().numpy().astype(np.float64), want), (kind, m)


def test_batch_of_every_kind(dev):
    from paper_1504_06474_gb300 import ssspmv as C
    keep, descs, wants, ys = [], [], [], []
    for i, kind in enumerate(KINDS * 2):
        m = (1, 33, 700, 5000)[i % 4]
        rp, col, val, x = _matrix(kind, m, 517, seed=100 + i)
        rpd, cd = _device(dev, (rp, col))
        vd, xd = (torch.as_tensor(a, device=dev).float() for a in (val, x))
        y = torch.full((m,), float("nan"), dtype=torch.float32, device=dev)
        keep.append((rpd, cd, vd, xd))
        descs.append((m, 517, int(rp[-1]), rpd, cd, vd, xd, y))
        wants.append(oracle.spmv(rp, col, val, x))
        ys.append(y)
    total = sum(d[2] for d in descs)
    desc = torch.frombuffer(bytearray(C.batch_descriptors(descs)), dtype=torch.uint8).to(dev)
    ws = torch.full((C.ssspmv_batched_workspace_bytes(len(descs), total),), 255,
                    dtype=torch.uint8, device=dev)
    for _ in range(2):
        C.check(C.ssspmv_csr_batched_f32(len(descs), desc, total, workspace=ws), "batched")
        assert C.ssspmv_device_status(ws) == 0
        for y, want in zip(ys, wants):
            assert np.array_equal(y.cpu().numpy().astype(np.float64), want)
            y.fill_(float("nan"))


def test_shown_workspace_may_be_written(dev):
    """The library's own workspace serves calls without one, whatever a caller
    that asked for its address left in it (here a batch by tiles, whose header
    counts dirty tiles where the row blocks count their lists)."""
    from paper_1504_06474_gb300 import ssspmv as C
    st = torch.cuda.Stream(dev)
    m = 5000
    rp, col, val, x = _matrix("uneven", m, 517, seed=9)
    rpd, cd, vd, xd = _device(dev, (rp, col, val, x))
    y = torch.empty(m, dtype=torch.float64, device=dev)
    rq, colq, valq, xq = _matrix("oversized", m, 517, seed=10)
    arrays = _device(dev, (rq, colq, valq, xq))
    want = oracle.spmv(rq, colq, valq, xq)
    y32, v32, x32 = torch.empty(m, device=dev), vd.float(), xd.float()
    desc = torch.frombuffer(bytearray(C.batch_descriptors(
        [(m, 517, int(rp[-1]), rpd, cd, v32, x32, y32)])), dtype=torch.uint8).to(dev)
    opts = C.make_opts(W=15, variant=C.VARIANT_SPECULATIVE)
    torch.cuda.synchronize()
    C.check(C.ssspmv_csr_f64(m, 517, int(rp[-1]), rpd, cd, vd, xd, y, stream=st), "csr")
    need = C.ssspmv_batched_workspace_bytes(1, int(rp[-1]), opts=opts)
    big = np.arange(0, 2_000_001, 4, dtype=np.int32)  # a matrix that grows it enough
    bm, bz = big.size - 1, int(big[-1])
    grow = (torch.as_tensor(big, device=dev), torch.zeros(bz, dtype=torch.int32, device=dev),
            torch.zeros(bz, dtype=torch.float64, device=dev), xd,
            torch.empty(bm, dtype=torch.float64, device=dev))
    torch.cuda.synchronize()
    C.check(C.ssspmv_csr_f64(bm, 517, bz, *grow, stream=st), "grow")
    ptr, size = C.ssspmv_cached_workspace(st)
    assert size >= need
    for _ in range(2):
        C.check(C.ssspmv_csr_batched_f32(1, desc, int(rp[-1]), opts=opts, workspace=ptr,
                                         ws_bytes=size, stream=st), "batched")
        C.check(C.ssspmv_csr_f64(m, 517, int(rq[-1]), *arrays, y, stream=st), "csr")
        st.synchronize()
        assert np.array_equal(y.cpu().numpy(), want)
    C.ssspmv_release_workspaces()


@pytest.mark.parametrize("kind", ["upto4", "oversized"])
def test_error_bits_of_the_first_kernel_reach_the_status(dev, kind):
    """A bit that a block of the first kernel sets (word 9 of the workspace, here
    set before the call) is the call's status whichever block runs first, with
    rows left to the second kernel and without, and gone after the next call."""
    from paper_1504_06474_gb300 import ssspmv as C
    m = 9001
    rp, col, val, x = _matrix(kind, m, 517, seed=3)
    nnz, want = int(rp[-1]), oracle.spmv(rp, col, val, x)
    rpd, cd, vd, xd = _device(dev, (rp, col, val, x))
    ws = torch.empty(C.ssspmv_workspace_bytes(m, nnz, 8, None), dtype=torch.uint8, device=dev)
    y = torch.empty(m, dtype=torch.float64, device=dev)
    plan = C.ssspmv_plan_create(m, 517, nnz, rpd, 8, workspace=ws)
    try:
        for bits in (0, C.SSSPMV_DEV_RANGE, 0, C.SSSPMV_DEV_TIMEOUT, 0):
            if bits:
                ws[36:40].view(torch.int32).fill_(bits)
            C.check(C.ssspmv_plan_execute(plan, cd, vd, xd, y), "execute")
            assert C.ssspmv_device_status(ws) == bits
            assert np.array_equal(y.cpu().numpy(), want)
    finally:
        C.ssspmv_plan_destroy(plan)


def _small_matrices(dev, count, seed):
    """A batch of `count` small matrices over one x (rows of 0 to 15 entries, some
    matrices without rows or entries): descriptors, all y in a row, the sum of
    nnz, and what y has to be."""
    rng = np.random.default_rng(seed)
    n = 517
    ms = rng.integers(20, 120, size=count)
    ms[rng.random(count) < 0.1] = 0
    ms[-3:] = 0
    lens = rng.integers(0, 16, size=int(ms.sum()))
    row0 = np.concatenate([[0], np.cumsum(ms)])
    lens[row0[count // 3]:row0[count // 3 + 2]] = 0
    nnz = np.array([lens[a:b].sum() for a, b in zip(row0[:-1], row0[1:])])
    at = np.concatenate([[0], np.cumsum((nnz + 3) // 4 * 4)])  # 16-byte aligned starts
    col = rng.integers(0, n, size=int(at[-1]) + 4).astype(np.int32)
    val = rng.integers(-6, 7, size=int(at[-1]) + 4).astype(np.float32)
    x = rng.integers(-6, 7, size=n).astype(np.float32)
    rps = [np.concatenate([[0], np.cumsum(lens[a:b])]) for a, b in zip(row0[:-1], row0[1:])]
    used = np.concatenate([np.arange(k) + a for k, a in zip(nnz, at)]).astype(np.int64)
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    want = oracle.spmv(rp, col[used], val[used].astype(float), x.astype(float))
    rpd, cd, vd, xd = _device(dev, (np.concatenate(rps).astype(np.int32), col, val, x))
    y = torch.full((int(row0[-1]),), float("nan"), device=dev)
    rec = np.zeros(count, dtype=[("m", "<i4"), ("n", "<i4"), ("nnz", "<i4"), ("reserved", "<i4"),
                                 ("rp", "<u8"), ("col", "<u8"), ("val", "<u8"), ("x", "<u8"),
                                 ("y", "<u8")])
    rec["m"], rec["n"], rec["nnz"] = ms, n, nnz
    rec["rp"] = rpd.data_ptr() + 4 * (row0[:-1] + np.arange(count))
    rec["col"], rec["val"] = cd.data_ptr() + 4 * at[:-1], vd.data_ptr() + 4 * at[:-1]
    rec["x"], rec["y"] = xd.data_ptr(), y.data_ptr() + 4 * row0[:-1]
    desc = torch.as_tensor(np.frombuffer(rec.tobytes(), np.uint8).copy(), device=dev)
    return desc, y, int(nnz.sum()), want, (rpd, cd, vd, xd)


@pytest.mark.parametrize("count", [31, 32, 33, 34, 1057, 8000])
def test_batch_finds_the_matrix_of_every_unit(dev, count):
    from paper_1504_06474_gb300 import ssspmv as C
    desc, y, total, want, keep = _small_matrices(dev, count, seed=count)
    ws = torch.empty(C.ssspmv_batched_workspace_bytes(count, total), dtype=torch.uint8, device=dev)
    C.check(C.ssspmv_csr_batched_f32(count, desc, total, workspace=ws), "batched")
    assert C.ssspmv_device_status(ws) == 0
    assert np.array_equal(y.cpu().numpy().astype(np.float64), want)


def _us(fn, reps=7):
    times = []
    for i in range(reps + 2):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        fn()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) * 1e3)
    return float(np.median(times[2:]))


def test_many_matrices_are_no_slower_than_by_tiles(dev):
    # (walking past every matrix, each warp took ten times as long as the tiles)
    from paper_1504_06474_gb300 import ssspmv as C
    count = 8000
    desc, y, total, want, keep = _small_matrices(dev, count, seed=1)
    us = []
    for opts in (None, C.make_opts(W=15, variant=C.VARIANT_SPECULATIVE)):
        ws = torch.empty(C.ssspmv_batched_workspace_bytes(count, total, 4, opts),
                         dtype=torch.uint8, device=dev)
        us.append(_us(lambda: C.check(C.ssspmv_csr_batched_f32(count, desc, total, opts=opts,
                                                               workspace=ws), "batched")))
    assert us[0] <= 1.5 * us[1], us


# several lanes per row and four groups at a time (the sizes are checked on the
# CPU in test_rowshape_host.py): kind, m, lanes per row
LANES = [("const28", 400_003, 2), ("upto56", 400_003, 2), ("const60", 200_003, 4),
         ("upto120", 200_003, 4), ("const120", 100_003, 8), ("upto240", 100_003, 8),
         ("const220", 50_003, 16), ("upto440", 50_003, 16), ("const440", 25_003, 32),
         ("upto900", 25_003, 32)]


@pytest.mark.parametrize("kind,m,lanes,prec",
                         [c + ("f64",) for c in LANES] +
                         [c + (p,) for c in LANES[1::2] for p in ("f32", "bf16")])
def test_several_lanes_per_row_in_units_of_four_groups(dev, kind, m, lanes, prec):
    from paper_1504_06474_gb300 import ssspmv as C
    rp, col, val, x = _matrix(kind, m, 517, seed=lanes)
    if kind.startswith("upto"):  # and a run of empty rows across units
        gone = slice(m // 3, m // 3 + 300)
        lens = np.diff(rp)
        lens[gone] = 0
        rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        col, val = col[: rp[-1]], val[: rp[-1]]
    nnz, want = int(rp[-1]), oracle.spmv(rp, col, val, x)
    vt = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[prec]
    fn = {"f64": C.ssspmv_csr_f64, "f32": C.ssspmv_csr_f32, "bf16": C.ssspmv_csr_bf16f32}[prec]
    rpd, cd, vd, xd = _device(dev, (rp, col, val, x))
    vd, xt = vd.to(vt), torch.float64 if prec == "f64" else torch.float32
    if prec == "bf16":
        vd = vd.view(torch.int16)
    y = torch.full((m,), float("nan"), dtype=xt, device=dev)
    C.check(fn(m, 517, nnz, rpd, cd, vd, xd.to(xt), y), prec)
    assert np.array_equal(y.cpu().numpy().astype(np.float64), want)


def test_several_lanes_per_row_in_a_batch(dev):
    from paper_1504_06474_gb300 import ssspmv as C
    keep, descs, wants, ys = [], [], [], []
    for i, (kind, m) in enumerate([("upto12", 700), ("upto120", 200_003), ("empty", 33),
                                   ("upto900", 25_003), ("pieces", 5000), ("upto56", 400_003)]):
        rp, col, val, x = _matrix(kind, m, 517, seed=200 + i)
        rpd, cd, vd, xd = _device(dev, (rp, col, val.astype(np.float32), x.astype(np.float32)))
        y = torch.full((m,), float("nan"), dtype=torch.float32, device=dev)
        keep.append((rpd, cd, vd, xd))
        descs.append((m, 517, int(rp[-1]), rpd, cd, vd, xd, y))
        wants.append(oracle.spmv(rp, col, val, x))
        ys.append(y)
    total = sum(d[2] for d in descs)
    desc = torch.frombuffer(bytearray(C.batch_descriptors(descs)), dtype=torch.uint8).to(dev)
    ws = torch.empty(C.ssspmv_batched_workspace_bytes(len(descs), total), dtype=torch.uint8,
                     device=dev)
    C.check(C.ssspmv_csr_batched_f32(len(descs), desc, total, workspace=ws), "batched")
    assert C.ssspmv_device_status(ws) == 0
    for y, want in zip(ys, wants):
        assert np.array_equal(y.cpu().numpy().astype(np.float64), want)


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("share", [0.0, 1e-6, 0.001, 0.5])
def test_many_rows_of_hardly_any_entries(dev, share, prec):
    """Units without entries (nothing is copied), alone and between others, up to
    a matrix without any; NaN beforehand shows a row that is not written."""
    from paper_1504_06474_gb300 import ssspmv as C
    rng = np.random.default_rng(4)
    m, n = 2_500_003, 517
    lens = (rng.random(m) < share) * rng.integers(1, 3, size=m)
    lens[400_000:900_000] = 0
    lens[700_001:700_400] = 3 if share else 0
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    nnz = int(rp[-1])
    col = rng.integers(0, n, size=nnz).astype(np.int32)
    val = rng.integers(-6, 7, size=nnz).astype(float)
    x = rng.integers(-6, 7, size=n).astype(float)
    want = oracle.spmv(rp, col, val, x)
    vt = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[prec]
    fn = {"f64": C.ssspmv_csr_f64, "f32": C.ssspmv_csr_f32, "bf16": C.ssspmv_csr_bf16f32}[prec]
    rpd, cd, vd, xd = _device(dev, (rp, col, val, x))
    xt = torch.float64 if prec == "f64" else torch.float32
    vd = vd.to(vt).view(torch.int16) if prec == "bf16" else vd.to(vt)
    y = torch.full((m,), float("nan"), dtype=xt, device=dev)
    C.check(fn(m, n, nnz, rpd, cd, vd, xd.to(xt), y), prec)
    assert np.array_equal(y.cpu().numpy().astype(np.float64), want)
    if prec == "f64":  # y = 2 A x + 3 y: rows without entries are scaled too
        C.check(C.ssspmv_csr_f64_axpby(m, n, nnz, rpd, cd, vd, xd, y, 2.0, 3.0), "axpby")
        assert np.array_equal(y.cpu().numpy(), 5.0 * want)
        y.fill_(1.0)
        C.check(C.ssspmv_csr_f64_axpby(m, n, nnz, rpd, cd, vd, xd, y, 2.0, 3.0), "axpby")
        assert np.array_equal(y.cpu().numpy(), 2.0 * want + 3.0)


def _long_rows(seed):
    """Rows of up to 7,200 entries, 24 million in all, so that rows of up to
    about 5,860 are worked off in several stages and longer ones in pieces; at
    the edges of stages (888), of both, and empty ones."""
    rng = np.random.default_rng(seed)
    lens = rng.integers(2500, 7200, size=5000)
    lens[rng.choice(5000, 500, replace=False)] = 0
    share = int(lens.sum()) >> 12
    edges = [0, 1, 31, 32, 33, 887, 888, 889, 896, 1775, 1776, 1777, 2663, 2664, 2665, 2672,
             share - 1, share, share + 1, 7104, 7105]
    lens[1000: 1000 + len(edges)] = edges
    lens[-1] = 3001
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
def test_rows_of_several_stages(dev, prec):
    from paper_1504_06474_gb300 import ssspmv as C
    rng = np.random.default_rng(8)
    n = 60_000
    rp = _long_rows(8)
    m, nnz = rp.size - 1, int(rp[-1])
    col = rng.integers(0, n, size=nnz).astype(np.int32)
    val, x = rng.integers(-6, 7, size=nnz).astype(float), rng.integers(-6, 7, size=n).astype(float)
    want = oracle.spmv(rp, col, val, x)
    vt = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[prec]
    fn = {"f64": C.ssspmv_csr_f64, "f32": C.ssspmv_csr_f32, "bf16": C.ssspmv_csr_bf16f32}[prec]
    xt = torch.float64 if prec == "f64" else torch.float32
    rpd, cd, vd, xd = _device(dev, (rp, col, val, x))
    vd = vd.to(vt).view(torch.int16) if prec == "bf16" else vd.to(vt)
    y = torch.full((m,), float("nan"), dtype=xt, device=dev)
    C.check(fn(m, n, nnz, rpd, cd, vd, xd.to(xt), y), prec)
    assert np.array_equal(y.cpu().numpy().astype(np.float64), want)
    if prec == "f32":  # the same bits in a batch
        val32, x32 = (torch.as_tensor(rng.uniform(-1, 1, k).astype(np.float32), device=dev)
                      for k in (nnz, n))
        C.check(fn(m, n, nnz, rpd, cd, val32, x32, y), "f32")
        yb = torch.full((m,), float("nan"), device=dev)
        desc = torch.frombuffer(bytearray(C.batch_descriptors(
            [(m, n, nnz, rpd, cd, val32, x32, yb)])), dtype=torch.uint8).to(dev)
        ws = torch.empty(C.ssspmv_batched_workspace_bytes(1, nnz), dtype=torch.uint8, device=dev)
        C.check(C.ssspmv_csr_batched_f32(1, desc, nnz, workspace=ws), "batched")
        assert torch.equal(y, yb)
    elif prec == "f64":
        C.check(C.ssspmv_csr_f64_axpby(m, n, nnz, rpd, cd, vd, xd, y, 2.0, -3.0), "axpby")
        assert np.array_equal(y.cpu().numpy(), -want)
        val, x = rng.uniform(-1, 1, nnz), rng.uniform(-1, 1, n)
        vd, xd = _device(dev, (val, x))
        C.check(fn(m, n, nnz, rpd, cd, vd, xd, y), "f64")
        yref, s = oracle.spmv_dot2(rp, col, val, x)
        assert np.all(np.abs(y.cpu().numpy() - yref) <= 1e-13 * s)


@pytest.mark.parametrize("prec,length", [("f32", 2100), ("bf16", 2100), ("f64", 2100),
                                         ("f32", 900)])
def test_long_rows_are_no_slower_than_by_tiles(dev, prec, length):
    # (all listed, rows of 2,100 took 1.35 to twice the tiles' time)
    from paper_1504_06474_gb300 import ssspmv as C
    m, n = 25_000_000 // length, 100_000
    nnz = m * length
    rp = torch.arange(m + 1, device=dev, dtype=torch.int32) * length
    col = (torch.arange(nnz, device=dev) % n).to(torch.int32)
    vt = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[prec]
    xt = torch.float64 if prec == "f64" else torch.float32
    val = torch.ones(nnz, dtype=vt, device=dev)
    if prec == "bf16":
        val = val.view(torch.int16)
    x = torch.ones(n, dtype=xt, device=dev)
    y = torch.empty(m, dtype=xt, device=dev)
    fn = {"f64": C.ssspmv_csr_f64, "f32": C.ssspmv_csr_f32, "bf16": C.ssspmv_csr_bf16f32}[prec]
    us = []
    for opts in (None, C.make_opts(variant=C.VARIANT_SPECULATIVE)):
        us.append(_us(lambda: C.check(fn(m, n, nnz, rp, col, val, x, y, opts=opts), prec)))
        assert torch.all(y == float(length))
    assert us[0] <= 1.25 * us[1], us


def _block_rows(lo, hi, total, rng):
    """Row lengths of a block-diagonal matrix of dense blocks of lo to hi rows."""
    sizes = rng.integers(lo, hi + 1, size=2 * total // ((lo + hi) * lo) + 50)
    lens = np.repeat(sizes, sizes)
    return lens[: np.searchsorted(np.cumsum(lens), total)]


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("lo,hi", [(32, 64), (30, 70), (32, 130), (40, 256), (200, 500)])
def test_groups_by_halves(dev, lo, hi, prec):
    """Equal rows in a group, several lanes each, more entries than a stage: by
    halves, next to groups that fit, with a few rows that break the evenness."""
    from paper_1504_06474_gb300 import ssspmv as C
    rng = np.random.default_rng(hi)
    lens = _block_rows(lo, hi, 3_000_000, rng)
    at = rng.choice(lens.size, 200, replace=False)
    lens[at[:100]] = 0
    lens[at[100:]] = rng.integers(1, 700, size=100)
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    m, n, nnz = lens.size, 517, int(rp[-1])
    col = rng.integers(0, n, size=nnz).astype(np.int32)
    val, x = rng.integers(-6, 7, size=nnz).astype(float), rng.integers(-6, 7, size=n).astype(float)
    want = oracle.spmv(rp, col, val, x)
    vt = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[prec]
    fn = {"f64": C.ssspmv_csr_f64, "f32": C.ssspmv_csr_f32, "bf16": C.ssspmv_csr_bf16f32}[prec]
    xt = torch.float64 if prec == "f64" else torch.float32
    rpd, cd, vd, xd = _device(dev, (rp, col, val, x))
    vd = vd.to(vt).view(torch.int16) if prec == "bf16" else vd.to(vt)
    y = torch.full((m,), float("nan"), dtype=xt, device=dev)
    C.check(fn(m, n, nnz, rpd, cd, vd, xd.to(xt), y), prec)
    assert np.array_equal(y.cpu().numpy().astype(np.float64), want)
    if prec == "f32":  # the same bits in a batch
        val32, x32 = (torch.as_tensor(rng.uniform(-1, 1, k).astype(np.float32), device=dev)
                      for k in (nnz, n))
        C.check(fn(m, n, nnz, rpd, cd, val32, x32, y), "f32")
        yb = torch.full((m,), float("nan"), device=dev)
        desc = torch.frombuffer(bytearray(C.batch_descriptors(
            [(m, n, nnz, rpd, cd, val32, x32, yb)])), dtype=torch.uint8).to(dev)
        ws = torch.empty(C.ssspmv_batched_workspace_bytes(1, nnz), dtype=torch.uint8, device=dev)
        C.check(C.ssspmv_csr_batched_f32(1, desc, nnz, workspace=ws), "batched")
        assert torch.equal(y, yb)


@pytest.mark.parametrize("prec", ["f32", "bf16", "f64"])
def test_diagonal_blocks_are_no_slower_than_by_tiles(dev, prec):
    # (split evenly, their two-stage groups took 1.1 to 1.3 times the tiles' time)
    from paper_1504_06474_gb300 import ssspmv as C
    lens = _block_rows(32, 64, 28_000_000, np.random.default_rng(1))
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    m, nnz = lens.size, int(rp[-1])
    rpd = torch.as_tensor(rp, device=dev)
    col = (torch.arange(nnz, device=dev) % 100_000).to(torch.int32)
    vt = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[prec]
    xt = torch.float64 if prec == "f64" else torch.float32
    val = torch.ones(nnz, dtype=vt, device=dev)
    if prec == "bf16":
        val = val.view(torch.int16)
    x = torch.ones(100_000, dtype=xt, device=dev)
    y = torch.empty(m, dtype=xt, device=dev)
    fn = {"f64": C.ssspmv_csr_f64, "f32": C.ssspmv_csr_f32, "bf16": C.ssspmv_csr_bf16f32}[prec]
    us = []
    for opts in (None, C.make_opts(variant=C.VARIANT_SPECULATIVE)):
        us.append(_us(lambda: C.check(fn(m, 100_000, nnz, rpd, col, val, x, y, opts=opts), prec)))
        assert np.array_equal(y.cpu().numpy(), lens)
    assert us[0] <= 1.05 * us[1], us


@pytest.mark.parametrize("m,long,every", [(64_000, 641, 64), (64_003, 639, 64), (200_000, 700, 128),
                                          (20_007, 1200, 96), (500_000, 1024, 352),
                                          (500_000, 1025, 352)])
def test_groups_that_one_row_fills(dev, m, long, every):
    """Groups just past the stage whose longest row has most of the entries, as
    many as the lists are sized for, between groups of short rows and empty ones."""
    from paper_1504_06474_gb300 import ssspmv as C
    rng = np.random.default_rng(every)
    lens = rng.integers(0, 2, size=m) * (np.arange(m) % every >= 32)
    lens[7::every] = long
    lens[9::every] = 1
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    n, nnz = 517, int(rp[-1])
    col = rng.integers(0, n, size=nnz).astype(np.int32)
    val, x = rng.integers(-6, 7, size=nnz).astype(float), rng.integers(-6, 7, size=n).astype(float)
    want = oracle.spmv(rp, col, val, x)
    rpd, cd, vd, xd = _device(dev, (rp, col, val, x))
    ws = torch.full((C.ssspmv_workspace_bytes(m, nnz, 8, None) + 256,), 255, dtype=torch.uint8,
                    device=dev)
    size = C.ssspmv_workspace_bytes(m, nnz, 8, None)
    for _ in range(2):
        y = torch.full((m,), float("nan"), dtype=torch.float64, device=dev)
        C.check(C.ssspmv_csr_f64(m, n, nnz, rpd, cd, vd, xd, y, workspace=ws, ws_bytes=size), "csr")
        assert C.ssspmv_device_status(ws) == 0
        assert np.array_equal(y.cpu().numpy(), want)
        assert bool((ws[size:] == 255).all())  # nothing past the workspace
    C.check(C.ssspmv_csr_f64_axpby(m, n, nnz, rpd, cd, vd, xd, y, 2.0, -3.0, workspace=ws,
                                   ws_bytes=size), "axpby")
    assert np.array_equal(y.cpu().numpy(), -want)
    y32 = torch.full((m,), float("nan"), device=dev)
    C.check(C.ssspmv_csr_f32(m, n, nnz, rpd, cd, vd.float(), xd.float(), y32), "f32")
    assert np.array_equal(y32.cpu().numpy().astype(np.float64), want)


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("m", [1_499_999, 1_500_000, 1_700_003])
def test_very_short_rows(dev, m, prec):
    """Both sides of the size from which matrices of very short rows have a
    kernel of their own: rows past its limit, uneven stages, listed groups and
    empty stretches among them, and in FP32 the bits of the batch."""
    from paper_1504_06474_gb300 import ssspmv as C
    rng = np.random.default_rng(m)
    n = 60_000
    lens = rng.integers(0, 4, size=m)
    lens[100_000:300_000] = rng.integers(0, 9, size=200_000)
    lens[rng.choice(m, 3000, replace=False)] = 40
    lens[rng.choice(m, 50, replace=False)] = rng.integers(300, 5000, size=50)
    lens[400_000:420_000] = 0
    lens[-40:] = 4
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    nnz = int(rp[-1])
    assert nnz <= 3 * m
    col = rng.integers(0, n, size=nnz).astype(np.int32)
    val, x = rng.integers(-6, 7, size=nnz).astype(float), rng.integers(-6, 7, size=n).astype(float)
    want = oracle.spmv(rp, col, val, x)
    vt = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[prec]
    fn = {"f64": C.ssspmv_csr_f64, "f32": C.ssspmv_csr_f32, "bf16": C.ssspmv_csr_bf16f32}[prec]
    xt = torch.float64 if prec == "f64" else torch.float32
    rpd, cd, vd, xd = _device(dev, (rp, col, val, x))
    vd = vd.to(vt).view(torch.int16) if prec == "bf16" else vd.to(vt)
    y = torch.full((m,), float("nan"), dtype=xt, device=dev)
    C.check(fn(m, n, nnz, rpd, cd, vd, xd.to(xt), y), prec)
    assert np.array_equal(y.cpu().numpy().astype(np.float64), want)
    if prec == "f32":
        val32, x32 = (torch.as_tensor(rng.uniform(-1, 1, k).astype(np.float32), device=dev)
                      for k in (nnz, n))
        C.check(fn(m, n, nnz, rpd, cd, val32, x32, y), "f32")
        yb = torch.full((m,), float("nan"), device=dev)
        desc = torch.frombuffer(bytearray(C.batch_descriptors(
            [(m, n, nnz, rpd, cd, val32, x32, yb)])), dtype=torch.uint8).to(dev)
        ws = torch.empty(C.ssspmv_batched_workspace_bytes(1, nnz), dtype=torch.uint8, device=dev)
        C.check(C.ssspmv_csr_batched_f32(1, desc, nnz, workspace=ws), "batched")
        assert torch.equal(y, yb)
    elif prec == "f64":
        C.check(C.ssspmv_csr_f64_axpby(m, n, nnz, rpd, cd, vd, xd, y, 2.0, -3.0), "axpby")
        assert np.array_equal(y.cpu().numpy(), -want)
        x_nan = x.copy()  # one column's NaN reaches exactly the rows that use it
        x_nan[123] = np.nan
        C.check(fn(m, n, nnz, rpd, cd, vd, torch.as_tensor(x_nan, device=dev), y), "nan")
        uses = np.zeros(m, bool)
        uses[np.repeat(np.arange(m), lens)[col == 123]] = True
        assert np.array_equal(np.isnan(y.cpu().numpy()), uses)


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_rows_of_one_entry_are_no_slower_than_by_tiles(dev, prec):
    # (one group after the other, 20 million rows took 1.1 to 1.6 times the tiles' time)
    from paper_1504_06474_gb300 import ssspmv as C
    m = 20_000_000
    xt = torch.float64 if prec == "f64" else torch.float32
    rp = torch.arange(m + 1, device=dev, dtype=torch.int32)
    col = torch.arange(m - 1, -1, -1, device=dev, dtype=torch.int32)
    val = torch.full((m,), 2.0, dtype=xt, device=dev)
    x = torch.arange(m, device=dev).to(xt)
    y = torch.empty(m, dtype=xt, device=dev)
    fn = C.ssspmv_csr_f64 if prec == "f64" else C.ssspmv_csr_f32
    us = []
    for opts in (None, C.make_opts(variant=C.VARIANT_SPECULATIVE)):
        us.append(_us(lambda: C.check(fn(m, m, m, rp, col, val, x, y, opts=opts), prec)))
        assert torch.equal(y, 2.0 * x.flip(0))
    assert us[0] <= 1.05 * us[1], us
