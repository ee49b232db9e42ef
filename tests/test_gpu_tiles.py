"""The segmented sum over tiles where a caller asks for it without a tile shape:
the variant alone, so that tile width, bunch size and block shape are the
library's.  (Calls without any option go by row blocks.)  Full-size products in
every precision, long dirty tiles in FP32, in a batch and in shards, batches
with bad descriptors, too small a bound and under graph replay, plans, the
fixed scratch and host buffers."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_batched import Batch, _C, _check_all, _mixed_batch  # noqa: E402
from test_gpu_long_tiles import long_tile_matrix  # noqa: E402
from test_gpu_parity import check_case  # noqa: E402
from test_gpu_reduced import _check  # noqa: E402
from test_gpu_shards import _ntiles, _run_shards, _small_int  # noqa: E402

TOL = 1e-13
VARIANTS = [1, 2]  # speculative, exact


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1504_06474_gb300 import _build
    _build.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("variant", VARIANTS)
@pytest.mark.parametrize("name", ["stencil160", "rmat22"])
def test_full_size_f64(dev, name, variant):
    A, x = synth.workload(name)
    check_case(dev, A.row_ptr, A.col, A.val, x, A.n, variant=variant)


def _reduced(dev, A, x, prec, variant):
    C = _C()
    opts = C.make_opts(variant=variant)
    if prec == "f32":
        v, vb, fn = torch.as_tensor(A.val.astype(np.float32)), 4, C.ssspmv_csr_f32
    else:
        v, vb, fn = torch.as_tensor(A.val).to(torch.bfloat16), 2, C.ssspmv_csr_bf16f32
    x32 = x.astype(np.float32)
    ws = torch.empty(C.ssspmv_workspace_bytes(A.m, A.nnz, vb, opts), dtype=torch.uint8, device=dev)
    y = torch.full((A.m,), float("nan"), dtype=torch.float32, device=dev)
    vd = v.to(dev) if prec == "f32" else v.to(dev).view(torch.int16)
    C.check(fn(A.m, A.n, A.nnz, torch.as_tensor(A.row_ptr, device=dev),
               torch.as_tensor(A.col, device=dev), vd, torch.as_tensor(x32, device=dev), y,
               opts=opts, workspace=ws), prec)
    assert C.ssspmv_device_status(ws) == 0
    _check(A, x, v.double().numpy(), x32.astype(np.float64), y.cpu().numpy().astype(np.float64),
           "%s tiles" % prec)


@pytest.mark.parametrize("variant", VARIANTS)
@pytest.mark.parametrize("prec", ["f32", "bf16"])
def test_long_tiles_reduced(dev, prec, variant):
    A, x = long_tile_matrix()
    _reduced(dev, A, x, prec, variant)


@pytest.mark.parametrize("prec", ["f32", "bf16"])
@pytest.mark.parametrize("name", ["rmat22", "uniform4096", "stencil100"])
def test_workloads_reduced(dev, name, prec):
    A, x = synth.workload(name)
    _reduced(dev, A, x, prec, 1)


@pytest.mark.parametrize("variant", VARIANTS)
def test_batch_with_long_tiles(dev, variant):
    A, x = long_tile_matrix()
    small = [synth.batch_matrix(s) for s in synth.batch_specs(6, seed=22, m_lo=40, m_hi=20000)]
    for mats in (small[:3] + [(A, x)] + small[3:], _mixed_batch()):
        b = Batch(mats, dev)
        opts = _C().make_opts(variant=variant)
        assert _C().ssspmv_device_status(b.run(opts)) == 0
        _check_all(b, opts)


def test_batch_refusals(dev):
    C = _C()
    opts = C.make_opts(variant=1)
    b = Batch(_mixed_batch()[:6], dev)
    assert C.ssspmv_device_status(b.run(opts, total_nnz=b.total_nnz // 4)) & C.SSSPMV_DEV_BATCH
    for y in b.y:
        assert torch.isnan(y).all()
    raw = b.desc.cpu().numpy().copy()
    raw[2 * 56 + 12: 2 * 56 + 16] = np.frombuffer(np.int32(1).tobytes(), np.uint8)  # reserved
    b.desc = torch.as_tensor(raw, device=dev)
    assert C.ssspmv_device_status(b.run(opts)) == C.SSSPMV_DEV_BATCH
    assert torch.isnan(b.y[2]).all()
    _check_all(b, opts, skip=(2,))


def test_batch_in_a_cuda_graph(dev):
    C = _C()
    opts = C.make_opts(variant=1)
    b = Batch(_mixed_batch(), dev)
    ws = torch.empty(C.ssspmv_batched_workspace_bytes(len(b.mats), b.total_nnz, 4, opts),
                     dtype=torch.uint8, device=dev)

    def call(stream):
        C.check(C.ssspmv_csr_batched_f32(len(b.mats), b.desc, b.total_nnz, opts=opts, workspace=ws,
                                         stream=stream), "batched")
    s = torch.cuda.Stream(dev)
    torch.cuda.synchronize()
    call(s)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        call(s)
    for y in b.y:
        y.fill_(float("nan"))
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert C.ssspmv_device_status(ws) == 0
    _check_all(b, opts)


@pytest.mark.parametrize("variant", VARIANTS)
def test_shards(dev, variant):
    from paper_1504_06474_gb300 import api
    opts = _C().make_opts(variant=variant)
    A, x = _small_int(1)
    for shards in (1, 3, 7):
        y = _run_shards(dev, A, x, api.split_tiles(_ntiles(A, opts), shards), opts)
        assert np.array_equal(y, oracle.spmv(A.row_ptr, A.col, A.val, x))
    for (A, x), shards in ((long_tile_matrix(), 4), (synth.workload("rmat22"), 3)):
        y = _run_shards(dev, A, x, api.split_tiles(_ntiles(A, opts), shards), opts)
        yref, s = oracle.spmv_dot2(A.row_ptr, A.col, A.val, x)
        assert np.all(np.abs(y - yref) <= TOL * s)
        assert np.all(y[s == 0] == 0.0)


@pytest.mark.parametrize("variant", VARIANTS)
def test_plans_scratch_and_host_buffers(dev, variant):
    """One product by every single-matrix entry point: the same y bit for bit,
    and y = alpha A x + beta y of it."""
    C = _C()
    lens = synth.random_lengths(20000, seed=21, mean=7.0, p_empty=0.25, p_long=0.0005,
                                long_len=4000)
    A = synth.from_lengths(lens, 6000, seed=21)
    x = synth.sym_vector(A.n, seed=21)
    opts = C.make_opts(variant=variant)
    rp, col, val, xd = (torch.as_tensor(a, device=dev) for a in (A.row_ptr, A.col, A.val, x))
    ys = [torch.full((A.m,), float("nan"), dtype=torch.float64, device=dev) for _ in range(3)]
    C.check(C.ssspmv_csr_f64(A.m, A.n, A.nnz, rp, col, val, xd, ys[0], opts=opts), "csr")
    C.check(C.ssspmv_csr_f64_noalloc(A.m, A.n, A.nnz, rp, col, val, xd, ys[1], opts=opts),
            "noalloc")
    plan = C.ssspmv_plan_create(A.m, A.n, A.nnz, rp, 8, opts)
    try:
        C.check(C.ssspmv_plan_execute(plan, col, val, xd, ys[2]), "execute")
        scaled = ys[2].clone()
        C.check(C.ssspmv_plan_execute_axpby(plan, col, val, xd, scaled, 0.5, 0.75), "axpby")
    finally:
        C.ssspmv_plan_destroy(plan)
    host = np.full(A.m, np.nan)
    buf = torch.empty(C.ssspmv_host_buffer_bytes(A.m, A.n, A.nnz, opts), dtype=torch.uint8,
                      device=dev)
    C.check(C.ssspmv_csr_f64_host(A.m, A.n, A.nnz, A.row_ptr, A.col, A.val, x, host,
                                  dev_buffer=buf, opts=opts), "host")
    yref, s = oracle.spmv_dot2(A.row_ptr, A.col, A.val, x)
    y = ys[0].cpu().numpy()
    assert np.all(np.abs(y - yref) <= TOL * s) and np.all(y[s == 0] == 0.0)
    for other in (ys[1].cpu().numpy(), ys[2].cpu().numpy(), host):
        assert np.array_equal(other, y)
    # fma(0.75, y, 0.5 A x): two more roundings
    assert np.all(np.abs(scaled.cpu().numpy() - 1.25 * yref) <= 2 * TOL * s)
