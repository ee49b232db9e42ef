"""The selector's network at the edges of the one-kernel path (tiles of 16
samples, scratch for fewer blocks than tiles, sizes it leaves to the layer
kernels) against the FP64 oracle."""
import numpy as np
import pytest

from oracle import selector as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1504_06474_gb300 import _build
    _build.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("B", [1, 14, 15, 16, 17, 65, 300])
@pytest.mark.parametrize("F,H,K", [(16, 64, 10), (32, 64, 32), (4, 64, 1), (15, 64, 10), (16, 48, 10)])
def test_network_sizes(dev, B, F, H, K):
    from paper_1504_06474_gb300 import ssspmv as C
    rng = np.random.default_rng(B * 100 + F + K)
    p = rng.normal(0, 0.3, O.sizes(F, H, H, K)).astype(np.float32)
    X = rng.normal(0, 1, (B, F)).astype(np.float32)
    T = rng.normal(3, 1, (B, K)).astype(np.float32)
    T[0, 0] = np.nan
    pd, Xd, Td = (torch.as_tensor(a, device=dev) for a in (p, X, T))
    scratch = torch.full((C.ssspmv_mlp_scratch_floats(B, F, H, H, K),), float("nan"), device=dev)
    out = torch.full((B, K), float("nan"), device=dev)
    C.check(C.ssspmv_mlp_forward(pd, Xd, B, F, H, H, K, scratch, out), "forward")
    ref, _ = O.forward(p.astype(np.float64), X.astype(np.float64), F, H, H, K)
    # sums of at most 65 products of order one, twice: FP32 to a few hundred ulps
    assert np.allclose(out.cpu().numpy(), ref, rtol=1e-4, atol=1e-4)
    g = torch.full((p.size,), float("nan"), device=dev)
    loss = torch.full((1,), float("nan"), device=dev)
    C.check(C.ssspmv_mlp_backward(pd, Xd, Td, B, F, H, H, K, scratch, g, loss), "backward")
    ref_loss, ref_g = O.loss_and_grad(p.astype(np.float64), X.astype(np.float64),
                                      T.astype(np.float64), F, H, H, K)
    assert np.isclose(float(loss.item()), ref_loss, rtol=1e-4)
    assert np.max(np.abs(g.cpu().numpy() - ref_g)) <= 1e-4 * max(1.0, np.max(np.abs(ref_g)))
    cls = torch.full((B,), -1, dtype=torch.int32, device=dev)
    C.check(C.ssspmv_mlp_select(pd, Xd, B, F, H, H, K, scratch, cls), "select")
    assert np.array_equal(cls.cpu().numpy(), out.cpu().numpy().argmin(axis=1))
