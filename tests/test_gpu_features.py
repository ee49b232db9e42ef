"""The selector's row statistics at the edges of their 32-row chunks, against
the FP64 oracle."""
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


@pytest.mark.parametrize("m", [0, 1, 31, 32, 33, 1023, 1025, 200_001])
def test_features_at_chunk_edges(dev, m):
    from paper_1504_06474_gb300 import selector as S
    rng = np.random.default_rng(m)
    lens = rng.integers(0, 12, size=m) * (rng.random(m) < 0.7)
    lens[rng.random(m) < 0.001] = 5000
    rp = np.zeros(m + 1, np.int64)
    np.cumsum(lens, out=rp[1:])
    rp = rp.astype(np.int32)
    f = S.device_features(torch.as_tensor(rp, device=dev), m, m + 1, int(rp[-1])).cpu().numpy()
    assert np.allclose(f.astype(np.float64), O.features(rp, m + 1), rtol=1e-6, atol=1e-7)
