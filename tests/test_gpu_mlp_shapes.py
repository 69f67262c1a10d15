"""Loss gradient of the network at the shapes around the fused kernel's rule (64-wide, batches of 32
rows and more) and beside it, against the oracle's FP64 network. Bar 1e-5 relative, the FP32 rounding of
sums over up to a few thousand rows and 64-wide layers."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_08417_gb300 import build, kitrt
    build.build()
    return kitrt


@pytest.mark.parametrize("din,H,dout", [(9, 64, 9), (2, 64, 2), (5, 64, 5), (20, 64, 20), (64, 64, 33), (65, 64, 3), (9, 48, 9)])
@pytest.mark.parametrize("B", [1, 31, 32, 33, 96, 1024, 2500])
def test_loss_grad(K, din, H, dout, B):
    rng = np.random.default_rng(B + din)
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    p, X, T = f(rng.normal(scale=0.3, size=O.mlp_param_count(din, H, dout))), f(rng.normal(size=(B, din))), f(rng.normal(size=(B, dout)))
    dev = lambda a: torch.from_numpy(a).cuda()
    loss, g = K.mlp_loss_grad(dev(p), dev(X), dev(T), din, H, dout)
    lo, go = O.mlp_loss_grad(p.astype(np.float64), X.astype(np.float64), T.astype(np.float64), din, H, dout)
    assert abs(float(loss[0]) - lo) <= 1e-5 * lo
    assert np.linalg.norm(g.cpu().numpy() - go) <= 1e-5 * np.linalg.norm(go)
