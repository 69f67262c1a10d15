"""The network's loss gradient at batch sizes of hundreds to thousands of tiles against FP64: its error must
not grow with the batch. A row's share has a few roundings of 2^-24, a tile adds 32 rows in FP32, and the
tiles' sums are compensated: 4 x 2^-24 of the gradient's norm."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [512, 8192, 20011, 65536])
def test_gradient_error_does_not_grow(rows):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_08417_gb300 import build, kitrt as K
    build.build()
    d, h = 9, 64
    g = torch.Generator().manual_seed(rows)
    parts = []
    for i, o in [(d, h), (h, h), (h, h), (h, d)]:
        parts += [(torch.rand(i * o, generator=g) * 2 - 1) * (6.0 / (i + o)) ** 0.5, 0.05 * torch.randn(o, generator=g)]
    p = torch.cat(parts).cuda()
    X, T = (torch.randn(rows, d, generator=g).cuda() for _ in range(2))
    loss, grad = K.mlp_loss_grad(p, X, T, d, h, d)
    q = p.double().requires_grad_(True)
    x, off = X.double(), 0
    for layer, (i, o) in enumerate([(d, h), (h, h), (h, h), (h, d)]):
        x = x @ q[off:off + i * o].view(i, o) + q[off + i * o:off + i * o + o]
        off += i * o + o
        if layer < 3:
            x = torch.nn.functional.softplus(x)
    ref = 0.5 * (x - T.double()).square().sum() / rows
    want, = torch.autograd.grad(ref, q)
    err = float((grad.double() - want).norm() / want.norm())
    print(rows, "gradient", err, "loss", abs(float(loss) / float(ref) - 1))
    assert err <= 4 * 2.0 ** -24
    assert abs(float(loss) / float(ref) - 1) <= 4 * 2.0 ** -24
