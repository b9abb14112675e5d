"""Convolutions on operand tensors (widths that are multiples of eight) at the
widths, images and batches where their tiles, chunk pairs and K ranges end."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1801_04577_gb300 import inputs as I  # noqa: E402
from paper_1801_04577_gb300.net import Net, layer_shapes  # noqa: E402

from test_gpu_surrogate import _layer_errors, _sparse_dyadic_params  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,cin,cout,base,levels,N", [
    (8, 5, 4, 8, 2, 1),      # one channel group (nine chunks of K), one partial tile
    (16, 1, 2, 8, 3, 3),     # deepest image 4^2, smallest input
    (48, 7, 4, 16, 4, 1),    # images that are no power of two, the widest unrolled first layer
    (32, 8, 8, 40, 3, 2),    # five and fifteen groups: pairs across taps; an eight-channel input and output
    (64, 5, 2, 8, 5, 5),     # five levels: several ranges of K in one block
])
def test_forward_exact_when_sums_are_exact(G, cin, cout, base, levels, N):
    """Sums of dyadic numbers are exact in any order, so the forward pass equals
    the reference bit for bit.  Gradients: where 2 / (N C G^2) is a power of two
    as in the whole-network test; else FP32's rounding of it can move an element
    to the next BF16 number, once (2^-8) a layer."""
    from oracle import surrogate as S
    shapes = layer_shapes(G, cin, cout, base, levels)
    net = Net(G, cin, cout, base, levels, N, seed=3, math="tensor")
    p = _sparse_dyadic_params(shapes, 100 + G + base)
    net.set_params(p)
    r = I.splitmix64_uniform(7, N * (cin + cout) * G * G)
    x = (np.floor(r[:N * cin * G * G] * 9 - 4) / 4).reshape(N, cin, G, G).astype(np.float32)
    t = (np.floor(r[N * cin * G * G:] * 9 - 4) / 4).reshape(N, cout, G, G).astype(np.float32)
    xd, td = (torch.from_numpy(a).cuda() for a in (x, t))
    y = torch.empty((N, cout, G, G), dtype=torch.float32, device="cuda")
    net.forward(xd, y)
    loss, g = net.gradients(xd, td, None)
    L_ref, g_ref, y_ref = S.loss_and_grad(p.astype(np.float64), shapes, levels, x, t, None, rnd=S.bf16)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(y.cpu().numpy(), y_ref.astype(np.float32))
    assert loss == pytest.approx(L_ref, rel=1e-9)
    e = _layer_errors(g, g_ref, shapes)
    assert e.max() <= (5e-5 if N & (N - 1) == 0 and G & (G - 1) == 0 else len(shapes) * 2.0 ** -8), e
    net.close()


def test_smaller_batches_after_larger_ones():
    """Operands of a larger batch stay behind a smaller one's: they must not be read."""
    G, base, levels = 16, 8, 3
    a, b = (Net(G, 5, 3, base, levels, 4, seed=9) for _ in range(2))
    r = torch.from_numpy(I.splitmix64_uniform(3, 4 * 8 * G * G).reshape(4, 8, G, G).astype(np.float32)).cuda()
    x, t = r[:, :5].contiguous() * 2 - 1, r[:, 5:].contiguous()
    a.gradients(x, t)
    for n in (1, 3):
        la, ga = a.gradients(x[:n].contiguous(), t[:n].contiguous())
        lb, gb = b.gradients(x[:n].contiguous(), t[:n].contiguous())
        assert la == lb
        np.testing.assert_array_equal(ga, gb)
    a.close()
    b.close()
