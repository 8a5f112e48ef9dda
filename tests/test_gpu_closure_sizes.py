"""Gradient and binary32 forward pass of the learned closure at the sizes where the tiled kernels
can go wrong: sides of one cell (every neighbour is the cell itself), sides below, at and just
above a tile (32 columns; 8, 16 and 32 rows), odd widths (no 16-byte stores), several snapshots,
more tiles than blocks, and a scratch buffer that grows and is reused."""
import numpy as np
import pytest

from oracle import closure as oc
from paper_1705_09807_gb300 import lbmhd
from paper_1705_09807_gb300.inputs import splitmix64_uniform

pytestmark = pytest.mark.gpu
ONES = (np.ones(12, np.float32), np.ones(4, np.float32))


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


@pytest.mark.parametrize("b,h,w", [(1, 1, 1), (1, 1, 3), (2, 2, 1), (1, 3, 40), (3, 7, 31), (1, 8, 32), (2, 9, 33),
                                   (1, 16, 32), (1, 17, 36), (5, 33, 65), (1, 31, 127), (70, 24, 61)])
def test_gradient_and_forward_at_tile_edges(b, h, w):
    """Binary32 sums of at most 3.4e5 terms, blocked by 256: relative L2 1e-5 of the gradient, as
    the tests of the ordinary sizes ask; forward 1e-5 of the largest output."""
    import torch
    rng = np.random.default_rng(b * 10007 + h * 101 + w)
    theta = (oc.init_params(4) + 0.02 * (2 * splitmix64_uniform(4, oc.num_params()) - 1)).astype(np.float32)
    x = rng.normal(size=(b, 12, h, w)).astype(np.float32)
    t = np.tanh(x[:, :4]) + 0.1 * rng.normal(size=(b, 4, h, w)).astype(np.float32)
    xd, td = torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda")
    out = torch.full((b * 4 * h * w + 64,), 7.0, dtype=torch.float32, device="cuda")
    with lbmhd.Closure(theta, *ONES) as cl:
        cl.gradient(xd[:1, :, :1, :1].contiguous(), td[:1, :, :1, :1].contiguous())  # small scratch first
        loss, g = cl.gradient(xd, td)
        loss2, g2 = cl.gradient(xd, td)
        cl.forward(xd, out[: b * 4 * h * w].view(b, 4, h, w), tensor_cores=False)
    assert loss == loss2 and np.array_equal(g, g2)  # deterministic
    L, ref = oc.gradient(theta.astype(np.float64), x.astype(np.float64), t.astype(np.float64))
    assert abs(loss - L) < 1e-5 * L
    assert np.linalg.norm(g - ref) < 1e-5 * np.linalg.norm(ref)
    for part in (slice(3456, 3488), slice(12704, 12736), slice(13888, 13892)):  # biases of the layers
        assert np.linalg.norm(g[part] - ref[part]) < 1e-5 * np.linalg.norm(ref[part]) + 1e-7
    y = oc.forward(theta.astype(np.float64), x.astype(np.float64))[-1]
    got = out.cpu().numpy()
    assert np.max(np.abs(got[:-64].reshape(y.shape) - y)) < 1e-5 * max(1.0, np.max(np.abs(y)))
    assert np.all(got[-64:] == 7.0)  # nothing written past the output
