"""conv1's weight and bias gradients, summed from the pooled gradient, against the FP64 oracle, at the
smallest batches and with snippets whose weight lies on the rows and columns where the kernel's quarters and
borders meet."""
import numpy as np
import pytest

from oracle import sifter as osf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_15361_gb300 as g  # noqa: E402

NW, NB = 16 * 9, 16


def _bf16_round(a):
    return torch.from_numpy(np.asarray(a, dtype=np.float32)).to(torch.bfloat16).float().numpy().astype(np.float64)


@pytest.mark.parametrize("n", [1, 2, 5])
def test_first_layer_gradients(n):
    """The gradients differ by the BF16 roundings between the layers (2^-9 each) and by the few pooling or
    ReLU decisions that those tip: 3e-2 in the 2-norm, cosine 0.999. The edge rows and columns carry four
    times the amplitude of the rest, so a tap that misses one of them moves the norm by more than 0.2."""
    rng = np.random.default_rng(40 + n)
    theta = osf.init_params(6)
    shapes = osf.param_shapes()
    offs = np.concatenate([[0], np.cumsum([int(np.prod(s)) for s in shapes])])
    for t in (1, 3, 5, 7, 9):
        theta[offs[t]:offs[t + 1]] = rng.normal(0, 0.05, offs[t + 1] - offs[t])
    x = rng.normal(size=(n, 64, 256))
    x[:, [0, 15, 16, 31, 32, 47, 48, 63]] *= 4.0
    x[:, :, [0, 255]] *= 4.0
    y = (np.arange(n) % 2 == 0).astype(np.float64)
    sf = g.Sifter(max_batch=8, training=True, seed=1)
    sf.set_params(theta.astype(np.float32))
    _, got = sf.gradients(torch.from_numpy(x.astype(np.float32)).cuda(), torch.from_numpy(y.astype(np.float32)).cuda())
    got = got.cpu().numpy().astype(np.float64)
    th = theta.astype(np.float32).astype(np.float64)
    for t in (0, 2, 4, 6):
        th[offs[t]:offs[t + 1]] = _bf16_round(th[offs[t]:offs[t + 1]])
    _, ref = osf.gradients(th, _bf16_round(x), y, act=_bf16_round)
    for lo, hi in ((0, NW), (NW, NW + NB)):
        a, b = got[lo:hi], ref[lo:hi]
        assert np.linalg.norm(a - b) <= 3e-2 * np.linalg.norm(b), (lo, np.linalg.norm(a - b) / np.linalg.norm(b))
        assert a @ b >= 0.999 * np.linalg.norm(a) * np.linalg.norm(b)


def test_a_pixel_that_is_not_finite_reaches_every_tap():
    """0 * inf is NaN: an infinite interior pixel makes every weight gradient of the layer NaN."""
    x = torch.randn((3, 64, 256), generator=torch.Generator().manual_seed(2))
    x[1, 20, 100] = float("inf")
    sf = g.Sifter(max_batch=4, training=True, seed=1)
    _, got = sf.gradients(x.cuda(), torch.tensor([1.0, 0.0, 1.0]).cuda())
    assert torch.isnan(got[:NW]).all()
