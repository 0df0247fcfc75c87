"""Kernels at the sizes where they can go wrong: remainders of tiles, the last block of a launch, values at the
edges of a number format.  Every tolerance follows from the arithmetic that is stated beside it."""
import numpy as np
import pytest

from oracle import learned as NL

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

CHANNEL = (1, 2, 3, 3, 3, 3)
PERIODIC = (0, 0, 0, 0, 0, 0)


@pytest.fixture(scope="module")
def L():
    from paper_2002_06206_gb300 import build
    build.build()
    from paper_2002_06206_gb300 import ibmles
    ibmles.lib()
    return ibmles


@pytest.mark.parametrize("shape", [(1, 1, 1), (9, 5, 33), (8, 4, 32), (17, 3, 70), (160, 64, 64)])
def test_weight_gradients_of_a_network_that_is_exact_in_bf16(L, shape):
    """Small integers and powers of two everywhere: every activation and gradient is exact in BF16 and every
    sum is an integer below 2^24, so only the division by N rounds (two FP32 roundings: 1.2e-7).  The last
    shape has more tiles (640) than the launch has blocks."""
    nz, ny, nx = shape
    N = nx * ny * nz
    rng = np.random.default_rng(3)
    flags = (rng.random(N) < 0.4).astype(np.uint8)
    W1, W2, W3 = np.zeros((8, 27, 8)), np.zeros((8, 27, 8)), np.zeros((1, 27, 8))
    W1[0, 4, 2] = 1.0                       # the mask of a neighbour
    W1[3, 13, 2] = 2.0
    W2[0, 22, 0] = W2[1, 10, 3] = W2[5, 13, 0] = 1.0
    W3[0, 16, 0] = W3[0, 0, 1] = 1.0
    B = [np.full(8, 1.0), np.full(8, 0.0), np.zeros(1)]
    target = rng.integers(-3, 4, shape).astype(np.float64)
    x = np.zeros(shape + (8,))
    x[..., 2] = flags.reshape(shape)
    # b = 0 and a pressure change of +-1, whose scale is 1: channel 1 of the features is +-1
    dp = np.where(rng.random(N) < 0.5, 1.0, -1.0)
    x[..., 1] = dp.reshape(shape)
    net = L.Net(np.concatenate([W1.ravel(), W2.ravel(), W3.ravel()] + B).astype(np.float32))
    t = lambda a, dt=torch.float64: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)
    zero = t(np.zeros(N))
    net.train_step(L.make_grid(nx, ny, nz), zero, t(dp), zero, t(target.ravel(), torch.float32), 0.0, t(flags, torch.uint8))
    _, dW, dB, _ = NL.loss_and_grads(x, target, [W1, W2, W3], B)
    ref = np.concatenate([dW[0].ravel(), dW[1].ravel(), dW[2].ravel(), dB[0], dB[1], dB[2]])
    assert np.abs(ref).max() * N < 2 ** 24 and np.any(ref)
    np.testing.assert_allclose(net.grads().astype(np.float64), ref, rtol=1.3e-7, atol=0.0)
    net.close()
