"""The velocity correction on pressures whose differences are small beside their size: a large constant, as a sealed
pocket or a closed box is free to have, must not cost the differences any bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

CLOSED = (3, 3, 3, 3, 4, 3)
PERIODIC = (0, 0, 0, 0, 0, 0)


@pytest.fixture(scope="module")
def L():
    from paper_2002_06206_gb300 import build
    build.build()
    from paper_2002_06206_gb300 import ibmles
    ibmles.lib()
    return ibmles


@pytest.mark.parametrize("bc", [CLOSED, PERIODIC])
@pytest.mark.parametrize("size,step", [(0.0, 1.0), (1e3, 1e-4), (1e6, 1e-5), (-3e9, 1e-3), (2.0, 2.0 ** -50), (4096.0, 1e-11)])
@pytest.mark.parametrize("shape", [(33, 9, 17), (64, 40, 5), (1, 3, 2)])
def test_differences_of_large_pressures_are_the_fp64_differences_rounded_once(L, shape, size, step, bc):
    """u* = U* = 0, so u = -c (p+ - p-) and U = -2 c (pR - pL): the FP64 difference rounded to FP32 and its product with
    the factor rounded, 2^-24 each, and 2^-53 of the difference where it is not exact."""
    nx, ny, nz = shape
    N = nx * ny * nz
    rng = np.random.default_rng(8)
    p = size + step * rng.standard_normal(N)
    dt = 0.2
    s = L.Solver(L.make_grid(nx, ny, nz), 0.01, dt, bc, precision=L.FP32_REFINE64)
    z = torch.zeros(3 * N, dtype=torch.float32, device="cuda")
    Z = torch.zeros(s.NF, dtype=torch.float32, device="cuda")
    u, U = torch.full_like(z, 7.0), torch.full_like(Z, 7.0)
    s.correct(z, Z, torch.from_numpy(p).cuda(), u, U)
    s.close()
    P = p.reshape(nz, ny, nx)
    off = 0
    for a, dim in ((0, 2), (1, 1), (2, 0)):
        n = P.shape[dim]
        ends = [-1, 0] if bc[2 * a] == 0 else [0, -1]
        E = np.concatenate([np.take(P, [ends[0]], dim), P, np.take(P, [ends[1]], dim)], dim)
        cut = lambda q0, q1: np.take(E, np.arange(q0, q1), dim)  # noqa: E731
        for got, d, c in ((u[a * N:(a + 1) * N], cut(2, n + 2) - cut(0, n), dt / 2), (U[off:off + (n + 1) * (N // n)], cut(1, n + 2) - cut(0, n + 1), dt)):
            ref = -float(np.float32(c)) * d
            got = got.cpu().numpy().astype(np.float64).reshape(ref.shape)
            assert np.all(np.abs(got - ref) <= (2.0 + 2.0 ** -20) * 2.0 ** -24 * np.abs(ref))
        off += (n + 1) * (N // n)
