"""Classification where FP32 cannot hold what the FP64 predicate decides on: every flag, cut face and position is the
oracle's, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def L():
    from paper_2002_06206_gb300 import build
    build.build()
    from paper_2002_06206_gb300 import ibmles
    ibmles.lib()
    return ibmles


def same_as_the_oracle(L, shape, soup, **eps):
    import oracle
    geo = L.Geometry(L.make_grid(*shape), torch.from_numpy(soup).cuda(), **eps)
    ref = oracle.Case(*shape)
    ref.classify(soup, **eps)
    assert geo.n_cut == len(ref.cut[0]) > 0
    assert np.array_equal(geo.flags.cpu().numpy() & 63, ref.flags & 63)
    for a, b in zip((geo.face_id, geo.t_lo, geo.t_hi), ref.cut):
        assert np.array_equal(a.cpu().numpy(), b)
    geo.close()


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_lines_beyond_the_whole_numbers_of_fp32(L, axis):
    """From 2^23 on j + 1/2 is no FP32 number.  Triangles of a few cells there, and a few below."""
    n = (1 << 23) + 40
    shape = [2, 2, 2]
    shape[axis] = n
    rng = np.random.default_rng(4)
    tri = rng.uniform(-0.2, 2.2, (400, 3, 3))
    tri[:, :, axis] = rng.integers(n - 38, n, (400, 1)) + rng.integers(-1, 2, (400, 3))
    tri[:40, :, axis] -= n // 2
    same_as_the_oracle(L, tuple(shape), tri.astype(np.float32))


@pytest.mark.parametrize("eps", [-0.3, -0.05, -1e-9, 0.0, 0.02, 5.0])
def test_edge_tolerances_of_either_sign(L, eps):
    """A negative tolerance keeps the inner part of a triangle, a large one reaches beyond it.  Small triangles with
    lines at any distance from their edges, and large ones."""
    import workloads as W
    shape = (40, 36, 33)
    soup = np.concatenate([W.random_soup(4000, (0, 0, 0), shape, 2.5, seed=3), W.random_soup(40, (0, 0, 0), shape, 30.0, seed=4)])
    same_as_the_oracle(L, shape, soup.astype(np.float32), eps_edge=eps)
