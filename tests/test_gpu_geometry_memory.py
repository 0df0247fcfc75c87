"""The memory of geometry handles: it is given back on request and found again by every thread."""
from concurrent.futures import ThreadPoolExecutor

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


def test_destroyed_geometries_leave_nothing_after_a_trim(L):
    import workloads as W
    shape = (512, 512, 256)                        # a table of 256 MiB
    soup = torch.from_numpy(W.icosphere(2, 20.0, (100.3, 99.8, 80.1)).astype(np.float32)).cuda()
    L.Geometry(L.make_grid(32, 32, 32), soup).close()
    torch.cuda.empty_cache()
    L.trim()
    L.trim()                                       # nothing left is no error
    free = torch.cuda.mem_get_info()[0]
    geo = L.Geometry(L.make_grid(*shape), soup)
    geo.close()
    del geo
    torch.cuda.empty_cache()
    kept = free - torch.cuda.mem_get_info()[0]
    L.trim()
    left = free - torch.cuda.mem_get_info()[0]
    assert kept >= 4 * 512 * 512 * 256 and left <= kept // 8, (kept, left)


def test_geometries_of_several_threads_with_trims_between(L):
    """Each worker's errors are its result's."""
    import workloads as W
    shapes = [(40, 30, 20), (64, 64, 64), (9, 8, 7)]
    soups = [torch.from_numpy(W.random_soup(80, (1, 1, 1), tuple(n - 1 for n in s), 4.0, seed=3).astype(np.float32)).cuda()
             for s in shapes]

    def tables(q):
        geo = L.Geometry(L.make_grid(*shapes[q]), soups[q])
        out = [v.cpu().numpy() for v in geo.export()]
        geo.close()
        return out

    first = [tables(q) for q in range(3)]

    def work(seed):
        done = 0
        with torch.cuda.stream(torch.cuda.Stream()):
            for n in range(8):
                q = (seed + n) % 3
                assert all(np.array_equal(a, b) for a, b in zip(tables(q), first[q]))
                if n % 3 == seed:
                    L.trim()
                done += 1
        return done

    with ThreadPoolExecutor(4) as ex:
        assert [f.result() for f in [ex.submit(work, s) for s in range(4)]] == [8] * 4
