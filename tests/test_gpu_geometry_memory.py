"""The memory of geometry handles: it is given back on request, found again by every thread, and a new one is made when the
context it belonged to is gone."""
import ctypes as C
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


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


CHILD = r"""
import ctypes as C, glob, sys
import numpy as np
sys.path.insert(0, ".")
import workloads as W
lib = C.CDLL("paper_2002_06206_gb300/libibmles.so")
lib.ibm_classify_workspace_bytes.restype = C.c_size_t
lib.ibm_last_error.restype = C.c_char_p
rt = C.CDLL(sys.argv[1])
i32, i64, f64, size = C.c_int32, C.c_int64, C.c_double, C.c_size_t
class Grid(C.Structure):
    _fields_ = [("n", i32 * 4), ("dx", f64)]
class GP(C.Structure):
    _fields_ = [("eps", f64 * 2), ("on", i32 * 2)]
g, gp, N, cap = Grid((i32 * 4)(40, 24, 20, 0), 1.0), GP((f64 * 2)(1e-9, 0.0), (i32 * 2)(0, 0)), 40 * 24 * 20, 4096
tri = np.ascontiguousarray(W.icosphere(2, 5.2, (13.3, 11.8, 10.1)), np.float32)
def malloc(n):
    p = C.c_void_p()
    assert rt.cudaMalloc(C.byref(p), size(n)) == 0
    return p
def once():
    d, f = malloc(tri.nbytes), malloc(N)
    assert rt.cudaMemcpy(d, C.c_void_p(tri.ctypes.data), size(tri.nbytes), 1) == 0
    ws = lib.ibm_classify_workspace_bytes(C.byref(g), i64(len(tri)))
    w, fid, lo, hi, n, t, h = malloc(ws), malloc(8 * cap), malloc(8 * cap), malloc(8 * cap), i64(), i64(), C.c_void_p()
    assert lib.ibm_classify(C.byref(g), d, i64(len(tri)), C.byref(gp), f, fid, lo, hi, i64(cap), C.byref(n), C.byref(t), w, size(ws),
                            None) == 0, lib.ibm_last_error()
    assert lib.ibm_setup(C.byref(g), C.byref(gp), f, fid, lo, hi, n, C.byref(h), None) == 0, lib.ibm_last_error()
    return n.value, h
for _ in range(3):
    for _ in range(2):
        n, h = once()
        assert n == 498
        lib.ibm_geom_destroy(h)
    assert lib.ibm_geom_trim() == 0
    assert rt.cudaDeviceReset() == 0
print("ok")
"""


def test_a_device_reset_between_geometries():
    """A process of its own: cudaDeviceReset ends its context and nothing else."""
    import glob
    runtime = sorted(glob.glob("/usr/local/cuda/lib64/libcudart.so.1*"))
    if not runtime:
        pytest.skip("no shared CUDA runtime")
    r = subprocess.run([sys.executable, "-c", CHILD, runtime[0]], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
