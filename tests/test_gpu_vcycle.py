"""One V-cycle of the library against its FP64 definition (oracle/multigrid.py): the numbering, the padded and the long
rows, the parents and children of every level, whether it runs in the one-launch tail, in kernels of its own or in the
single block for a coarsest level that does not fit the tail, with even and odd numbers of positions along periodic axes.

FP64: about a hundred dependent operations of 2^-53 per value, 1e-12 of the result's norm with room.  FP32: the same
count of 2^-24, and the residuals that a smoothed colour keeps to rounding only, 2e-5."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

CHANNEL = (1, 2, 3, 3, 3, 3)
BOX = (0,) * 6


@pytest.fixture(scope="module")
def L():
    from paper_2002_06206_gb300 import build
    build.build()
    from paper_2002_06206_gb300 import ibmles
    ibmles.lib()
    return ibmles


def vcycle(L, shape, bc, prec, r, soup=None, **kw):
    g = L.make_grid(*shape, dx=0.5)
    geo = None if soup is None else L.Geometry(g, torch.from_numpy(soup).cuda())
    s = L.Solver(g, 0.01, 0.2, bc, precision=prec, geometry=geo, precond=L.MULTIGRID, **kw)
    r = r.to("cuda", s.dtype)
    z = [torch.full_like(r, 5.0) for _ in range(2)]
    for v in z:
        s.precond(r, v)
    assert torch.equal(z[0], z[1])                 # no value depends on the order of the threads
    flags = None if geo is None else geo.flags.cpu().numpy()
    info = s.mg_info()
    s.close()
    return z[0].cpu().numpy().astype(np.float64), flags, info


def walls(shape):
    """Two triangles over every second face plane of each axis, one more along x: pockets of one to eight cells."""
    out = []
    for a, n in enumerate(shape):
        b, c = (a + 1) % 3, (a + 2) % 3
        for k in range(1, n, 1 if a == 0 else 2):
            q = np.zeros((4, 3))
            q[:, a] = k + 0.01
            q[:, b] = np.array([-1, 1, 1, -1]) * 2 * shape[b]
            q[:, c] = np.array([-1, -1, 1, 1]) * 2 * shape[c]
            out += [q[[0, 1, 2]], q[[0, 2, 3]]]
    return np.array(out, np.float32)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("body", ["none", "soup", "walls"])
@pytest.mark.parametrize("shape,bc", [
    ((131, 61, 47), CHANNEL),                      # first levels in kernels of their own, the others in the tail
    ((64, 32, 32), CHANNEL), ((20, 18, 9), (2, 2, 4, 2, 2, 1)),
    ((40, 32, 24), (1, 2, 0, 0, 3, 3)),            # periodic, every level even
    ((24, 22, 14), (1, 2, 0, 0, 0, 0)),            # odd coarsest level
    ((44, 44, 20), (0, 0, 0, 0, 3, 3)),
    ((60, 52, 44), BOX),                           # odd level in the tail
    ((62, 58, 50), BOX),                           # odd level 1 in kernels of its own, odd levels in the tail
    ((37, 33, 29), BOX), ((36, 33, 28), (1, 2, 0, 0, 0, 0)),   # odd grids: rows of any length, of whole quads
    ((9, 7, 5), BOX), ((12, 7, 8), BOX)])          # the fine grid alone
def test_one_vcycle_is_its_definition(L, shape, bc, body, prec):
    import workloads as W
    from oracle.multigrid import VCycle
    soup = {"none": None, "walls": walls(shape),
            "soup": W.random_soup(60, (0.5, 0.5, 0.5), tuple(n - 0.5 for n in shape), 5.0, seed=8).astype(np.float32)}[body]
    rng = np.random.default_rng(4)
    r = torch.from_numpy(rng.standard_normal(int(np.prod(shape))).astype(np.float32))
    z, flags, info = vcycle(L, shape, bc, prec, r, soup)
    V = VCycle(shape, bc, flags, dx=0.5)
    assert info[0] == len(V.lev) and list(info[2]) == [v.n for v in V.lev]
    ref = V(r.numpy().astype(np.float64))
    assert np.linalg.norm(z - ref) <= (2e-5 if prec else 1e-12) * np.linalg.norm(ref)


def dense_vcycle(r, n, omega):
    """The same on a closed box without a body whose extents are multiples of the blocks: r [nz, ny, nx] on the device in
    FP64, `n` levels."""
    def neighbours(x, g):
        s = torch.zeros_like(x)
        for d in range(3):
            m = x.shape[d] - 1
            s.narrow(d, 0, m).add_(x.narrow(d, 1, m), alpha=g)
            s.narrow(d, 1, m).add_(x.narrow(d, 0, m), alpha=g)
        return s

    def level(b, l):
        g = 4.0 ** l
        dg = neighbours(torch.ones_like(b), g)
        inv = 1.0 / dg if l == 0 else (1.0 / dg).float().double()
        par = sum(torch.arange(m, device=b.device).view([-1 if d == e else 1 for e in range(3)]) for d, m in enumerate(b.shape)) & 1
        x = torch.zeros_like(b)

        def half(c):
            x.copy_(torch.where(par == c, (neighbours(x, g) - b) * inv, x))
        if l == n - 1:
            for q in range(32):
                half((q & 1) ^ (q // 16))
            return x
        sweeps = 2 if l == 0 else 1
        for _ in range(sweeps):
            half(0)
            half(1)
        res = b - (neighbours(x, g) - dg * x)
        s = [m // 2 for m in b.shape]
        xc = level(res.view(s[0], 2, s[1], 2, s[2], 2).sum((1, 3, 5)), l + 1)
        x.view(s[0], 2, s[1], 2, s[2], 2).add_(xc.view(s[0], 1, s[1], 1, s[2], 1), alpha=omega)
        for _ in range(sweeps):
            half(1)
            half(0)
        return x

    return level(r, 0)


@pytest.mark.parametrize("prec", [0, 1])
def test_levels_whose_conductances_are_no_bytes(L, prec):
    """Blocks of 16^3 cells share 256 faces: the rows of a level of more than 16384 such blocks are read as floats."""
    shape = (576, 512, 256)
    gen = torch.Generator(device="cuda").manual_seed(2)
    r = torch.randn(int(np.prod(shape)), generator=gen, device="cuda")
    z, _, info = vcycle(L, shape, (3,) * 6, prec, r)
    M = list(info[2])
    assert M[4] == 36 * 32 * 16 and info[0] == 7
    ref = dense_vcycle(r.double().view(256, 512, 576) * 0.25, 7, 1.6).flatten()
    assert float((torch.from_numpy(z).cuda() - ref).norm()) <= (2e-5 if prec else 1e-12) * float(ref.norm())


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shape,bc", [((37, 33, 29), BOX), ((36, 33, 28), (1, 2, 0, 0, 0, 0)), ((62, 58, 50), BOX), ((44, 44, 20), (0, 0, 0, 0, 3, 3))])
def test_solves_on_grids_whose_seams_join_a_colour(L, shape, bc, prec):
    """The V-cycle inside the replayed iteration: a symmetric preconditioner of this strength takes about a digit per two
    iterations (the oracle's takes at most 12 to 1e-8 on smaller boxes)."""
    import workloads as W
    g = L.make_grid(*shape)
    soup = W.random_soup(40, (0.5, 0.5, 0.5), tuple(n - 0.5 for n in shape), 5.0, seed=8).astype(np.float32)
    geo = L.Geometry(g, torch.from_numpy(soup).cuda())
    s = L.Solver(g, 0.01, 0.2, bc, precision=prec, geometry=geo, precond=L.MULTIGRID)
    x = torch.from_numpy(np.random.default_rng(7).standard_normal(int(np.prod(shape)))).cuda()
    b, r, p = torch.empty_like(x), torch.empty_like(x), torch.zeros_like(x)
    s.apply(x, b)
    st = s.solve(b, p, 1e-8, 400)
    s.apply(p, r)
    assert st.status == 0 and float((b - r).norm()) <= 1.001e-8 * float(b.norm())
    assert st.iters <= 40, st.iters
    s.close()
