"""The multigrid V-cycle that preconditions the pressure solve, written out with sparse matrices in FP64.

Unknowns of a level are the connected parts of the 2x2x2 blocks of positions of the level below (links inside the block
join), the operators are the Galerkin sums under piecewise constant transfer, and the smoother is red-black Gauss-Seidel
by the parity of a position.  Where a periodic axis has an odd number of positions its seam joins two of one colour: these
take each other's values from before the half-sweep, so that a half-sweep is one simultaneous update of its colour and the
sweeps before and after the coarse correction stay adjoint to one another.

Coarse diagonals enter through their reciprocal rounded to FP32, as the library stores it.
"""
import numpy as np
from scipy.sparse import coo_matrix, csr_matrix
from scipy.sparse.csgraph import connected_components

PERIODIC, OUTFLOW = 0, 2


class Level:
    """Off-diagonal conductances W, Dirichlet term d, colour and position of every unknown."""

    def __init__(self, W, d, pos, dims):
        self.W, self.d, self.pos, self.dims = W, d, pos, dims
        self.n = W.shape[0]
        self.dg = np.asarray(W.sum(1)).ravel() + d
        self.colour = pos.sum(1) & 1
        self.rows = [np.flatnonzero(self.colour == c) for c in (0, 1)]
        self.Wc = [W[r] for r in self.rows]


def fine_level(shape, bc, flags=None):
    nx, ny, nz = shape
    N = nx * ny * nz
    f = np.zeros((nz, ny, nx), np.uint8) if flags is None else flags.reshape(nz, ny, nx)
    idx = np.arange(N).reshape(nz, ny, nx)
    d = np.zeros((nz, ny, nx))
    r, c = [], []
    for a, dim in ((0, 2), (1, 1), (2, 0)):
        n = shape[a]
        take = lambda v, k: np.take(v, k, dim).ravel()  # noqa: E731
        lo, hi = np.arange(n - 1), np.arange(1, n)
        open_ = (take(f, lo) >> (2 * a + 1) & 1) == 0
        pairs = [(take(idx, lo)[open_], take(idx, hi)[open_])]
        if bc[2 * a] == PERIODIC:
            assert n > 1
            pairs.append((take(idx, [n - 1]), take(idx, [0])))
        for p, q in pairs:
            r += [p, q]
            c += [q, p]
        for s, k in ((0, 0), (1, n - 1)):
            if bc[2 * a + s] == OUTFLOW:
                at = [slice(None)] * 3
                at[dim] = k
                d[tuple(at)] += 2.0
    r, c = np.concatenate(r), np.concatenate(c)
    W = coo_matrix((np.ones(len(r)), (r, c)), shape=(N, N)).tocsr()
    pos = np.stack([idx.ravel() % nx, idx.ravel() // nx % ny, idx.ravel() // (nx * ny)], 1)
    return Level(W, d.ravel(), pos, shape)


def coarsen(F):
    """(next level, parent of every unknown)."""
    up = F.pos >> 1
    dims = tuple((n + 1) // 2 for n in F.dims)
    key = up[:, 0] + dims[0] * (up[:, 1] + dims[1] * up[:, 2])
    A = F.W.tocoo()
    inside = key[A.row] == key[A.col]
    n, parent = connected_components(csr_matrix((A.data[inside], (A.row[inside], A.col[inside])), shape=A.shape), directed=False)
    out = parent[A.row] != parent[A.col]
    W = coo_matrix((A.data[out], (parent[A.row[out]], parent[A.col[out]])), shape=(n, n)).tocsr()
    pos = np.zeros((n, 3), np.int64)
    pos[parent] = up
    return Level(W, np.bincount(parent, F.d, n), pos, dims), parent


class VCycle:
    def __init__(self, shape, bc, flags=None, dx=1.0, sweeps=2, omega=1.6, coarse_sweeps=8, target=1024):
        self.scale, self.sweeps, self.omega, self.coarse_sweeps = dx * dx, sweeps, omega, coarse_sweeps
        self.lev, self.parent = [fine_level(shape, bc, flags)], []
        while (F := self.lev[-1]).n > target and max(F.dims) > 1:
            C, parent = coarsen(F)
            if len(self.lev) > 1 and (C.n > F.n * 4 // 5 or np.diff(C.W.indptr).max() > 64):
                break
            self.lev.append(C)
            self.parent.append(parent)
        for k, v in enumerate(self.lev):
            inv = np.zeros(v.n)
            np.divide(1.0, v.dg, out=inv, where=v.dg > 0)
            v.inv = inv if k == 0 else inv.astype(np.float32).astype(np.float64)

    @staticmethod
    def half(L, c, x, b):
        x[L.rows[c]] = (L.Wc[c] @ x - b[L.rows[c]]) * L.inv[L.rows[c]]

    def coarse(self, k, b):
        L = self.lev[k]
        x = np.zeros(L.n)
        if k == len(self.lev) - 1:
            for q in range(4 * self.coarse_sweeps):
                self.half(L, (q & 1) ^ (q // (2 * self.coarse_sweeps)), x, b)
            return x
        self.half(L, 0, x, b)
        self.half(L, 1, x, b)
        x += self.omega * self.correction(k, b - (L.W @ x - L.dg * x))
        self.half(L, 1, x, b)
        self.half(L, 0, x, b)
        return x

    def correction(self, k, res):
        return self.coarse(k + 1, np.bincount(self.parent[k], res, self.lev[k + 1].n))[self.parent[k]]

    def __call__(self, r):
        L = self.lev[0]
        b = self.scale * r
        z = np.zeros(L.n)
        for _ in range(self.sweeps):
            self.half(L, 0, z, b)
            self.half(L, 1, z, b)
        if len(self.lev) > 1:
            z += self.omega * self.correction(0, b - (L.W @ z - L.dg * z))
        for _ in range(self.sweeps):
            self.half(L, 1, z, b)
            self.half(L, 0, z, b)
        return z
