// mg.cu -- geometric multigrid V-cycle used as the preconditioner of CG for the pressure Poisson
// equation (Eq. poisson).  The paper solves it with BiCGStab or red-black SOR; red-black Gauss-Seidel
// is the smoother here.
//
// Level 0 is the fine grid: the conductance of a link is 1 when its face is uncut and inside the
// domain (or across a periodic seam), 0 otherwise, and an outflow face adds 2 to the diagonal (ghost
// -p).  A position of level l >= 1 is a block of 2x2x2 positions of level l - 1, and its unknowns are
// the connected parts of that block: unknowns of level l - 1 inside the block joined by their links
// inside the block.  So an aggregate never spans a wall -- a block cut in two by a thin plate gives
// two coarse unknowns, and a sealed pocket (the inside of a closed part of the soup) never merges
// with its surroundings on any level.  (Aggregating whole blocks instead joins the two sides of every
// wall on the coarse levels; on a dirty multi-part soup that costs several times the iterations.)
// With piecewise-constant prolongation P and restriction R = P^T the Galerkin coarse operator R A P
// is again a weighted graph Laplacian plus the outflow terms: the conductance between two coarse
// unknowns is the sum of the fine conductances between their aggregates.  Links join only
// face-neighbouring positions, so the parity of a position two-colours every level without an odd number of positions
// (three or more) along a periodic axis.  On an `odd` level the seam joins positions of one colour; a half-sweep then
// takes the values its own colour had before it (one simultaneous update of the colour), so the sweeps before and after
// the correction stay adjoint and no thread reads what another writes.  The V-cycle
// (pre-smoothing red then black, post-smoothing black then red, the coarse correction scaled by
// omega < 2, symmetric sweeps on the coarsest level) is a symmetric operator, as CG requires.
//
// Equations are solved in the unscaled form  sum_links g (x_N - x_P) - d x_P = dx^2 r.
#include <cooperative_groups.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "scan.cuh"
#include "solver.cuh"

namespace cg = cooperative_groups;

// Levels first .. nlev - 1 of the one-launch tail (see k_mg_tail), with each level's share of a block.
struct MGTailLev {
    int M, M0;               // unknowns; the first M0 have colour 0
    int odd;                 // links within a colour
    int s0, s1;              // unknowns of either colour per block (all of them for the coarsest: block 0)
    unsigned i0, i1;         // floor(2^32 / s) + 1
    int x, b, t;             // byte offsets of its arrays in shared memory: iterate, right-hand side, residual,
    int col, pc, g, dg, d;   // neighbours' places, their parents' places, conductances, 1 / dg, Dirichlet term,
    int cv, ch;              // children of its unknowns (start | count << 18, places on the level below),
    int oc, op, og;          // links of rows longer than MG_ELL: places, parents' places, conductances
};
struct MGTail {
    MGTailLev t[IBM_MG_MAXLEV];
    MGLev lev[IBM_MG_MAXLEV];
    int first, nlev, coarse_sweeps;
    int ctas, shift;         // blocks of the cluster; a place is block << shift | index
    int image;               // bytes of a block's constant arrays (the first in its shared memory)
    const uint4* img;        // their image in global memory, block after block
    double omega;
};

namespace {

#define MG_TAIL_BIG 16          // blocks of the tail's cluster where the GPU can hold it; 8, the portable size, elsewhere
#define MG_TAIL_MAX (1LL << 14) // levels with at most this many unknowns run in the one-launch tail
#define MG_COARSE_TARGET 1024   // coarsening stops at this many unknowns (or one position)
#define MG_ELL 6                // links of an unknown kept in the padded rows (more: its CSR row)
#define MG_MAXL 64              // distinct neighbours of a coarse unknown (more: the level is dropped)
#define MG_L1L 24               // level 1: a 2x2x2 block has at most 24 links leaving it

__device__ __forceinline__ unsigned flags_at(const Dom& D, long long P) { return D.flags ? (unsigned)D.flags[P] : 0u; }


// Cell coordinates from a linear index (grids hold fewer than 2^31 cells: 32-bit division).
__device__ __forceinline__ void coords3(long long c, int nx, int ny, int x[3]) {
    const unsigned u = (unsigned)c, unx = (unsigned)nx, uny = (unsigned)ny;
    const unsigned r = u / unx;
    x[0] = (int)(u - r * unx);
    const unsigned z = r / uny;
    x[1] = (int)(r - z * uny);
    x[2] = (int)z;
}


__device__ __forceinline__ long long pos_index(const MGLev& L, const int X[3]) {
    return X[0] + (long long)L.px * (X[1] + (long long)L.py * X[2]);
}

// ---- fine-grid smoothing ----------------------------------------------------------------------

// Gauss-Seidel value of a fine cell:  z_P = (sum_links z_N - scale r_P) / dg, 0 for an isolated cell (dg = 0).
template <class T>
__device__ __forceinline__ T gs_value(const Dom& D, const T* __restrict__ r, const T* z, T scale, long long P, int i,
                                      int j, int k, bool zero) {
    const CellLinks L = cell_links(D, i, j, k, flags_at(D, P));
    const int dg = __popc(L.open) + 2 * __popc(L.out);
    const T s = zero ? (T)0 : open_sum<T>(L, P, [&](long long c) { return z[c]; });
    return dg == 0 ? (T)0 : over_num<T>(s - scale * r[P], dg);
}

// One red-black Gauss-Seidel pass of colour `col` on level 0 for  A^ z = scale * r.  Each thread takes KU pairs of
// planes of one (i, j) column and updates the cell of colour `col` in each pair.  With `zero` the iterate is taken
// as 0 (first pass of a V-cycle) and the other cell of each pair is cleared.  zin: the iterate before the pass (z itself
// unless the grid is odd).  Small grids are bound by latency: 64 x 32 x 32 in FP64 takes 2.7 us with one pair per
// thread, 9.5 us with four and an FP64 division at every domain face.
template <class T, int KU>
__global__ void __launch_bounds__(256) k_mg_smooth0(Dom D, const T* __restrict__ r, T* z, const T* zin, T scale,
                                                    int col, int zero, const SolveScal* sc) {
    if (sc->done) return;
    const int i = blockIdx.x * IBM_TX + threadIdx.x, j = blockIdx.y * IBM_TY + threadIdx.y;
    if (i >= D.nx || j >= D.ny) return;
    const int kb = blockIdx.z * (2 * KU);
    const int par = (col + i + j) & 1;
#pragma unroll
    for (int u = 0; u < KU; ++u) {
        const int k = kb + 2 * u + par;
        const long long P = i + (long long)D.sy * j + D.sz * k;
        if (k < D.nz) z[P] = gs_value<T>(D, r, zin, scale, P, i, j, k, zero != 0);
        if (zero) {
            const int k2 = kb + 2 * u + (par ^ 1);
            if (k2 < D.nz) z[i + (long long)D.sy * j + D.sz * k2] = (T)0;
        }
    }
}

// Last pass of the V-cycle on level 0 (colour 0) fused with rho = (r, z) over both colours.
template <class T, int KU>
__global__ void __launch_bounds__(256) k_mg_final0(Dom D, const T* __restrict__ r, T* z, const T* zin, T scale,
                                                   SolveScal* sc, double* partials, unsigned* counter) {
    if (sc->done) return;
    const int i = blockIdx.x * IBM_TX + threadIdx.x, j = blockIdx.y * IBM_TY + threadIdx.y;
    const bool active = i < D.nx && j < D.ny;
    const int kb = blockIdx.z * (2 * KU);
    const int par = (i + j) & 1;                 // plane offset of the colour-0 cell in each pair
    T part = 0;
    if (active) {
#pragma unroll
        for (int u = 0; u < KU; ++u) {
            const int k = kb + 2 * u + par, k2 = kb + 2 * u + (par ^ 1);
            if (k < D.nz) {
                const long long P = i + (long long)D.sy * j + D.sz * k;
                const T zv = gs_value<T>(D, r, zin, scale, P, i, j, k, false);
                z[P] = zv;
                part += r[P] * zv;
            }
            if (k2 < D.nz) {
                const long long P2 = i + (long long)D.sy * j + D.sz * k2;
                part += r[P2] * z[P2];
            }
        }
    }
    decltype(part) acc[1] = {part};
    grid_reduce<1>(acc, partials, counter, [&](double* t) {
        sc->rz_old = sc->rz;
        sc->rz = t[0];
    });
}

// ---- parts of a block -----------------------------------------------------------------------------

// Flags of the 2x2x2 fine cells below level-1 position X (cell m = di + 2 dj + 4 dk); bit m of the
// result says that cell m lies inside the domain.  Out-of-domain cells get flags 0.
__device__ __forceinline__ unsigned block_flags(const Dom& D, const int X[3], unsigned (&fl)[8], long long (&P)[8]) {
    unsigned in = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const int x = 2 * X[0] + (m & 1), y = 2 * X[1] + ((m >> 1) & 1), z = 2 * X[2] + (m >> 2);
        const bool ok = x < D.nx && y < D.ny && z < D.nz;
        P[m] = ok ? x + (long long)D.sy * y + D.sz * z : 0;
        fl[m] = ok ? flags_at(D, P[m]) : 0u;
        in |= (ok ? 1u : 0u) << m;
    }
    return in;
}

// Connected parts of a fine block: two in-domain cells of the block are joined when the face between
// them is uncut, or when their axis is periodic with only two cells (the seam joins them too).
// part[m] = the part of cell m, parts numbered in the order of their lowest cell; returns the count.
__device__ __forceinline__ int fine_parts(const Dom& D, const unsigned (&fl)[8], unsigned in, int (&part)[8]) {
    const unsigned cut = ((fl[0] | fl[2] | fl[4] | fl[6]) & 2u) | ((fl[0] | fl[1] | fl[4] | fl[5]) & 8u) |
                         ((fl[0] | fl[1] | fl[2] | fl[3]) & 32u);
    if (in == 0xffu && cut == 0u) {
#pragma unroll
        for (int m = 0; m < 8; ++m) part[m] = 0;
        return 1;
    }
    const bool seam[3] = {D.bc[0] == IBM_BC_PERIODIC && D.nx == 2, D.bc[2] == IBM_BC_PERIODIC && D.ny == 2,
                          D.bc[4] == IBM_BC_PERIODIC && D.nz == 2};
    int lab[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) lab[m] = m;
    // minimum-label propagation; a path through the block has at most 7 links
    for (int it = 0; it < 8; ++it) {
        bool changed = false;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                if (m & (1 << a)) continue;
                const int h = m | (1 << a);
                if (!((in >> m) & 1u) || !((in >> h) & 1u)) continue;
                if ((fl[m] & (2u << (2 * a))) && !seam[a]) continue;
                const int lo = lab[m] < lab[h] ? lab[m] : lab[h];
                if (lab[m] != lo || lab[h] != lo) {
                    lab[m] = lo;
                    lab[h] = lo;
                    changed = true;
                }
            }
        if (!changed) break;
    }
    unsigned roots = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m)
        if (((in >> m) & 1u) && lab[m] == m) roots |= 1u << m;
#pragma unroll
    for (int m = 0; m < 8; ++m) part[m] = __popc(roots & ((1u << lab[m]) - 1u));
    return __popc(roots);
}

// Level-1 right-hand side of unknown u, with the first half-sweep of that level from x = 0.
template <class T>
__device__ __forceinline__ void put_b1(const MGLev& C, int u, T b) {
    ((T*)C.b)[u] = b;
    ((T*)C.x)[u] = -b * (T)C.invdg[u];
}

// ---- fused fine-grid passes: all four red-black half-sweeps of a smoothing phase in one pass ------
//
// A block of 512 threads marches an (x, y) tile along z over a chunk of planes.  A thread owns a column of
// 4 x 2 cells (a 16-byte quad in two rows) and keeps its planes in registers, so the neighbours above and
// below cost nothing; the x neighbours within a quad are registers, across quads one shuffle, the y
// neighbours the other row or, across threads, two values through shared memory.  At step t half-sweep s
// (s = 1 .. 4) runs on plane t - s + 1: its in-plane neighbours were finished in step t - 1 and its upper
// neighbour by half-sweep s - 1 of the same step in the same thread, so one barrier per plane orders
// everything and the four half-sweeps are independent until they meet in the column.  Only the colour
// just updated is published (two float2 per thread and half-sweep, double buffered by step parity); tile
// origins and x quads are even, so which cells of a quad a half-sweep updates depends on the step's parity
// alone and is known to the compiler.  The halo (4 cells) holds values that turn wrong one ring per
// half-sweep from the outside; the tile's own cells see exactly the values of separate passes.  A tile at a
// domain face has no halo there.
//
// Cells with no cut link and off the first and last plane take the plain form (s - scale r) * inv with inv
// = 1 / (open links + outflow terms), fixed per column: neighbours outside the domain hold z = 0.  A warp
// with a cut link in its plane takes the general form for that plane.
//
// Neither issue (65 and 54 % of the active cycles) nor HBM (35 and 39 %) is full: what is left is the latency of one
// barrier per plane with 16 warps on an SM.  512x256x256 under ncu: 132 us (pre) and 149 us (post) for 9.1 and 13 bytes
// per cell; 744 and 585 us with planes in a TMA ring and one barrier per half-sweep.
#define FTP_NT 512
#define FTP_RING 5

template <int LX>
struct FTile {
    static constexpr int W = 4 * LX;               // cells along x, halo included
    static constexpr int NRP = FTP_NT / LX;        // row pairs
    static constexpr int H = 2 * NRP;              // rows, halo included
    static constexpr int EXN = 2 * (NRP + 2) * LX; // float2 of one exchange buffer: two rows of every pair, padded
    static constexpr size_t smem() {
        return (size_t)8 * EXN * sizeof(float2) + (size_t)FTP_RING * FTP_NT * (2 * sizeof(float4) + sizeof(uint2)) +
               16 * sizeof(float);
    }
};

// A thread's column: constants of the march (NI = 3: nx a multiple of 4, else 4).
template <int NI>
struct FCol {
    int xl;                 // quad within the row of the tile
    int gx, gy;             // global coordinates of its first cell
    bool in0, in1;          // rows inside the domain
    bool own0, own1;        // rows of the tile's own cells
    float inv[2][NI];       // 1 / dg per row and cell, 0 outside the domain
    int dg[2][NI];
    // a quad of a grid with nx a multiple of 4 lies inside or outside as a whole: its middle cells share a value
    static __device__ __forceinline__ constexpr int at(int m) { return NI == 4 ? m : (m == 0 ? 0 : (m == 3 ? 2 : 1)); }
};

template <int LX, int NI>
__device__ __forceinline__ FCol<NI> ftp_column(const Dom& D, int tx, int ty, int ntx, int nty) {
    using T = FTile<LX>;
    FCol<NI> c;
    c.xl = threadIdx.x % LX;
    const int rp = threadIdx.x / LX;
    const int X0 = tx * (T::W - 8), Y0 = ty * (T::H - 8);
    c.gx = X0 + 4 * c.xl;
    c.gy = Y0 + 2 * rp;
    const bool inx = c.gx < D.nx;
    c.in0 = inx && c.gy < D.ny;
    c.in1 = inx && c.gy + 1 < D.ny;
    const bool ox = (tx == 0 || c.xl > 0) && (tx == ntx - 1 || c.xl < LX - 1);
    const bool oy = (ty == 0 || rp > 1) && (ty == nty - 1 || rp < T::NRP - 2);
    c.own0 = c.in0 && ox && oy;
    c.own1 = c.in1 && ox && oy;
    auto term = [&](int f) { return D.bc[f] == IBM_BC_OUTFLOW ? 1 : -1; };   // a closed link, plus 2 at an outflow
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int y = c.gy + r;
        const int d = 6 + (y == 0 ? term(2) : 0) + (y == D.ny - 1 ? term(3) : 0);
        const bool in = r ? c.in1 : c.in0;
#pragma unroll
        for (int m = 0; m < NI; ++m) {
            const int x = c.gx + (NI == 3 && m == 2 ? 3 : m);
            c.dg[r][m] = in && x < D.nx ? d + (x == 0 ? term(0) : 0) + (x == D.nx - 1 ? term(1) : 0) : 0;
            c.inv[r][m] = c.dg[r][m] > 0 ? 1.f / (float)c.dg[r][m] : 0.f;
        }
    }
    return c;
}

// Sum of z over the open links of a cell with flags f.
__device__ __forceinline__ float ftp_open_sum(unsigned f, float xm, float xp, float ym, float yp, float zm, float zp) {
    const float sx = ((f & 1u) ? 0.f : xm) + ((f & 2u) ? 0.f : xp);
    const float sy = ((f & 4u) ? 0.f : ym) + ((f & 8u) ? 0.f : yp);
    const float sz = ((f & 16u) ? 0.f : zm) + ((f & 32u) ? 0.f : zp);
    return (sx + sy) + sz;
}

// x neighbours of the cells D0, D0 + 2 of row 0 and 1 - D0, 3 - D0 of row 1 that lie in another quad.
template <int LX, int D0, int NI>
__device__ __forceinline__ void ftp_xside(const FCol<NI>& c, const float (&zc)[2][4], float& e0, float& e1) {
    const float a = D0 == 0 ? __shfl_up_sync(0xffffffffu, zc[0][3], 1) : __shfl_down_sync(0xffffffffu, zc[0][0], 1);
    const float b = D0 == 0 ? __shfl_down_sync(0xffffffffu, zc[1][0], 1) : __shfl_up_sync(0xffffffffu, zc[1][3], 1);
    const bool first = c.xl == 0, last = c.xl == LX - 1;
    e0 = (D0 == 0 ? first : last) ? 0.f : a;
    e1 = (D0 == 0 ? last : first) ? 0.f : b;
}

// The two cells D, D + 2 of row `zr` and their neighbours: calls f(cell, xm, xp, ym, yp, zm, zp, which).
template <int D, class Fn>
__device__ __forceinline__ void ftp_pair(const float (&zr)[4], float e, float ym0, float ym1, float yp0, float yp1,
                                         const float (&zm)[4], const float (&zp)[4], Fn f) {
    f(D, D == 0 ? e : zr[0], zr[D + 1], ym0, yp0, zm[D], zp[D], 0);
    f(D + 2, zr[D + 1], D == 0 ? zr[3] : e, ym1, yp1, zm[D + 2], zp[D + 2], 1);
}

// One half-sweep on a thread's cells of one plane: cells D0, D0 + 2 of row 0 and 1 - D0, 3 - D0 of row 1.
// yb, yt: the rows below and above (another thread's); r0, r1: the right-hand side at the updated cells.
template <int LX, int D0, int NI>
__device__ __forceinline__ void ftp_sweep(const FCol<NI>& c, float (&zc)[2][4], const float (&zm)[2][4], const float (&zp)[2][4],
                                          float2 yb, float2 yt, float2 r0, float2 r1, float scale, bool general,
                                          const uint2* fl, int zadj, const float* rcp) {
    float e0, e1;
    ftp_xside<LX, D0, NI>(c, zc, e0, e1);
    constexpr int D1 = 1 - D0;
    float v0[2], v1[2];
    if (!general) {
        ftp_pair<D0>(zc[0], e0, yb.x, yb.y, zc[1][D0], zc[1][D0 + 2], zm[0], zp[0],
                     [&](int m, float a, float b, float p, float q, float l, float u, int w) {
                         v0[w] = fmaf(-scale, w ? r0.y : r0.x, ((a + b) + (p + q)) + (l + u)) * c.inv[0][FCol<NI>::at(m)];
                     });
        ftp_pair<D1>(zc[1], e1, zc[0][D1], zc[0][D1 + 2], yt.x, yt.y, zm[1], zp[1],
                     [&](int m, float a, float b, float p, float q, float l, float u, int w) {
                         v1[w] = fmaf(-scale, w ? r1.y : r1.x, ((a + b) + (p + q)) + (l + u)) * c.inv[1][FCol<NI>::at(m)];
                     });
    } else {
        const uint2 ff = *fl;
        auto cell = [&](int row, int m, float s, unsigned f, float r) {
            const int d = c.dg[row][FCol<NI>::at(m)];
            return fmaf(-scale, r, s) * rcp[d ? d + zadj - __popc(f & 63u) : 0];
        };
        ftp_pair<D0>(zc[0], e0, yb.x, yb.y, zc[1][D0], zc[1][D0 + 2], zm[0], zp[0],
                     [&](int m, float a, float b, float p, float q, float l, float u, int w) {
                         const unsigned f = ff.x >> (8 * m);
                         v0[w] = cell(0, m, ftp_open_sum(f, a, b, p, q, l, u), f, w ? r0.y : r0.x);
                     });
        ftp_pair<D1>(zc[1], e1, zc[0][D1], zc[0][D1 + 2], yt.x, yt.y, zm[1], zp[1],
                     [&](int m, float a, float b, float p, float q, float l, float u, int w) {
                         const unsigned f = ff.y >> (8 * m);
                         v1[w] = cell(1, m, ftp_open_sum(f, a, b, p, q, l, u), f, w ? r1.y : r1.x);
                     });
    }
    zc[0][D0] = v0[0];
    zc[0][D0 + 2] = v0[1];
    zc[1][D1] = v1[0];
    zc[1][D1 + 2] = v1[1];
}

__device__ __forceinline__ void ftp_zero(float (&z)[2][4]) {
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int m = 0; m < 4; ++m) z[r][m] = 0.f;
}
__device__ __forceinline__ void ftp_copy(float (&a)[2][4], const float (&b)[2][4]) {
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int m = 0; m < 4; ++m) a[r][m] = b[r][m];
}
__device__ __forceinline__ void ftp_set(float (&a)[2][4], float4 x, float4 y) {
    a[0][0] = x.x; a[0][1] = x.y; a[0][2] = x.z; a[0][3] = x.w;
    a[1][0] = y.x; a[1][1] = y.y; a[1][2] = y.z; a[1][3] = y.w;
}

// A quad of a row: 16 bytes where rows start on 16-byte boundaries (NI = 3), cell by cell within the domain.
template <int NI>
__device__ __forceinline__ float4 ftp_load(const float* p, int left) {
    if (NI == 3) return *reinterpret_cast<const float4*>(p);
    return make_float4(p[0], left > 1 ? p[1] : 0.f, left > 2 ? p[2] : 0.f, left > 3 ? p[3] : 0.f);
}
template <int NI>
__device__ __forceinline__ unsigned ftp_load_flags(const uint8_t* p, int left) {
    if (NI == 3) return *reinterpret_cast<const unsigned*>(p);
    return (unsigned)p[0] | (left > 1 ? (unsigned)p[1] << 8 : 0u) | (left > 2 ? (unsigned)p[2] << 16 : 0u) |
           (left > 3 ? (unsigned)p[3] << 24 : 0u);
}
template <int NI>
__device__ __forceinline__ void ftp_store(float* p, int left, const float (&z)[4]) {
    if constexpr (NI == 3) {
        *reinterpret_cast<float4*>(p) = make_float4(z[0], z[1], z[2], z[3]);
    } else {
#pragma unroll
        for (int m = 0; m < 4; ++m)
            if (m < left) p[m] = z[m];
    }
}

// Shared memory of a block and the thread's places in it.
template <int LX>
struct FShared {
    float2* ex;          // [buffer 0 .. 3][step parity][row][pair + 1][quad]
    float4* r;           // [slot][row][thread]: right-hand side, colour 0 then colour 1 (two cells each)
    uint2* f;            // [slot][thread]: flags of the two quads
    float* rcp;          // 1 / n, 0 for n = 0
    int mine;            // index of the thread's pair and quad in a buffer row
    __device__ __forceinline__ float2* at(int b, int par, int row, int dpair) const {
        return ex + ((b * 2 + par) * 2 + row) * ((FTile<LX>::NRP + 2) * LX) + mine + dpair * LX;
    }
    __device__ __forceinline__ void publish(int b, int par, const float (&z)[2][4], int d0) const {
        *at(b, par, 0, 0) = d0 ? make_float2(z[0][1], z[0][3]) : make_float2(z[0][0], z[0][2]);
        *at(b, par, 1, 0) = d0 ? make_float2(z[1][0], z[1][2]) : make_float2(z[1][1], z[1][3]);
    }
    __device__ __forceinline__ float2 below(int b, int par) const { return *at(b, par, 1, -1); }
    __device__ __forceinline__ float2 above(int b, int par) const { return *at(b, par, 0, 1); }
    __device__ __forceinline__ float2 rhs(int slot, int row, int col) const {
        return reinterpret_cast<const float2*>(r + (slot * 2 + row) * FTP_NT + threadIdx.x)[col];
    }
};

template <int LX>
__device__ __forceinline__ FShared<LX> ftp_shared(unsigned char* base) {
    using T = FTile<LX>;
    FShared<LX> S;
    S.ex = reinterpret_cast<float2*>(base);
    S.r = reinterpret_cast<float4*>(S.ex + 8 * T::EXN);
    S.f = reinterpret_cast<uint2*>(S.r + FTP_RING * 2 * FTP_NT);
    S.rcp = reinterpret_cast<float*>(S.f + FTP_RING * FTP_NT);
    S.mine = (threadIdx.x / LX + 1) * LX + threadIdx.x % LX;
    for (int e = threadIdx.x; e < 8 * T::EXN; e += FTP_NT) S.ex[e] = make_float2(0.f, 0.f);
    if (threadIdx.x < 16) S.rcp[threadIdx.x] = threadIdx.x ? 1.f / (float)threadIdx.x : 0.f;
    __syncthreads();
    return S;
}

__device__ __forceinline__ int ftp_back(int slot, int k) { return slot >= k ? slot - k : slot - k + FTP_RING; }

// Extra diagonal of the first and last plane.
__device__ __forceinline__ int ftp_zadj(const Dom& D, int p) {
    return (p == 0 ? (D.bc[4] == IBM_BC_OUTFLOW ? 1 : -1) : 0) + (p == D.nz - 1 ? (D.bc[5] == IBM_BC_OUTFLOW ? 1 : -1) : 0);
}

// Pre-smoothing (from z = 0, colours 0, 1, 0, 1) and the restriction of  scale r - A z  to the parts of the
// level-1 blocks.  Writes z on its chunk's planes [k0, k1) and b_1.  The last half-sweep leaves the residual
// of colour 1 zero, so only colour 0 is evaluated (one plane behind the last half-sweep).
template <int LX, int NI>
__global__ void __launch_bounds__(FTP_NT, 1) k_mg_pre_fused(Dom D, const float* __restrict__ rg, float* __restrict__ zg,
                                                            float scale, MGLev C1, const int4* __restrict__ chunks, int ntx,
                                                            int nty, const SolveScal* sc) {
    if (sc->done) return;
    extern __shared__ __align__(16) unsigned char ftp_raw[];
    const FShared<LX> S = ftp_shared<LX>(ftp_raw);
    const int4 item = chunks[blockIdx.x];       // tile, its planes
    const FCol<NI> c = ftp_column<LX, NI>(D, item.x, item.y, ntx, nty);
    const int left = D.nx - c.gx;       // cells from the quad's first to the end of the row
    const int k0 = item.z, k1 = item.w;
    const int tlo = max(0, k0 - 4), thi = k1 + 3;
    const int row0 = c.gx + D.sy * c.gy;
    float Z[6][2][4];
#pragma unroll
    for (int q = 0; q < 6; ++q) ftp_zero(Z[q]);
    float4 nr0 = make_float4(0.f, 0.f, 0.f, 0.f), nr1 = nr0;
    unsigned nf0 = 0u, nf1 = 0u;
    auto fetch = [&](int t) {
        nr0 = nr1 = make_float4(0.f, 0.f, 0.f, 0.f);
        nf0 = nf1 = 0u;
        if (t >= D.nz) return;
        const long long P = row0 + D.sz * t;
        if (c.in0) {
            nr0 = ftp_load<NI>(rg + P, left);
            if (D.flags) nf0 = ftp_load_flags<NI>(D.flags + P, left);
        }
        if (c.in1) {
            nr1 = ftp_load<NI>(rg + P + D.sy, left);
            if (D.flags) nf1 = ftp_load_flags<NI>(D.flags + P + D.sy, left);
        }
    };
    fetch(tlo);
    unsigned gen = 0u;                  // bit k: plane t - k takes the general form in this warp
    int slot = 0;                       // ring slot of plane t
    float er[2][2] = {{0.f, 0.f}, {0.f, 0.f}};       // residuals of the even plane [row][position]
    // the two positions of level 1: their first unknowns, loaded with the even plane, and 1 / dg, loaded a step later
    // (at the point of use the two loads, one after the other, took a quarter of the pass)
    const bool two = NI == 3 || left > 2;                // the second position lies in the domain
    int2 bo = make_int2(0, 0);
    float2 bi = make_float2(0.f, 0.f);
    auto step = [&](auto par, int t) {
        constexpr int D0 = decltype(par)::value;      // = t & 1
        const int pw = D0, pr = 1 - D0;                // exchange buffers written and read in this step
        // plane t arrives: right-hand side and flags into the ring, colour 0 first
        const float4 c0 = D0 ? make_float4(nr0.y, nr0.w, nr0.x, nr0.z) : make_float4(nr0.x, nr0.z, nr0.y, nr0.w);
        const float4 c1 = D0 ? make_float4(nr1.x, nr1.z, nr1.y, nr1.w) : make_float4(nr1.y, nr1.w, nr1.x, nr1.z);
        S.r[(slot * 2 + 0) * FTP_NT + threadIdx.x] = c0;
        S.r[(slot * 2 + 1) * FTP_NT + threadIdx.x] = c1;
        const uint2 ft = make_uint2(nf0, nf1);
        S.f[slot * FTP_NT + threadIdx.x] = ft;
        gen = (gen << 1) | ((__any_sync(0xffffffffu, ((nf0 | nf1) & 0x3f3f3f3fu) != 0u) || t == 0 || t == D.nz - 1) ? 1u : 0u);
        fetch(t + 1);
        if (c.own0 && t - 4 >= k0 && t - 4 < k1) {
            if (D0 == 0) {
                const int* o = C1.off + (c.gx >> 1) + (long long)C1.px * ((c.gy >> 1) + (long long)C1.py * ((t - 4) >> 1));
                if (NI == 3) bo = *reinterpret_cast<const int2*>(o);
                else bo = make_int2(o[0], two ? o[1] : 0);
            } else {
                bi = make_float2(C1.invdg[bo.x], two ? C1.invdg[bo.y] : 0.f);
            }
        }
        // half-sweep 1 on plane t, from z = 0
        ftp_zero(Z[0]);
        if (t < D.nz) {
            const float q[2][2] = {{-scale * c0.x, -scale * c0.y}, {-scale * c1.x, -scale * c1.y}};
            const int zadj = (gen & 1u) ? ftp_zadj(D, t) : 0;
#pragma unroll
            for (int row = 0; row < 2; ++row)
#pragma unroll
                for (int w = 0; w < 2; ++w) {
                    const int m = (row ? 1 - D0 : D0) + 2 * w, mi = FCol<NI>::at(m);
                    float iv = c.inv[row][mi];
                    if (gen & 1u) {
                        const unsigned f = (row ? ft.y : ft.x) >> (8 * m);
                        const int d = c.dg[row][mi];
                        iv = S.rcp[d ? d + zadj - __popc(f & 63u) : 0];
                    }
                    Z[0][row][m] = q[row][w] * iv;
                }
            S.publish(0, pw, Z[0], D0);
        }
        // half-sweeps 2, 3, 4 on planes t - 1, t - 2, t - 3 (colours 1, 0, 1)
#pragma unroll
        for (int k = 1; k <= 3; ++k) {
            const int p = t - k;
            if (p >= tlo && p < D.nz) {
                const int sl = ftp_back(slot, k);
                const bool g = (gen >> k) & 1u;
                ftp_sweep<LX, D0, NI>(c, Z[k], Z[k + 1], Z[k - 1], S.below(k - 1, pr), S.above(k - 1, pr), S.rhs(sl, 0, k & 1),
                                  S.rhs(sl, 1, k & 1), scale, g, S.f + sl * FTP_NT + threadIdx.x, g ? ftp_zadj(D, p) : 0, S.rcp);
                S.publish(k, pw, Z[k], D0);
            }
        }
        // plane t - 3 is final
        const int tw = t - 3;
        if (tw >= k0 && tw < k1) {
            float* zo = zg + row0 + D.sz * tw;
            if (c.own0) ftp_store<NI>(zo, left, Z[3][0]);
            if (c.own1) ftp_store<NI>(zo + D.sy, left, Z[3][1]);
        }
        // residual of colour 0 on plane t - 4
        const int tr = t - 4;
        if (tr >= k0 && tr < k1) {
            const int sl = ftp_back(slot, 4);
            const bool g = (gen >> 4) & 1u;
            const float2 yb = S.below(3, pr), yt = S.above(3, pr), r0 = S.rhs(sl, 0, 0), r1 = S.rhs(sl, 1, 0);
            float e0, e1;
            ftp_xside<LX, D0, NI>(c, Z[4], e0, e1);
            const uint2 ff = g ? S.f[sl * FTP_NT + threadIdx.x] : make_uint2(0u, 0u);
            const int zadj = g ? ftp_zadj(D, tr) : 0;
            float res[2][2];
            auto cell = [&](int row, int m, float a, float b, float p, float q, float l, float u, float r) {
                int d = c.dg[row][FCol<NI>::at(m)];
                if (NI == 4 && d == 0) return 0.f;                // outside the domain
                float s;
                if (!g) {
                    s = ((a + b) + (p + q)) + (l + u);
                } else {
                    const unsigned f = (row ? ff.y : ff.x) >> (8 * m);
                    s = ftp_open_sum(f, a, b, p, q, l, u);
                    d += zadj - __popc(f & 63u);
                }
                return scale * r - (s - (float)d * Z[4][row][m]);
            };
            constexpr int D1 = 1 - D0;
            ftp_pair<D0>(Z[4][0], e0, yb.x, yb.y, Z[4][1][D0], Z[4][1][D0 + 2], Z[5][0], Z[3][0],
                         [&](int m, float a, float b, float p, float q, float l, float u, int w) {
                             res[0][w] = cell(0, m, a, b, p, q, l, u, w ? r0.y : r0.x);
                         });
            ftp_pair<D1>(Z[4][1], e1, Z[4][0][D1], Z[4][0][D1 + 2], yt.x, yt.y, Z[5][1], Z[3][1],
                         [&](int m, float a, float b, float p, float q, float l, float u, int w) {
                             res[1][w] = cell(1, m, a, b, p, q, l, u, w ? r1.y : r1.x);
                         });
            if (!c.in1) res[1][0] = res[1][1] = 0.f;
            const bool lastp = tr == D.nz - 1;
            if (D0 == 0) {              // an even plane (tr and t have the same parity)
#pragma unroll
                for (int w = 0; w < 2; ++w) {
                    er[0][w] = res[0][w];
                    er[1][w] = res[1][w];
                }
            }
            if ((D0 == 1 || lastp) && c.own0) {
                const int2 o = bo;
                const bool odd = D0 == 1;                // both planes of the block are there
                if (!odd) bi = make_float2(C1.invdg[o.x], two ? C1.invdg[o.y] : 0.f);
                // a warp without a cut link in the two planes: whole blocks
                if (!((gen >> 4) & 1u) && !(odd && ((gen >> 5) & 1u))) {
                    auto put = [&](int u, float b, float inv) {
                        ((float*)C1.b)[u] = b;
                        ((float*)C1.x)[u] = -b * inv;
                    };
                    put(o.x, odd ? (er[0][0] + er[1][0]) + (res[0][0] + res[1][0]) : er[0][0] + er[1][0], bi.x);
                    if (two) put(o.y, odd ? (er[0][1] + er[1][1]) + (res[0][1] + res[1][1]) : er[0][1] + er[1][1], bi.y);
                } else {
                    const long long Pe = row0 + D.sz * (tr & ~1);
                    unsigned fe[2], fo[2];
                    fe[0] = D.flags ? ftp_load_flags<NI>(D.flags + Pe, left) : 0u;
                    fe[1] = D.flags && c.in1 ? ftp_load_flags<NI>(D.flags + Pe + D.sy, left) : 0u;
                    fo[0] = D.flags && odd ? ftp_load_flags<NI>(D.flags + Pe + D.sz, left) : 0u;
                    fo[1] = D.flags && odd && c.in1 ? ftp_load_flags<NI>(D.flags + Pe + D.sz + D.sy, left) : 0u;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h == 1 && !two) break;
                        unsigned fl[8], in = 0;
                        float rv[8];
#pragma unroll
                        for (int m = 0; m < 8; ++m) {
                            const int di = m & 1, dj = (m >> 1) & 1, dk = m >> 2;
                            const bool ok = (dj == 0 || c.in1) && (dk == 0 || odd) && (NI == 3 || 2 * h + di < left);
                            fl[m] = ok ? ((dk ? fo[dj] : fe[dj]) >> (8 * (2 * h + di))) & 0xffu : 0u;
                            in |= (ok ? 1u : 0u) << m;
                            // colour 0: x + y + z even within the block
                            rv[m] = ((di + dj + dk) & 1) ? 0.f : (dk ? res[dj][h] : er[dj][h]);
                        }
                        int part[8];
                        const int np = fine_parts(D, fl, in, part);
                        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int m = 0; m < 8; ++m)
#pragma unroll
                            for (int s2 = 0; s2 < 8; ++s2) acc[s2] += (((in >> m) & 1u) && part[m] == s2) ? rv[m] : 0.f;
                        const int oo = h ? o.y : o.x;
#pragma unroll
                        for (int s2 = 0; s2 < 8; ++s2)
                            if (s2 < np) put_b1<float>(C1, oo + s2, acc[s2]);
                    }
                }
            }
        }
#pragma unroll
        for (int q = 5; q > 0; --q) ftp_copy(Z[q], Z[q - 1]);
        slot = slot == FTP_RING - 1 ? 0 : slot + 1;
        __syncthreads();
    };
    for (int t = tlo; t <= thi; t += 2) {
        step(std::integral_constant<int, 0>{}, t);
        step(std::integral_constant<int, 1>{}, t + 1);
    }
}

// Post-smoothing (colours 1, 0, 1, 0) of the iterate the coarse correction left, read from zin (an array
// this pass does not write: neighbouring tiles read each other's cells), into z; then (r, z) over the grid:
// rz_old = rz, rz = (r, z).
template <int LX, int NI>
__global__ void __launch_bounds__(FTP_NT, 1) k_mg_post_fused(Dom D, const float* __restrict__ rg, const float* __restrict__ zin,
                                                             float* __restrict__ zg, float scale, const int4* __restrict__ chunks,
                                                             int ntx, int nty, SolveScal* sc,
                                                             double* partials, unsigned* counter) {
    if (sc->done) return;
    extern __shared__ __align__(16) unsigned char ftp_raw[];
    const FShared<LX> S = ftp_shared<LX>(ftp_raw);
    const int4 item = chunks[blockIdx.x];       // tile, its planes
    const FCol<NI> c = ftp_column<LX, NI>(D, item.x, item.y, ntx, nty);
    const int left = D.nx - c.gx;       // cells from the quad's first to the end of the row
    const int k0 = item.z, k1 = item.w;
    const int tlo = max(0, k0 - 4), thi = k1 + 2;
    const int row0 = c.gx + D.sy * c.gy;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float Z[5][2][4], zn[2][4];          // planes t .. t - 4 and t + 1
    float4 nr0, nr1, nz0, nz1;           // r of plane t + 1 and z of plane t + 2, in flight
    unsigned nf0, nf1;
    auto fetch_r = [&](int t) {
        nr0 = nr1 = zero4;
        nf0 = nf1 = 0u;
        if (t >= D.nz) return;
        const long long P = row0 + D.sz * t;
        if (c.in0) {
            nr0 = ftp_load<NI>(rg + P, left);
            if (D.flags) nf0 = ftp_load_flags<NI>(D.flags + P, left);
        }
        if (c.in1) {
            nr1 = ftp_load<NI>(rg + P + D.sy, left);
            if (D.flags) nf1 = ftp_load_flags<NI>(D.flags + P + D.sy, left);
        }
    };
    auto fetch_z = [&](int t) {
        nz0 = nz1 = zero4;
        if (t >= D.nz) return;
        const long long P = row0 + D.sz * t;
        if (c.in0) nz0 = ftp_load<NI>(zin + P, left);
        if (c.in1) nz1 = ftp_load<NI>(zin + P + D.sy, left);
    };
#pragma unroll
    for (int q = 1; q < 5; ++q) ftp_zero(Z[q]);
    fetch_z(tlo);
    ftp_set(Z[0], nz0, nz1);
    // colour 0 of plane tlo, read by step tlo (even) from the buffers of odd steps
    S.publish(0, 1, Z[0], 0);
    fetch_z(tlo + 1);
    ftp_set(zn, nz0, nz1);
    fetch_z(tlo + 2);
    fetch_r(tlo);
    __syncthreads();
    unsigned gen = 0u;
    int slot = 0;
    float part = 0.f;
    auto step = [&](auto par, int t) {
        constexpr int PT = decltype(par)::value;      // t & 1
        constexpr int D0 = 1 - PT;                    // cells of row 0 the step's half-sweeps update
        const int pw = PT, pr = 1 - PT;
        const float4 c0 = PT ? make_float4(nr0.y, nr0.w, nr0.x, nr0.z) : make_float4(nr0.x, nr0.z, nr0.y, nr0.w);
        const float4 c1 = PT ? make_float4(nr1.x, nr1.z, nr1.y, nr1.w) : make_float4(nr1.y, nr1.w, nr1.x, nr1.z);
        S.r[(slot * 2 + 0) * FTP_NT + threadIdx.x] = c0;
        S.r[(slot * 2 + 1) * FTP_NT + threadIdx.x] = c1;
        S.f[slot * FTP_NT + threadIdx.x] = make_uint2(nf0, nf1);
        gen = (gen << 1) | ((__any_sync(0xffffffffu, ((nf0 | nf1) & 0x3f3f3f3fu) != 0u) || t == 0 || t == D.nz - 1) ? 1u : 0u);
        fetch_r(t + 1);
        S.publish(0, pw, zn, D0);                     // colour 0 of plane t + 1
        // half-sweeps 1 .. 4 on planes t .. t - 3 (colours 1, 0, 1, 0)
#pragma unroll
        for (int k = 0; k <= 3; ++k) {
            const int p = t - k;
            if (p >= tlo && p < D.nz) {
                const int sl = ftp_back(slot, k);
                const bool g = (gen >> k) & 1u;
                ftp_sweep<LX, D0, NI>(c, Z[k], Z[k + 1], k ? Z[k > 0 ? k - 1 : 0] : zn, S.below(k, pr), S.above(k, pr),
                                  S.rhs(sl, 0, (k + 1) & 1), S.rhs(sl, 1, (k + 1) & 1), scale, g,
                                  S.f + sl * FTP_NT + threadIdx.x, g ? ftp_zadj(D, p) : 0, S.rcp);
                if (k < 3) S.publish(k + 1, pw, Z[k], D0);
            }
        }
        const int tf = t - 3;
        if (tf >= k0 && tf < k1) {
            const int sl = ftp_back(slot, 3);
            float* zo = zg + row0 + D.sz * tf;
            // row 0 of plane t - 3: colour 0 holds the cells D0, D0 + 2; row 1 the others
            if (c.own0) {
                ftp_store<NI>(zo, left, Z[3][0]);
                const float2 a = S.rhs(sl, 0, 0), b = S.rhs(sl, 0, 1);
                part += (a.x * Z[3][0][D0] + a.y * Z[3][0][D0 + 2]) + (b.x * Z[3][0][1 - D0] + b.y * Z[3][0][3 - D0]);
            }
            if (c.own1) {
                ftp_store<NI>(zo + D.sy, left, Z[3][1]);
                const float2 a = S.rhs(sl, 1, 0), b = S.rhs(sl, 1, 1);
                part += (a.x * Z[3][1][1 - D0] + a.y * Z[3][1][3 - D0]) + (b.x * Z[3][1][D0] + b.y * Z[3][1][D0 + 2]);
            }
        }
#pragma unroll
        for (int q = 4; q > 0; --q) ftp_copy(Z[q], Z[q - 1]);
        ftp_copy(Z[0], zn);
        ftp_set(zn, nz0, nz1);
        fetch_z(t + 3);
        slot = slot == FTP_RING - 1 ? 0 : slot + 1;
        __syncthreads();
    };
    for (int t = tlo; t <= thi; t += 2) {
        step(std::integral_constant<int, 0>{}, t);
        step(std::integral_constant<int, 1>{}, t + 1);
    }
    decltype(part) acc[1] = {part};
    grid_reduce<1>(acc, partials, counter, [&](double* tt) {
        sc->rz_old = sc->rz;
        sc->rz = tt[0];
    });
}

// ---- set-up -------------------------------------------------------------------------------------

// Level 1: parts of every block (cnt) and the part of every fine cell (sub0).
__global__ void k_parts1(Dom D, MGLev L, uint8_t* __restrict__ sub0) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < L.P; q += (long long)gridDim.x * blockDim.x) {
        int X[3];
        coords3(q, L.px, L.py, X);
        unsigned fl[8];
        long long P[8];
        const unsigned in = block_flags(D, X, fl, P);
        int part[8];
        L.cnt[q] = fine_parts(D, fl, in, part);
#pragma unroll
        for (int m = 0; m < 8; ++m)
            if ((in >> m) & 1u) sub0[P[m]] = (uint8_t)part[m];
    }
}

// Adds conductance g towards unknown v to a small table of distinct neighbours; false when full.
template <int CAP>
__device__ __forceinline__ bool table_add(int (&nb)[CAP], float (&gv)[CAP], int& n, int v, float g) {
    for (int e = 0; e < n; ++e)
        if (nb[e] == v) {
            gv[e] += g;
            return true;
        }
    if (n == CAP) return false;
    nb[n] = v;
    gv[n] = g;
    ++n;
    return true;
}

// Writes a row sorted by neighbour index (insertion sort; rows are short).
template <int CAP>
__device__ __forceinline__ float write_row(const MGLev& L, long long u, int (&nb)[CAP], float (&gv)[CAP], int n) {
    for (int e = 1; e < n; ++e) {
        const int v = nb[e];
        const float w = gv[e];
        int f = e - 1;
        while (f >= 0 && nb[f] > v) {
            nb[f + 1] = nb[f];
            gv[f + 1] = gv[f];
            --f;
        }
        nb[f + 1] = v;
        gv[f + 1] = w;
    }
    const long long k0 = L.rp[u];
    float gs = 0.f;
    for (int e = 0; e < n; ++e) {
        L.col[k0 + e] = nb[e];
        L.g[k0 + e] = gv[e];
        gs += gv[e];
    }
    return gs;
}

// Level 1 links.  Count pass (fill = 0): rp[u] = distinct neighbours, d, pos.  Fill pass: the sorted
// row, invdg.  A fine link leaving the block joins the part of its cell to the part of the cell across.
__global__ void k_links1(Dom D, MGLev L, const uint8_t* __restrict__ sub0, int fill, int* ovf) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < L.P; q += (long long)gridDim.x * blockDim.x) {
        int X[3];
        coords3(q, L.px, L.py, X);
        unsigned fl[8];
        long long P[8];
        const unsigned in = block_flags(D, X, fl, P);
        const int np = L.cnt[q];
        const int n3[3] = {D.nx, D.ny, D.nz};
        for (int s = 0; s < np; ++s) {
            const long long u = L.off[q] + s;
            int nb[MG_L1L];
            float gv[MG_L1L];
            int n = 0;
            float dsum = 0.f;
            for (int m = 0; m < 8; ++m) {
                if (!((in >> m) & 1u) || sub0[P[m]] != s) continue;
                const int x[3] = {2 * X[0] + (m & 1), 2 * X[1] + ((m >> 1) & 1), 2 * X[2] + (m >> 2)};
                for (int b = 0; b < 6; ++b) {
                    if (fl[m] & (1u << b)) continue;
                    const int a = b >> 1, sd = (b & 1) ? 1 : -1;
                    long long o;
                    if (!nb_offset(D, a, sd, x[a], o)) {
                        if (D.bc[b] == IBM_BC_OUTFLOW) dsum += 2.f;
                        continue;
                    }
                    int y[3] = {x[0], x[1], x[2]};
                    y[a] += sd;
                    if (y[a] < 0) y[a] = n3[a] - 1;
                    if (y[a] >= n3[a]) y[a] = 0;
                    const int Y[3] = {y[0] >> 1, y[1] >> 1, y[2] >> 1};
                    if (Y[0] == X[0] && Y[1] == X[1] && Y[2] == X[2]) continue;      // inside the block
                    const int v = L.off[pos_index(L, Y)] + sub0[P[m] + o];
                    if (!table_add<MG_L1L>(nb, gv, n, v, 1.f)) *ovf = 1;
                }
            }
            if (!fill) {
                L.rp[u] = n;
                L.d[u] = dsum;
                L.pos[u] = (int32_t)q;
            } else {
                const float gs = write_row<MG_L1L>(L, u, nb, gv, n);
                L.invdg[u] = gs + dsum > 0.f ? 1.f / (gs + dsum) : 0.f;
            }
        }
    }
}

// Level l + 1 from level l (= F): the parts of each block of 8 positions are the connected components of its
// unknowns under the links inside the block.  Lock-free union of every such link over all unknowns at once
// (the larger root is hung below the smaller, so a component's root is its smallest unknown whatever the
// order of the threads), however many unknowns a block holds: if some were left out they would become parts
// of their own, linked inside one position, and the two colours would no longer separate neighbours.
__device__ __forceinline__ int uf_find(const int* lab, int u) {
    int p = ((const volatile int*)lab)[u];
    while (p != u) {
        u = p;
        p = ((const volatile int*)lab)[u];
    }
    return u;
}

__global__ void k_uf_init(long long n, int* __restrict__ lab, int* __restrict__ num) {
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < n; u += (long long)gridDim.x * blockDim.x) {
        lab[u] = (int)u;
        num[u] = -1;
    }
}

__global__ void k_uf_union(MGLev F, int* lab) {
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < F.M; u += (long long)gridDim.x * blockDim.x) {
        int X[3];
        coords3(F.pos[u], F.px, F.py, X);
        for (int e = F.rp[u]; e < F.rp[u + 1]; ++e) {
            const int w = F.col[e];
            if (w > u) continue;                           // each link once
            int Y[3];
            coords3(F.pos[w], F.px, F.py, Y);
            if ((Y[0] >> 1) != (X[0] >> 1) || (Y[1] >> 1) != (X[1] >> 1) || (Y[2] >> 1) != (X[2] >> 1)) continue;
            int a = uf_find(lab, (int)u), b = uf_find(lab, w);
            while (a != b) {
                if (a < b) { const int t = a; a = b; b = t; }
                const int old = atomicCAS(&lab[a], a, b);  // hang root a below b
                if (old == a) break;
                a = uf_find(lab, a);
                b = uf_find(lab, b);
            }
        }
    }
}

// Numbers the parts of a block in the order in which its unknowns (by position) first meet them;
// F.parent[u] receives the part of u within its block (made global by k_parent_next).
__global__ void k_parts_next(MGLev F, MGLev C, const int* __restrict__ lab, int* __restrict__ num) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < C.P; q += (long long)gridDim.x * blockDim.x) {
        int Y[3];
        coords3(q, C.px, C.py, Y);
        int n = 0;
        for (int m = 0; m < 8; ++m) {
            const int X[3] = {2 * Y[0] + (m & 1), 2 * Y[1] + ((m >> 1) & 1), 2 * Y[2] + (m >> 2)};
            if (X[0] >= F.px || X[1] >= F.py || X[2] >= F.pz) continue;
            const long long qx = pos_index(F, X);
            for (int u = F.off[qx]; u < F.off[qx] + F.cnt[qx]; ++u) {
                const int r = uf_find(lab, u);             // a component lies in one block: no other thread
                int k = num[r];
                if (k < 0) num[r] = k = n++;
                F.parent[u] = k;
            }
        }
        C.cnt[q] = n;
    }
}

__global__ void k_parent_next(MGLev F, MGLev C) {
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < F.M; u += (long long)gridDim.x * blockDim.x) {
        int X[3];
        coords3(F.pos[u], F.px, F.py, X);
        const int Y[3] = {X[0] >> 1, X[1] >> 1, X[2] >> 1};
        F.parent[u] = C.off[pos_index(C, Y)] + F.parent[u];
    }
}

// Level l + 1 links (Galerkin sums) and lists of the children: of colour 0, or `all` (see grestrict).  Count pass: rp[v] = distinct neighbours, cp[v] = children, d, pos.  Fill pass: sorted rows, invdg, children.
__global__ void k_links_next(MGLev F, MGLev C, int fill, int all, int* ovf) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < C.P; q += (long long)gridDim.x * blockDim.x) {
        int Y[3];
        coords3(q, C.px, C.py, Y);
        const int np = C.cnt[q];
        for (int s = 0; s < np; ++s) {
            const int v = C.off[q] + s;
            int nb[MG_MAXL];
            float gv[MG_MAXL];
            int n = 0, nch = 0;
            float dsum = 0.f;
            for (int m = 0; m < 8; ++m) {
                const int X[3] = {2 * Y[0] + (m & 1), 2 * Y[1] + ((m >> 1) & 1), 2 * Y[2] + (m >> 2)};
                if (X[0] >= F.px || X[1] >= F.py || X[2] >= F.pz) continue;
                const long long qx = pos_index(F, X);
                for (int u = F.off[qx]; u < F.off[qx] + F.cnt[qx]; ++u) {
                    if (F.parent[u] != v) continue;
                    if (all || u < F.M0) {
                        if (fill) C.ch[C.cp[v] + nch] = u;
                        ++nch;
                    }
                    dsum += F.d[u];
                    for (int e = F.rp[u]; e < F.rp[u + 1]; ++e) {
                        const int pw = F.parent[F.col[e]];
                        if (pw == v) continue;
                        if (!table_add<MG_MAXL>(nb, gv, n, pw, F.g[e])) *ovf = 1;
                    }
                }
            }
            if (!fill) {
                C.rp[v] = n;
                C.cp[v] = nch;
                C.d[v] = dsum;
                C.pos[v] = (int32_t)q;
            } else {
                const float gs = write_row<MG_MAXL>(C, v, nb, gv, n);
                C.invdg[v] = gs + dsum > 0.f ? 1.f / (gs + dsum) : 0.f;
            }
        }
    }
}

// Colour-major numbering of the unknowns: positions of colour c contribute cnt[q] unknowns each, in
// position order, after all unknowns of colour 0 when c = 1.
struct PosCount {
    const int32_t* cnt;
    int px, py, colour;
    __device__ long long operator()(long long i) const {
        int x[3];
        coords3(i, px, py, x);
        return ((x[0] + x[1] + x[2]) & 1) == colour ? cnt[i] : 0;
    }
};
struct PosEmit {
    int32_t* off;
    int px, py, colour;
    const long long* base;
    __device__ void operator()(long long i, long long o, long long) const {
        int x[3];
        coords3(i, px, py, x);
        if (((x[0] + x[1] + x[2]) & 1) == colour) off[i] = (int32_t)(o + (base ? *base : 0));
    }
};
// In-place exclusive scan of a count array (rows, children).
struct ArrCount {
    const int32_t* a;
    __device__ long long operator()(long long i) const { return a[i]; }
};
struct ArrEmit {
    int32_t* a;
    __device__ void operator()(long long i, long long o, long long) const { a[i] = (int32_t)o; }
};

// Padded rows of the V-cycle: link e of unknown u at [e M + u], so a warp's rows are read whole; padding has
// g = 0.  A row with more than MG_ELL links stores -1 as its first column and is read from the CSR arrays.
// A conductance counts the fine faces between two parts: where all of a level's are whole numbers below 256 the
// V-cycle reads them as bytes, a row's six in one load (eg8), else as floats (eg).  `wide` is set if one is not.
__global__ void k_ell(MGLev L, int* wide) {
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < L.M; u += (long long)gridDim.x * blockDim.x) {
        const int k0 = L.rp[u], n = L.rp[u + 1] - k0;
        unsigned w[2] = {0u, 0u};
        for (int e = 0; e < MG_ELL; ++e) {
            const float g = n <= MG_ELL && e < n ? L.g[k0 + e] : 0.f;
            if (L.eg) {
                L.eg[e * L.M + u] = g;
                continue;
            }
            L.ecol[e * L.M + u] = n > MG_ELL ? -1 : (e < n ? L.col[k0 + e] : (int)u);
            const unsigned q = g >= 0.f && g < 256.f ? (unsigned)g : 0u;
            if ((float)q != g) atomicExch(wide, 1);
            w[e >> 2] |= q << (8 * (e & 3));
        }
        if (!L.eg) L.eg8[u] = make_uint2(w[0], w[1]);
    }
}

// ---- the V-cycle on the coarse levels -----------------------------------------------------------
//
// One red-black sweep before and after the coarse correction.  From x = 0 the first colour is x = -b / dg,
// written with b by whoever forms b; the residual of colour 0 after colour 1 is then  -sum g x_w  and that
// of colour 1 is zero, so the restriction reads colour 0 only.  After the correction colour 1 reads its
// neighbours' prolongated values on the fly and colour 0 reads colour 1: neither needs its own old value,
// so no pass adds the correction.  Four passes per level: colour 1, restriction, colour 1, colour 0.  An odd level's
// residual is evaluated in full and its passes after the correction write a second array (godd).

// sum over the links of u of g f(neighbour).
template <class T, class Fn>
__device__ __forceinline__ T row_sum(const MGLev& L, long long u, Fn f) {
    T s = 0;
    int c[MG_ELL];
    float g[MG_ELL];
#pragma unroll
    for (int e = 0; e < MG_ELL; ++e) c[e] = L.ecol[e * L.M + u];
    if (!L.eg) {
        const uint2 w = L.eg8[u];
#pragma unroll
        for (int e = 0; e < MG_ELL; ++e) g[e] = (float)(((e < 4 ? w.x : w.y) >> (8 * (e & 3))) & 255u);
    } else {
#pragma unroll
        for (int e = 0; e < MG_ELL; ++e) g[e] = L.eg[e * L.M + u];
    }
    if (c[0] < 0) {
        for (int e = L.rp[u]; e < L.rp[u + 1]; ++e) s += (T)L.g[e] * f(L.col[e]);
        return s;
    }
    // padding points at the unknown itself with g = 0 (its value is always set): the reads do not wait for one another
    T v[MG_ELL];
#pragma unroll
    for (int e = 0; e < MG_ELL; ++e) v[e] = f(c[e]);
#pragma unroll
    for (int e = 0; e < MG_ELL; ++e) s += (T)g[e] * v[e];
    return s;
}

// Colour `col` from its neighbours, into `out`.
template <class T>
__device__ __forceinline__ void gsmooth(const MGLev& L, int col, long long t0, long long nt, T* out) {
    const T* b = (const T*)L.b;
    const T* x = (const T*)L.x;
    const long long lo = col ? L.M0 : 0, hi = col ? L.M : L.M0;
    for (long long u = lo + t0; u < hi; u += nt)
        out[u] = (row_sum<T>(L, u, [&](int w) { return x[w]; }) - b[u]) * (T)L.invdg[u];
}

// Colour 1 after the coarse correction: the neighbours (colour 0) count with x + omega x_C(parent).
template <class T>
__device__ __forceinline__ void gup(const MGLev& L, const MGLev& C, T omega, long long t0, long long nt) {
    const T* b = (const T*)L.b;
    T* x = (T*)L.x;
    const T* xc = (const T*)C.x;
    for (long long u = L.M0 + t0; u < L.M; u += nt)
        x[u] = (row_sum<T>(L, u, [&](int w) { return x[w] + omega * xc[L.parent[w]]; }) - b[u]) * (T)L.invdg[u];
}

// The passes of an odd level.  0: colour 1 before the correction (its own old value is 0); 1: colour 1 after it, into
// y; 2: colour 0 after it, into y.  What has no new value yet counts with its old one and the correction.
template <class T>
__device__ __forceinline__ void godd(const MGLev& L, const MGLev& C, T omega, int pass, long long t0, long long nt) {
    const T* b = (const T*)L.b;
    const T* xc = (const T*)C.x;
    T *x = (T*)L.x, *y = (T*)L.y;
    const long long lo = pass < 2 ? L.M0 : 0, hi = pass < 2 ? L.M : L.M0;
    for (long long u = lo + t0; u < hi; u += nt) {
        const T s = row_sum<T>(L, u, [&](int w) {
            if (pass == 0) return w < L.M0 ? x[w] : (T)0;
            return pass == 2 && w >= L.M0 ? y[w] : x[w] + omega * xc[L.parent[w]];
        });
        (pass == 0 ? x : y)[u] = (s - b[u]) * (T)L.invdg[u];
    }
}

// b_C[v] = -sum over the children u of v of colour 0 of  sum g x_w; x_C = -b_C / dg.  Four lanes per coarse
// unknown (a plain 2x2x2 block has four children of each colour).  The thread count is a multiple of 32.
// FULL (FP64, where 1 / dg is stored in FP32 and the smoothed residuals vanish to 2^-24 only, and odd levels): the
// residuals are evaluated as they are, over all children.
template <class T, bool FULL>
__device__ __forceinline__ void grestrict(const MGLev& F, const MGLev& C, long long t0, long long nt) {
    const T* xf = (const T*)F.x;
    T* bc = (T*)C.b;
    T* xc = (T*)C.x;
    const int lane = (int)(t0 & 3);
    const long long rounds = (4 * C.M + nt - 1) / nt;
    for (long long q = 0; q < rounds; ++q) {
        const long long v = (t0 + q * nt) >> 2;
        T acc = 0;
        if (v < C.M)
            for (int k = C.cp[v] + lane; k < C.cp[v + 1]; k += 4) {
                const int u = C.ch[k];
                if constexpr (FULL) {
                    const T xu = xf[u];
                    acc += ((const T*)F.b)[u] - (row_sum<T>(F, u, [&](int w) { return xf[w] - xu; }) - (T)F.d[u] * xu);
                } else {
                    acc -= row_sum<T>(F, u, [&](int w) { return xf[w]; });
                }
            }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if (v < C.M && lane == 0) {
            bc[v] = acc;
            xc[v] = -acc * (T)C.invdg[v];
        }
    }
}

// Coarsest level, one block, in global memory: x = 0, then `sweeps` red-black passes and as many black-red (a
// symmetric operator).
template <class T>
__global__ void __launch_bounds__(1024) k_gcoarsest(MGLev L, int sweeps, const SolveScal* sc) {
    if (sc->done) return;
    T* x = (T*)L.x;
    for (long long u = threadIdx.x; u < L.M; u += blockDim.x) x[u] = (T)0;
    __syncthreads();
    for (int pass = 0; pass < 4 * sweeps; ++pass) {
        const int half = pass / (2 * sweeps), col = (pass & 1) ^ half;
        gsmooth<T>(L, col, threadIdx.x, blockDim.x, L.odd ? (T*)L.y : x);
        __syncthreads();
        if (!L.odd) continue;
        for (long long u = (col ? L.M0 : 0) + threadIdx.x; u < (col ? L.M : L.M0); u += blockDim.x) x[u] = ((T*)L.y)[u];
        __syncthreads();
    }
}

template <class T>
__global__ void __launch_bounds__(256) k_gsmooth(MGLev L, int col, const SolveScal* sc) {
    if (sc->done) return;
    gsmooth<T>(L, col, blockIdx.x * (long long)blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x, (T*)L.x);
}

template <class T>
__global__ void __launch_bounds__(256) k_godd(MGLev L, MGLev C, T omega, int pass, const SolveScal* sc) {
    if (sc->done) return;
    godd<T>(L, C, omega, pass, blockIdx.x * (long long)blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
}

template <class T, bool FULL>
__global__ void __launch_bounds__(256) k_grestrict(MGLev F, MGLev C, const SolveScal* sc) {
    if (sc->done) return;
    grestrict<T, FULL>(F, C, blockIdx.x * (long long)blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
}

template <class T>
__global__ void __launch_bounds__(256) k_gup(MGLev F, MGLev C, T omega, const SolveScal* sc) {
    if (sc->done) return;
    gup<T>(F, C, omega, blockIdx.x * (long long)blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
}

// The small levels first .. nlev-1 of a V-cycle in one launch of one cluster of M.ctas blocks.  Every
// block keeps its share of each level (half of it of either colour) in shared memory; neighbours are read
// from the other blocks' shared memory and a cluster barrier (hardware, release/acquire at cluster scope)
// separates dependent passes.  The coarsest level belongs to block 0 as a whole and is solved there with
// barriers of the warps it needs, its rows in registers.  All of it is latency: five passes per level and 32
// on the coarsest.  So everything that does not change between V-cycles (rows, parents of neighbours,
// children, as places: block << M.shift | index) is laid out once as an image of the blocks' shared memory and
// copied in by 16-byte loads that are all in flight at once, and a row's reads do not wait for one another.
// Levels of 8227, 1032 and 136 unknowns: 18 us (FP64 32, of which the FP64 units of 16 SMs are half); with eight
// blocks 20 us (FP64 38), 48 us through L2 with device-wide fences and rows read where they are used (FP64 80).
#define MG_TAIL_NT 512
#define MG_FAR 0xffffu          // first place of a row with more than MG_ELL links: start and count follow

struct TailPlace {
    MGTailLev t;
    int shift;
    __device__ __forceinline__ unsigned operator()(int u) const {
        const bool c = u >= t.M0;
        const unsigned w = (unsigned)(c ? u - t.M0 : u), s = (unsigned)(c ? t.s1 : t.s0);
        const unsigned r = __umulhi(w, c ? t.i1 : t.i0);
        return r << shift | ((c ? (unsigned)t.s0 : 0u) + w - r * s);
    }
};

template <class T>
struct TailLevel {
    MGTailLev t;
    unsigned char* sm;
    int rank, shift;
    __device__ __forceinline__ TailLevel(const MGTail& M, int l, unsigned char* s, int r)
        : t(M.t[l]), sm(s), rank(r), shift(M.shift) {}
    template <class V>
    __device__ __forceinline__ V* arr(int o) const { return reinterpret_cast<V*>(sm + o); }
    __device__ __forceinline__ T* x() const { return arr<T>(t.x); }
    __device__ __forceinline__ T* b() const { return arr<T>(t.b); }
    __device__ __forceinline__ T* tmp() const { return arr<T>(t.t); }
    __device__ __forceinline__ T* dg() const { return arr<T>(t.dg); }
    __device__ __forceinline__ T* d() const { return arr<T>(t.d); }
    // the block's unknowns of colour c: local [base, base + n), global from lo
    __device__ __forceinline__ void span(int c, int& base, int& n, int& lo) const {
        const int s = c ? t.s1 : t.s0, all = c ? t.M - t.M0 : t.M0;
        base = c ? t.s0 : 0;
        const int f = rank * s;
        n = f < all ? (all - f < s ? all - f : s) : 0;
        lo = (c ? t.M0 : 0) + f;
    }
    // value of an array (a pointer into this block's shared memory) at a place
    __device__ __forceinline__ T at(const T* a, unsigned place) const {
        return *cg::this_cluster().map_shared_rank(const_cast<T*>(a) + (place & ((1u << shift) - 1u)), place >> shift);
    }
    // sum over the links of local unknown i of g f(place of the neighbour, place of its parent)
    template <bool PARENT, class Fn>
    __device__ __forceinline__ T row(int i, Fn f) const {
        const int S = t.s0 + t.s1;
        unsigned c[MG_ELL], p[MG_ELL];
        T g[MG_ELL], v[MG_ELL];
#pragma unroll
        for (int e = 0; e < MG_ELL; ++e) {
            c[e] = arr<uint16_t>(t.col)[e * S + i];
            p[e] = PARENT ? arr<uint16_t>(t.pc)[e * S + i] : 0u;
            g[e] = arr<T>(t.g)[e * S + i];
        }
        if (c[0] == MG_FAR) {
            T s = 0;
            for (unsigned k = c[1]; k < c[1] + c[2]; ++k)
                s += arr<T>(t.og)[k] * f((unsigned)arr<uint16_t>(t.oc)[k], PARENT ? (unsigned)arr<uint16_t>(t.op)[k] : 0u);
            return s;
        }
        // padding points at the unknown itself with g = 0
#pragma unroll
        for (int e = 0; e < MG_ELL; ++e) v[e] = f(c[e], p[e]);
        T s = 0;
#pragma unroll
        for (int e = 0; e < MG_ELL; ++e) s += g[e] * v[e];
        return s;
    }
};

// The constant arrays of every block's shares, in the layout of its shared memory (set-up; 32-bit cursors of
// the long rows in `cur`, zero before).
template <class T>
__global__ void __launch_bounds__(256) k_tail_image(MGTail M, unsigned char* img, int* cur) {
    const int rank = blockIdx.x, last = M.nlev - 1;
    unsigned char* sm = img + (size_t)rank * M.image;
    for (int l = M.first; l <= last; ++l) {
        const TailLevel<T> A(M, l, sm, rank);
        const MGLev& L = M.lev[l];
        const TailPlace here{A.t, M.shift}, up{M.t[l < last ? l + 1 : l], M.shift}, below{M.t[l > M.first ? l - 1 : l], M.shift};
        const int S = A.t.s0 + A.t.s1;
        int nch = 0;
        for (int c = 0; c < 2; ++c) {
            int base, n, lo;
            A.span(c, base, n, lo);
            const int k0 = l > M.first && n > 0 ? L.cp[lo] : 0, k1 = l > M.first && n > 0 ? L.cp[lo + n] : 0;
            for (int i = threadIdx.x; i < n; i += blockDim.x) {
                const int u = lo + i, r0 = L.rp[u], nr = L.rp[u + 1] - r0;
                A.dg()[base + i] = (T)L.invdg[u];
                if (sizeof(T) == 8 || A.t.odd) A.d()[base + i] = (T)L.d[u];
                int at = 0;
                if (nr > MG_ELL) {
                    at = atomicAdd(&cur[rank * IBM_MG_MAXLEV + l], nr);
                    for (int e = 0; e < nr; ++e) {
                        const int w = L.col[r0 + e];
                        A.template arr<uint16_t>(A.t.oc)[at + e] = (uint16_t)here(w);
                        if (l < last) A.template arr<uint16_t>(A.t.op)[at + e] = (uint16_t)up(L.parent[w]);
                        A.template arr<T>(A.t.og)[at + e] = (T)L.g[r0 + e];
                    }
                }
                for (int e = 0; e < MG_ELL; ++e) {
                    const int w = e < nr ? L.col[r0 + e] : u;
                    unsigned q = here(w);
                    if (nr > MG_ELL) q = e == 0 ? MG_FAR : (unsigned)(e == 1 ? at : nr);
                    A.template arr<uint16_t>(A.t.col)[e * S + base + i] = (uint16_t)q;
                    if (l < last) A.template arr<uint16_t>(A.t.pc)[e * S + base + i] = (uint16_t)up(L.parent[w]);
                    A.template arr<T>(A.t.g)[e * S + base + i] = e < nr ? (T)L.g[r0 + e] : (T)0;
                }
                if (l > M.first) A.template arr<int>(A.t.cv)[base + i] = (nch + L.cp[u] - k0) | (L.cp[u + 1] - L.cp[u]) << 18;
            }
            for (int k = k0 + threadIdx.x; k < k1; k += blockDim.x)
                A.template arr<uint16_t>(A.t.ch)[nch + k - k0] = (uint16_t)below(L.ch[k]);
            nch += k1 - k0;
        }
    }
}

// ODD: a level may be odd.
template <class T, bool ODD>
__global__ void __launch_bounds__(MG_TAIL_NT, 1) k_mg_tail(const __grid_constant__ MGTail M, const SolveScal* sc) {
    if (sc->done) return;                       // the flag is uniform: set by an earlier kernel
    extern __shared__ __align__(16) unsigned char tail_smem[];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), last = M.nlev - 1, tid = threadIdx.x;
    {
        const uint4* __restrict__ src = M.img + (size_t)rank * (M.image / 16);
        uint4* dst = reinterpret_cast<uint4*>(tail_smem);
        const int n = M.image / 16;
        for (int q0 = tid; q0 < n; q0 += 8 * MG_TAIL_NT) {
            uint4 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q0 + q * MG_TAIL_NT < n) v[q] = src[q0 + q * MG_TAIL_NT];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q0 + q * MG_TAIL_NT < n) dst[q0 + q * MG_TAIL_NT] = v[q];
        }
        // b and x of the first level from global memory, x = 0 on the coarsest (also where padding is read)
        const TailLevel<T> A(M, M.first, tail_smem, rank);
        for (int c = 0; c < 2; ++c) {
            int base, nn, lo;
            A.span(c, base, nn, lo);
            const T *bg = (const T*)M.lev[M.first].b, *xg = (const T*)M.lev[M.first].x;
            for (int i = tid; i < nn; i += MG_TAIL_NT) {
                A.b()[base + i] = bg[lo + i];
                if (M.first < last) A.x()[base + i] = xg[lo + i];
            }
        }
        const TailLevel<T> C(M, last, tail_smem, rank);
        if (rank == 0)
            for (int i = tid; i < C.t.M; i += MG_TAIL_NT) C.x()[i] = (T)0;
    }
    cl.sync();
    // a place on level A belongs to colour 0
    auto first = [&](const TailLevel<T>& A, unsigned q) { return (q & ((1u << A.shift) - 1u)) < (unsigned)A.t.s0; };
    // colour c of a level from its neighbours (odd levels: colour 1 from those of colour 0, its own old value is 0)
    auto smooth = [&](const TailLevel<T>& A, int c) {
        int base, n, lo;
        A.span(c, base, n, lo);
        T* x = A.x();
        if (ODD && A.t.odd) {
            for (int i = base + tid; i < base + n; i += MG_TAIL_NT)
                x[i] = (A.template row<false>(i, [&](unsigned q, unsigned) { return first(A, q) ? A.at(x, q) : (T)0; }) - A.b()[i]) * A.dg()[i];
            return;
        }
        for (int i = base + tid; i < base + n; i += MG_TAIL_NT)
            x[i] = (A.template row<false>(i, [&](unsigned q, unsigned) { return A.at(x, q); }) - A.b()[i]) * A.dg()[i];
    };
    for (int l = M.first; l < last; ++l) {
        const TailLevel<T> A(M, l, tail_smem, rank), C(M, l + 1, tail_smem, rank);
        T* x = A.x();
        smooth(A, 1);
        cl.sync();
        // residuals (in full: of both colours, see grestrict)
        const bool full = sizeof(T) == 8 || (ODD && A.t.odd);
        for (int c = 0; c < (full ? 2 : 1); ++c) {
            int base, n, lo;
            A.span(c, base, n, lo);
            for (int i = base + tid; i < base + n; i += MG_TAIL_NT) {
                const T xu = x[i];
                if (full)
                    A.tmp()[i] = A.b()[i] - (A.template row<false>(i, [&](unsigned q, unsigned) { return A.at(x, q) - xu; }) - A.d()[i] * xu);
                else
                    A.tmp()[i] = -A.template row<false>(i, [&](unsigned q, unsigned) { return A.at(x, q); });
            }
        }
        cl.sync();
        // b of the next level and its first half-sweep: four lanes per unknown
        for (int c = 0; c < 2; ++c) {
            int base, n, lo;
            C.span(c, base, n, lo);
            for (int q = 0; q < (4 * n + MG_TAIL_NT - 1) / MG_TAIL_NT; ++q) {
                const int i = (tid + q * MG_TAIL_NT) >> 2;
                T acc = 0;
                if (i < n) {
                    const int v = C.template arr<int>(C.t.cv)[base + i], k0 = v & 0x3ffff, nk = v >> 18;
                    for (int k = tid & 3; k < nk; k += 4) acc += A.at(A.tmp(), C.template arr<uint16_t>(C.t.ch)[k0 + k]);
                }
                acc += __shfl_xor_sync(0xffffffffu, acc, 1);
                acc += __shfl_xor_sync(0xffffffffu, acc, 2);
                if (i < n && (tid & 3) == 0) {
                    C.b()[base + i] = acc;
                    if (l + 1 < last) C.x()[base + i] = -acc * C.dg()[base + i];
                }
            }
        }
        cl.sync();
    }
    if (rank == 0) {
        // coarsest level: x = 0, then sweeps red-black passes and as many black-red (a symmetric operator)
        const TailLevel<T> A(M, last, tail_smem, 0);
        const int most = max(A.t.s0, A.t.s1), nth = min(MG_TAIL_NT, (most + 31) & ~31), S = A.t.s0 + A.t.s1;
        T* x = A.x();
        if (most <= MG_TAIL_NT && tid < nth) {
            // one row of either colour per thread, in registers
            unsigned q[2][MG_ELL];
            T g[2][MG_ELL], b[2] = {0, 0}, dg[2] = {0, 0};
            bool on[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                on[c] = tid < (c ? A.t.M - A.t.M0 : A.t.M0);
                const int i = (c ? A.t.s0 : 0) + (on[c] ? tid : 0);
                if (on[c]) {
                    b[c] = A.b()[i];
                    dg[c] = A.dg()[i];
                }
#pragma unroll
                for (int e = 0; e < MG_ELL; ++e) {
                    q[c][e] = on[c] ? A.template arr<uint16_t>(A.t.col)[e * S + i] : 0u;
                    g[c][e] = on[c] ? A.template arr<T>(A.t.g)[e * S + i] : (T)0;
                }
            }
            for (int pass = 0; pass < 2 * M.coarse_sweeps; ++pass) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // (the barriers stand outside what only some lanes of a warp run)
                    auto colour = [&](auto cc) {
                        constexpr int c = decltype(cc)::value;
                        const int i = (c ? A.t.s0 : 0) + tid;
                        T s = 0;
                        if (on[c]) {
                            if (q[c][0] == MG_FAR) {
                                s = A.template row<false>(i, [&](unsigned p, unsigned) { return x[p]; });
                            } else {
                                T v[MG_ELL];
#pragma unroll
                                for (int e = 0; e < MG_ELL; ++e) v[e] = x[q[c][e]];
#pragma unroll
                                for (int e = 0; e < MG_ELL; ++e) s += g[c][e] * v[e];
                            }
                        }
                        if (ODD && A.t.odd) {                       // every value of the colour is read before one is written
                            __syncwarp();
                            asm volatile("bar.sync 1, %0;" ::"r"(nth) : "memory");
                        }
                        if (on[c]) x[i] = (s - b[c]) * dg[c];
                        __syncwarp();
                    };
                    if (h ^ (pass >= M.coarse_sweeps ? 1 : 0)) colour(std::integral_constant<int, 1>{});
                    else colour(std::integral_constant<int, 0>{});
                    asm volatile("bar.sync 1, %0;" ::"r"(nth) : "memory");
                }
            }
        } else if (most > MG_TAIL_NT) {
            for (int pass = 0; pass < 4 * M.coarse_sweeps; ++pass) {
                const int c = (pass & 1) ^ (pass / (2 * M.coarse_sweeps));
                const int lo = c ? A.t.M0 : 0, hi = c ? A.t.M : A.t.M0;
                T* out = ODD && A.t.odd ? A.tmp() : x;
                for (int i = lo + tid; i < hi; i += MG_TAIL_NT)
                    out[i] = (A.template row<false>(i, [&](unsigned p, unsigned) { return x[p]; }) - A.b()[i]) * A.dg()[i];
                __syncthreads();
                if (ODD && A.t.odd) {
                    for (int i = lo + tid; i < hi; i += MG_TAIL_NT) x[i] = out[i];
                    __syncthreads();
                }
            }
        }
    }
    cl.sync();
    for (int l = last - 1; l >= M.first; --l) {
        const TailLevel<T> A(M, l, tail_smem, rank), C(M, l + 1, tail_smem, rank);
        if (ODD && A.t.odd) {
            // as godd, into tmp
            T *x = A.x(), *y = A.tmp();
            const T om = (T)M.omega;
            for (int c = 1; c >= 0; --c) {
                int base, n, lo;
                A.span(c, base, n, lo);
                for (int i = base + tid; i < base + n; i += MG_TAIL_NT)
                    y[i] = (A.template row<true>(i, [&](unsigned q, unsigned p) {
                               return c == 0 && !first(A, q) ? A.at(y, q) : A.at(x, q) + om * C.at(C.x(), p);
                           }) - A.b()[i]) * A.dg()[i];
                cl.sync();
            }
            for (int i = tid; i < A.t.s0 + A.t.s1; i += MG_TAIL_NT) x[i] = y[i];
            if (l > M.first) cl.sync();
            continue;
        }
        {
            // colour 1: the neighbours count with their prolongated correction
            int base, n, lo;
            A.span(1, base, n, lo);
            T* x = A.x();
            const T om = (T)M.omega;
            for (int i = base + tid; i < base + n; i += MG_TAIL_NT)
                x[i] = (A.template row<true>(i, [&](unsigned q, unsigned p) { return A.at(x, q) + om * C.at(C.x(), p); }) - A.b()[i]) *
                       A.dg()[i];
        }
        cl.sync();
        smooth(A, 0);
        if (l > M.first) cl.sync();
    }
    {
        const TailLevel<T> A(M, M.first, tail_smem, rank);
        __syncthreads();
        for (int c = 0; c < 2; ++c) {
            int base, n, lo;
            A.span(c, base, n, lo);
            for (int i = tid; i < n; i += MG_TAIL_NT) ((T*)M.lev[M.first].x)[lo + i] = A.x()[base + i];
        }
    }
    cl.sync();                                  // no block leaves while others may read its shared memory
}

// ---- transfer between the fine grid and level 1 -------------------------------------------------

// b_1 of each part of a level-1 block = the sum of the fine residuals  scale r - (A z)  of its cells, and the
// first half-sweep of level 1, x_1 = -b_1 / dg.  Eight lanes per block, one per cell, for the latency of small grids:
// 64 x 32 x 32 in FP64 4.8 us, 21.5 us with one lane.
template <class T>
__global__ void __launch_bounds__(256) k_mg_restrict0(Dom D, const T* __restrict__ r, const T* __restrict__ z, T scale,
                                                      MGLev C, const SolveScal* sc) {
    if (sc->done) return;
    const int m = threadIdx.x & 7;
    const unsigned gm = 0xffu << (threadIdx.x & 24);
    auto zv = [&](long long c) { return z[c]; };
    for (long long q = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 3; q < C.P;
         q += ((long long)gridDim.x * blockDim.x) >> 3) {
        int X[3];
        coords3(q, C.px, C.py, X);
        const int i = 2 * X[0] + (m & 1), j = 2 * X[1] + ((m >> 1) & 1), k = 2 * X[2] + (m >> 2);
        const bool on = i < D.nx && j < D.ny && k < D.nz;
        const long long P = i + (long long)D.sy * j + D.sz * k;
        const int o = C.off[q];
        unsigned f = 0u;
        T res = (T)0;
        if (on) {
            f = flags_at(D, P);
            const CellLinks L = cell_links(D, i, j, k, f);
            const int dg = __popc(L.open) + 2 * __popc(L.out & ~f);
            res = scale * r[P] - (open_sum<T>(L, P, zv) - small_num<T>(dg) * z[P]);
        }
        const unsigned in = (__ballot_sync(gm, on) >> (threadIdx.x & 24)) & 0xffu;
        int np = 1, mine = 0;
        if (__ballot_sync(gm, f != 0u) != 0u || in != 0xffu) {
            unsigned fl[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) fl[e] = __shfl_sync(gm, f, e, 8);
            int part[8];
            np = fine_parts(D, fl, in, part);
#pragma unroll
            for (int e = 0; e < 8; ++e) mine = m == e ? part[e] : mine;
        }
        for (int s = 0; s < np; ++s) {
            T v = mine == s ? res : (T)0;
#pragma unroll
            for (int d = 1; d < 8; d *= 2) v += __shfl_xor_sync(gm, v, d);
            if (m == s) put_b1<T>(C, o + s, v);
        }
    }
}

// z += omega x_1(part of the cell).
template <class T>
__global__ void __launch_bounds__(256) k_mg_prolong0(Dom D, T* __restrict__ z, MGLev C, T omega, const SolveScal* sc) {
    if (sc->done) return;
    const T* __restrict__ xc = (const T*)C.x;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < C.P; q += (long long)gridDim.x * blockDim.x) {
        int X[3];
        coords3(q, C.px, C.py, X);
        unsigned fl[8];
        long long P[8];
        const unsigned in = block_flags(D, X, fl, P);
        int part[8];
        const int np = fine_parts(D, fl, in, part);
        const int o = C.off[q];
        T v[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) v[s] = s < np ? xc[o + s] : (T)0;
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            if (!((in >> m) & 1u)) continue;
            T w = v[0];
#pragma unroll
            for (int s = 1; s < 8; ++s) w = part[m] == s ? v[s] : w;
            z[P[m]] = z[P[m]] + omega * w;
        }
    }
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ unsigned flags4(const Dom& D, long long P) {
    return D.flags ? *reinterpret_cast<const unsigned*>(D.flags + P) : 0u;
}

// FP32 restriction with nx a multiple of 4: one thread per pair of level-1 positions (2 xp, 2 xp + 1)
// at (Y, Z), i.e. the 4 fine cells [4 xp, 4 xp + 4) of each of the (up to) 4 fine rows below them,
// with 16-byte loads.
__global__ void __launch_bounds__(256) k_mg_restrict0_x4(Dom D, const float* __restrict__ r,
                                                         const float* __restrict__ z, float scale, MGLev C,
                                                         const SolveScal* sc) {
    if (sc->done) return;
    const int px = D.nx / 4;
    const long long npairs = (long long)px * C.py * C.pz;
    auto zv = [&](long long c) { return z[c]; };
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < npairs;
         t += (long long)gridDim.x * blockDim.x) {
        const unsigned tu = (unsigned)t, rq = tu / (unsigned)px;
        const int xp = (int)(tu - rq * (unsigned)px), Y = (int)(rq % (unsigned)C.py), Z = (int)(rq / (unsigned)C.py);
        const int i0 = 4 * xp;
        float res[2][2][4];
        unsigned f4[2][2];
        unsigned rows = 0;
#pragma unroll
        for (int dk = 0; dk < 2; ++dk)
#pragma unroll
            for (int dj = 0; dj < 2; ++dj) {
                const int j = 2 * Y + dj, k = 2 * Z + dk;
                f4[dk][dj] = 0u;
#pragma unroll
                for (int m = 0; m < 4; ++m) res[dk][dj][m] = 0.f;
                if (j >= D.ny || k >= D.nz) continue;
                rows |= 1u << (2 * dk + dj);
                const long long P = i0 + (long long)D.sy * j + D.sz * k;
                const unsigned fl4 = flags4(D, P);
                f4[dk][dj] = fl4;
                const float4 r4 = ld4(r + P), z4 = ld4(z + P);
                const float zc[4] = {z4.x, z4.y, z4.z, z4.w}, rr[4] = {r4.x, r4.y, r4.z, r4.w};
                if (fl4 == 0u && i0 > 0 && i0 + 4 < D.nx && j > 0 && j < D.ny - 1 && k > 0 && k < D.nz - 1) {
                    const float4 ym = ld4(z + P - D.sy), yp = ld4(z + P + D.sy);
                    const float4 zm = ld4(z + P - D.sz), zp = ld4(z + P + D.sz);
                    const float xl = z[P - 1], xr = z[P + 4];
                    const float a[4] = {ym.x + yp.x + zm.x + zp.x, ym.y + yp.y + zm.y + zp.y,
                                        ym.z + yp.z + zm.z + zp.z, ym.w + yp.w + zm.w + zp.w};
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const float xm = m == 0 ? xl : zc[m - 1];
                        const float xq = m == 3 ? xr : zc[m + 1];
                        res[dk][dj][m] = scale * rr[m] - ((xm + xq) + a[m] - 6.f * zc[m]);
                    }
                } else {
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const unsigned fl = (fl4 >> (8 * m)) & 0xffu;
                        res[dk][dj][m] = scale * rr[m] - link_sum7<float>(D, P + m, i0 + m, j, k, fl, zc[m], zv);
                    }
                }
            }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            unsigned fl[8];
            unsigned in = 0;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int di = m & 1, dj = (m >> 1) & 1, dk = m >> 2;
                fl[m] = (f4[dk][dj] >> (8 * (2 * h + di))) & 0xffu;
                in |= ((rows >> (2 * dk + dj)) & 1u) << m;
            }
            int part[8];
            const int np = fine_parts(D, fl, in, part);
            float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const float v = res[m >> 2][(m >> 1) & 1][2 * h + (m & 1)];
#pragma unroll
                for (int s = 0; s < 8; ++s) acc[s] += part[m] == s ? v : 0.f;
            }
            const int o = C.off[(2 * xp + h) + (long long)C.px * (Y + (long long)C.py * Z)];
#pragma unroll
            for (int s = 0; s < 8; ++s)
                if (s < np) put_b1<float>(C, o + s, acc[s]);
        }
    }
}

// FP32 prolongation with nx a multiple of 4: a thread takes two positions of level 1 along x, two rows of two planes.
// Flags, offsets and the iterate are loaded together, so that the coarse values are the only loads that wait for
// others, and a warp without a cut link skips the search for parts.  Bound by HBM (71 %): 8 bytes per cell and the
// coarse values, 49 us at 512 x 256 x 256; 92 us with loads that wait for one another.
__global__ void __launch_bounds__(256, 4) k_mg_prolong0_x4(Dom D, float* __restrict__ z, MGLev C, float omega,
                                                        const SolveScal* sc) {
    if (sc->done) return;
    const float* __restrict__ xc = (const float*)C.x;
    const unsigned px = (unsigned)D.nx / 4;
    const long long npairs = (long long)px * C.py * C.pz;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < npairs;
         t += (long long)gridDim.x * blockDim.x) {
        const unsigned tu = (unsigned)t, rq = tu / px;
        const int xp = (int)(tu - rq * px), Y = (int)(rq % (unsigned)C.py), Z = (int)(rq / (unsigned)C.py);
        const long long P0 = 4 * xp + (long long)D.sy * (2 * Y) + D.sz * (2 * Z);
        const bool y2 = 2 * Y + 1 < D.ny, z2 = 2 * Z + 1 < D.nz;
        float4 zv[2][2];
        unsigned f4[2][2], any = 0u;
#pragma unroll
        for (int dk = 0; dk < 2; ++dk)
#pragma unroll
            for (int dj = 0; dj < 2; ++dj) {
                const bool ok = (dj == 0 || y2) && (dk == 0 || z2);
                const long long P = P0 + dj * (long long)D.sy + dk * D.sz;
                zv[dk][dj] = ok ? ld4(z + P) : make_float4(0.f, 0.f, 0.f, 0.f);
                f4[dk][dj] = ok ? flags4(D, P) : 0u;
                any |= f4[dk][dj];
            }
        const int2 o = *reinterpret_cast<const int2*>(C.off + 2 * xp + (long long)C.px * (Y + (long long)C.py * Z));
        if (!any) {
            const float a = omega * xc[o.x], b = omega * xc[o.y];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float4& v = zv[q >> 1][q & 1];
                v.x += a;
                v.y += a;
                v.z += b;
                v.w += b;
            }
        } else {
            const unsigned rows = 1u | (y2 ? 2u : 0u) | (z2 ? 4u : 0u) | (y2 && z2 ? 8u : 0u);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                unsigned fl[8], in = 0;
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const int di = m & 1, dj = (m >> 1) & 1, dk = m >> 2;
                    fl[m] = (f4[dk][dj] >> (8 * (2 * h + di))) & 0xffu;
                    in |= ((rows >> (2 * dk + dj)) & 1u) << m;
                }
                int part[8];
                const int np = fine_parts(D, fl, in, part);
                const int oo = h ? o.y : o.x;
                float v[8];
#pragma unroll
                for (int s = 0; s < 8; ++s) v[s] = s < np ? xc[oo + s] : 0.f;
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const int di = m & 1, dj = (m >> 1) & 1, dk = m >> 2;
                    float a = v[0];
#pragma unroll
                    for (int s = 1; s < 8; ++s) a = part[m] == s ? v[s] : a;
                    float4& u = zv[dk][dj];
                    if (h == 0 && di == 0) u.x += omega * a;
                    else if (h == 0) u.y += omega * a;
                    else if (di == 0) u.z += omega * a;
                    else u.w += omega * a;
                }
            }
        }
#pragma unroll
        for (int dk = 0; dk < 2; ++dk)
#pragma unroll
            for (int dj = 0; dj < 2; ++dj)
                if ((dj == 0 || y2) && (dk == 0 || z2)) st4(z + P0 + dj * (long long)D.sy + dk * D.sz, zv[dk][dj]);
    }
}

unsigned lin_blocks(long long n) {
    long long b = (n + 255) / 256;
    long long cap = 8LL * IBM_NSM;
    if (b > cap) b = cap;
    return (unsigned)(b < 1 ? 1 : b);
}

// Planes of a tile (halo included) with a cut link: the passes take the general half-sweeps there.
__global__ void __launch_bounds__(256) k_tile_marks(Dom D, int w, int h, unsigned tx, unsigned ty, uint8_t* marks) {
    const unsigned row = blockIdx.x / tx;
    const int x0 = (int)(blockIdx.x - row * tx) * (w - 8), y0 = (int)(row % ty) * (h - 8), k = (int)(row / ty);
    unsigned any = 0u;
    for (int q = threadIdx.x; q < w * h; q += blockDim.x) {
        const int x = x0 + q % w, y = y0 + q / w;
        if (x < D.nx && y < D.ny) any |= D.flags[x + (long long)D.sy * y + D.sz * k] & 63u;
    }
    any = __syncthreads_or(any != 0u);
    if (threadIdx.x == 0) marks[blockIdx.x] = any ? 1 : 0;
}

// The launch of the fused passes: of the two tile widths (64 x 64 or 128 x 32 cells, halo included; 64 x 64 has the
// smaller halo, 128 x 32 fits some grids better), each tile cut into chunks of whole pairs of planes.  A chunk costs
// its planes and eight more, planes with cut links FZ_GENERAL as much as others (measured 2.57 and 1.57 us), and
// blocks run one per SM; for eight numbers of rounds the limit on a chunk's cost is bisected that lets the
// chunks fit the rounds, and the cheapest is kept.  With chunks of equal height the tiles around a body came last: 52
// and 42 us in place of 43 and 34 on 256 x 128 x 128 cells around a dirty sphere.  1.3 to 1.4 and 1.9 to 2.5 for
// FZ_GENERAL are slower there and around the vehicle.
#define FZ_GENERAL 1.65f

struct FzPlan {
    int tx, ty, nz;
    const float* sum;           // [tile][nz + 9] sums of the planes' costs from plane -4 on, nz + 4 the last
    // chunks of at most `limit` (a pair of planes at least); their number, or -1 if more than `most`
    long long cut(float limit, long long most, int4* out, float* cost) const {
        long long n = 0;
        for (int t = 0; t < tx * ty; ++t) {
            const float* s = sum + (long long)t * (nz + 9);
            for (int k0 = 0; k0 < nz;) {
                int k1 = k0 + 2;
                while (k1 < nz && at(s, k0, k1 + 2) <= limit) k1 += 2;
                if (k1 > nz) k1 = nz;
                if (n == most) return -1;
                if (out) {
                    out[n] = make_int4(t % tx, t / tx, k0, k1);
                    cost[n] = at(s, k0, k1);
                }
                ++n;
                k0 = k1;
            }
        }
        return n;
    }
    float at(const float* s, int k0, int k1) const { return s[(k1 > nz ? nz : k1) + 8] - s[k0]; }
};

int fused_plan(const LesCtx& c, MG& mg, int sb) {
    const Dom& D = c.D;
    bool per = false;
    for (int f = 0; f < 6; ++f) per = per || D.bc[f] == IBM_BC_PERIODIC;
    mg.fused = mg.allow_fused && sb == 4 && mg.sweeps == 2 && mg.nlev > 1 && !per;
    if (!mg.fused) return IBM_OK;
    float best = -1.f;
    for (int lx = 16; lx <= 32; lx *= 2) {
        const int w = 4 * lx, h = 2 * (FTP_NT / lx);
        FzPlan p;
        p.tx = D.nx > w ? (D.nx - 8 + w - 9) / (w - 8) : 1;
        p.ty = D.ny > h ? (D.ny - 8 + h - 9) / (h - 8) : 1;
        p.nz = D.nz;
        const long long tiles = (long long)p.tx * p.ty, cap = tiles * ((D.nz + 1) / 2);
        uint8_t *dev = nullptr, *marks = (uint8_t*)calloc(tiles, D.nz);
        float* sum = (float*)malloc(sizeof(float) * tiles * (D.nz + 9));
        int4* out = (int4*)malloc(sizeof(int4) * cap);
        float* cost = (float*)malloc(sizeof(float) * cap);
        int* order = (int*)malloc(sizeof(int) * cap);
        cudaError_t e = marks && sum && out && cost && order ? cudaSuccess : cudaErrorMemoryAllocation;
        if (e == cudaSuccess && D.flags) {
            e = ibm_malloc(&dev, tiles * D.nz);
            if (e == cudaSuccess) {
                k_tile_marks<<<(unsigned)(tiles * D.nz), 256>>>(D, w, h, p.tx, p.ty, dev);
                e = cudaMemcpy(marks, dev, tiles * D.nz, cudaMemcpyDeviceToHost);
            }
            cudaFree(dev);
        }
        if (e == cudaSuccess) {
            for (long long t = 0; t < tiles; ++t) {
                float* s = sum + t * (D.nz + 9);
                float a = 0.f;
                for (int k = -4; k < D.nz + 4; ++k) {
                    s[k + 4] = a;
                    if (k < 0) continue;
                    a += k == 0 || k == D.nz - 1 || (k < D.nz && marks[t + tiles * k]) ? FZ_GENERAL : 1.f;
                }
                s[D.nz + 8] = a;
            }
            p.sum = sum;
            const int first = (int)((tiles + IBM_NSM - 1) / IBM_NSM);
            for (int rounds = first; rounds < first + 8; ++rounds) {
                float lo = 0.f, hi = FZ_GENERAL * (D.nz + 9);
                const long long most = (long long)rounds * IBM_NSM;
                if (best >= 0.f && 0.999f * best / rounds < hi) hi = 0.999f * best / rounds;     // dearer than the best so far
                if (p.cut(hi, most, nullptr, nullptr) < 0) continue;
                for (int it = 0; it < 14; ++it) {
                    const float mid = 0.5f * (lo + hi);
                    if (p.cut(mid, most, nullptr, nullptr) >= 0) hi = mid;
                    else lo = mid;
                }
                long long n = p.cut(hi, most, out, cost);
                float worst = 0.f;
                for (long long q = 0; q < n; ++q) {
                    worst = cost[q] > worst ? cost[q] : worst;
                    order[q] = (int)q;
                }
                const float total = worst * ((n + IBM_NSM - 1) / IBM_NSM);
                if (best >= 0.f && total >= 0.999f * best) continue;
                // the dearest first
                std::sort(order, order + n, [&](int a, int b) { return cost[a] != cost[b] ? cost[a] > cost[b] : a < b; });
                int4* sorted = (int4*)malloc(sizeof(int4) * n);
                if (!sorted) { e = cudaErrorMemoryAllocation; break; }
                for (long long q = 0; q < n; ++q) sorted[q] = out[order[q]];
                cudaFree(mg.fz);
                mg.fz = nullptr;
                e = ibm_malloc(&mg.fz, sizeof(int4) * n);
                if (e == cudaSuccess) e = cudaMemcpy(mg.fz, sorted, sizeof(int4) * n, cudaMemcpyHostToDevice);
                free(sorted);
                if (e != cudaSuccess) break;
                best = total;
                mg.flx = lx;
                mg.fz_items = (int)n;
                mg.fz_tx = p.tx;
                mg.fz_ty = p.ty;
            }
        }
        free(marks);
        free(sum);
        free(out);
        free(cost);
        free(order);
        if (e != cudaSuccess) return ibm_cuda_check(e, "multigrid set-up: plan of the fused passes");
    }
    return IBM_OK;
}

// ---- host side of the set-up --------------------------------------------------------------------

struct SetupTmp {
    long long* tiles = nullptr;     // scan tiles + 4 totals
    long long nt = 0;
    int* ovf = nullptr;
    uint8_t* sub0 = nullptr;
    int* lab = nullptr;             // union-find labels and part numbers of a level's unknowns
    int* num = nullptr;
    ~SetupTmp() {
        cudaFree(lab);
        cudaFree(num);
        cudaFree(tiles);
        cudaFree(ovf);
        cudaFree(sub0);
    }
};

void free_level(MGLev& L) {
    cudaFree(L.off); cudaFree(L.cnt); cudaFree(L.pos); cudaFree(L.rp); cudaFree(L.col); cudaFree(L.g);
    cudaFree(L.ecol); cudaFree(L.eg); cudaFree(L.eg8); cudaFree(L.d); cudaFree(L.invdg); cudaFree(L.parent); cudaFree(L.cp); cudaFree(L.ch); cudaFree(L.b);
    cudaFree(L.x); cudaFree(L.y);
    const int px = L.px, py = L.py, pz = L.pz;
    const long long P = L.P;
    memset(&L, 0, sizeof(L));
    L.px = px; L.py = py; L.pz = pz; L.P = P;
}

#define MG_ALLOC(ptr, n)                                                                         \
    do {                                                                                         \
        cudaError_t e_ = ibm_malloc(&(ptr), ((n) > 0 ? (size_t)(n) : 1) * sizeof(*(ptr))); \
        if (e_ != cudaSuccess) return ibm_cuda_check(e_, "multigrid set-up: " #ptr);              \
    } while (0)
#define MG_ALLOCB(ptr, bytes)                                                                    \
    do {                                                                                         \
        cudaError_t e_ = ibm_malloc(&(ptr), (size_t)(bytes) > 0 ? (size_t)(bytes) : 16); \
        if (e_ != cudaSuccess) return ibm_cuda_check(e_, "multigrid set-up: " #ptr);              \
    } while (0)

long long read_ll(const long long* d) {
    long long h = 0;
    cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost);
    return h;
}

// Colour-major offsets of the positions' unknowns; sets L.M0 and L.M.
int number_unknowns(MGLev& L, SetupTmp& t) {
    long long* tot = t.tiles + t.nt;
    IBM_CUDA(scan_emit(L.P, PosCount{L.cnt, L.px, L.py, 0}, PosEmit{L.off, L.px, L.py, 0, nullptr}, t.tiles, tot, 0));
    IBM_CUDA(scan_emit(L.P, PosCount{L.cnt, L.px, L.py, 1}, PosEmit{L.off, L.px, L.py, 1, tot}, t.tiles, tot + 1, 0));
    IBM_CUDA(cudaDeviceSynchronize());
    L.M0 = read_ll(tot);
    L.M = L.M0 + read_ll(tot + 1);
    if (L.M >= (1LL << 31)) return ibm_fail(IBM_E_INVALID, "multigrid set-up: too many unknowns");
    return IBM_OK;
}

// Exclusive scan of a[0..n) in place; a[n] = total.  Returns the total in *total.
int scan_in_place(int32_t* a, long long n, SetupTmp& t, long long* total) {
    long long* tot = t.tiles + t.nt + 2;
    IBM_CUDA(scan_emit(n, ArrCount{a}, ArrEmit{a}, t.tiles, tot, 0));
    IBM_CUDA(cudaDeviceSynchronize());
    *total = read_ll(tot);
    if (*total >= (1LL << 31)) return ibm_fail(IBM_E_INVALID, "multigrid set-up: too many links");
    const int32_t h = (int32_t)*total;
    IBM_CUDA(cudaMemcpy(a + n, &h, sizeof(h), cudaMemcpyHostToDevice));
    return IBM_OK;
}

int build_ell(MGLev& L, SetupTmp& t) {
    MG_ALLOC(L.ecol, MG_ELL * L.M);
    MG_ALLOC(L.eg8, L.M);
    IBM_CUDA(cudaMemset(t.ovf, 0, sizeof(int)));
    k_ell<<<lin_blocks(L.M), 256>>>(L, t.ovf);
    IBM_LAUNCHED("k_ell");
    int wide = 0;
    IBM_CUDA(cudaMemcpy(&wide, t.ovf, sizeof(int), cudaMemcpyDeviceToHost));
    if (!wide) return IBM_OK;
    cudaFree(L.eg8);
    L.eg8 = nullptr;
    MG_ALLOC(L.eg, MG_ELL * L.M);
    k_ell<<<lin_blocks(L.M), 256>>>(L, t.ovf);
    IBM_LAUNCHED("k_ell");
    return IBM_OK;
}

// Shares and shared-memory layout of the tail for levels first .. nlev - 1; its bytes per block (0: too large).
long long tail_layout(const MG& mg, MGTail& M, int first, int sb, int& rc) {
    const int last = mg.nlev - 1, blocks = first < last ? M.ctas : 1, most = (1 << M.shift) - 1;
    long long o = 0;
    auto take = [&](long long bytes) {
        const long long at = o;
        o += (bytes + 15) & ~15LL;
        return (int)at;
    };
    rc = IBM_OK;
    for (int l = first; l <= last; ++l) {
        const MGLev& L = mg.lev[l];
        MGTailLev& t = M.t[l];
        t.odd = L.odd;
        const long long M1 = L.M - L.M0;
        if (L.M > (long long)most * M.ctas || (l == last && L.M > most)) return 0;
        t.M = (int)L.M;
        t.M0 = (int)L.M0;
        const int nb = l < last ? blocks : 1;
        t.s0 = (int)((L.M0 + nb - 1) / nb);
        t.s1 = (int)((M1 + nb - 1) / nb);
        if (t.s0 < 1) t.s0 = 1;
        if (t.s1 < 1) t.s1 = 1;
        t.i0 = (unsigned)(0x100000000ULL / (unsigned)t.s0 + 1);      // s = 1 gives 2^32 + 1 = 1: see below
        t.i1 = (unsigned)(0x100000000ULL / (unsigned)t.s1 + 1);
        if ((t.s0 == 1 && L.M0 > 1) || (t.s1 == 1 && M1 > 1)) return 0;   // (a share of one: no such level is built)
        if (t.s0 == 1) t.i0 = 0;
        if (t.s1 == 1) t.i1 = 0;
        const long long S = t.s0 + t.s1;
        if (S > most) return 0;
        t.col = take(S * 2 * MG_ELL);
        t.pc = take(l < last ? S * 2 * MG_ELL : 0);
        t.g = take(S * sb * MG_ELL);
        t.dg = take(S * sb);
        t.d = take(sb == 8 || t.odd ? S * sb : 0);
        // the most children and the most links of long rows that any block holds
        int32_t *cp = nullptr, *rp = (int32_t*)malloc(sizeof(int32_t) * (L.M + 1));
        if (l > first) cp = (int32_t*)malloc(sizeof(int32_t) * (L.M + 1));
        cudaError_t e = cudaSuccess;
        if (rp) e = cudaMemcpy(rp, L.rp, sizeof(int32_t) * (L.M + 1), cudaMemcpyDeviceToHost);
        if (cp && e == cudaSuccess) e = cudaMemcpy(cp, L.cp, sizeof(int32_t) * (L.M + 1), cudaMemcpyDeviceToHost);
        long long children = 0, links = 0;
        bool fits = rp && (l == first || cp) && e == cudaSuccess;
        for (int r = 0; fits && r < nb; ++r) {
            long long nc = 0, nl = 0;
            for (int c = 0; c < 2; ++c) {
                const long long s1 = c ? t.s1 : t.s0, end = c ? L.M : L.M0, u0 = (c ? L.M0 : 0) + r * s1;
                for (long long u = u0; u < u0 + s1 && u < end; ++u) {
                    const int n = rp[u + 1] - rp[u];
                    if (n > MG_ELL) nl += n;
                    if (cp) {
                        nc += cp[u + 1] - cp[u];
                        fits = fits && cp[u + 1] - cp[u] < (1 << 13);
                    }
                }
            }
            children = nc > children ? nc : children;
            links = nl > links ? nl : links;
        }
        if (!rp || (l > first && !cp)) rc = ibm_fail(IBM_E_NOMEM, "multigrid set-up: host allocation");
        else if (e != cudaSuccess) rc = ibm_cuda_check(e, "multigrid set-up: tail");
        free(rp);
        free(cp);
        if (!fits || children >= (1 << 18) || links >= 65536) return 0;
        t.cv = take(l > first ? S * 4 : 0);
        t.ch = take(children * 2);
        t.oc = take(links * 2);
        t.op = take(l < last ? links * 2 : 0);
        t.og = take(links * sb);
    }
    M.image = (int)o;
    for (int l = first; l <= last; ++l) {
        MGTailLev& t = M.t[l];
        const long long S = t.s0 + t.s1;
        t.x = take(S * sb);
        t.b = take(S * sb);
        t.t = take(l < last || t.odd ? S * sb : 0);
    }
    return o <= 220 * 1024 ? o : 0;
}

cudaLaunchConfig_t tail_config(int blocks, int smem, cudaLaunchAttribute* at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(MG_TAIL_NT);
    cfg.dynamicSmemBytes = smem;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = blocks;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

template <class T>
auto tail_kernel(bool odd) { return odd ? k_mg_tail<T, true> : k_mg_tail<T, false>; }

// Whether the GPU can hold a cluster of MG_TAIL_BIG blocks (above the portable size).
bool tail_fits(int sb, int smem, bool odd) {
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = tail_config(MG_TAIL_BIG, smem, at);
    int n = 0;
    const cudaError_t e = sb == 8 ? cudaOccupancyMaxActiveClusters(&n, tail_kernel<double>(odd), &cfg)
                                  : cudaOccupancyMaxActiveClusters(&n, tail_kernel<float>(odd), &cfg);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess && n > 0;
}

// The tail starts at the first level whose shares fit, of those with at most MG_TAIL_MAX unknowns; a coarsest
// level too large for one block's shared memory runs from global memory (tail_smem = 0).
int tail_plan(MG& mg, int sb) {
    const int last = mg.nlev - 1;
    mg.tail_first = last;
    mg.tail_smem = 0;
    if (last < 1) return IBM_OK;
    bool odd = false;
    for (int l = 1; l <= last; ++l) odd = odd || mg.lev[l].odd;
    mg.tail_odd = odd;
    const void* const kernel = sb == 8 ? (const void*)tail_kernel<double>(odd) : (const void*)tail_kernel<float>(odd);
    IBM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    IBM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    mg.tail = (MGTail*)calloc(1, sizeof(MGTail));
    if (!mg.tail) return ibm_fail(IBM_E_NOMEM, "multigrid set-up: host allocation");
    for (int l = 0; l < IBM_MG_MAXLEV; ++l) mg.tail->lev[l] = mg.lev[l];
    mg.tail->nlev = mg.nlev;
    mg.tail->coarse_sweeps = mg.coarse_sweeps;
    mg.tail->omega = mg.omega;
    for (int l = 1; l <= last; ++l) {
        if (l < last && mg.lev[l].M > MG_TAIL_MAX) continue;
        for (int big = 1; big >= 0 && mg.tail_smem == 0; --big) {
            int rc;
            mg.tail->ctas = big ? MG_TAIL_BIG : 8;
            mg.tail->shift = big ? 12 : 13;
            const long long bytes = tail_layout(mg, *mg.tail, l, sb, rc);
            if (rc) return rc;
            if (bytes == 0 || (big && l < last && !tail_fits(sb, (int)bytes, odd))) continue;
            mg.tail->first = mg.tail_first = l;
            mg.tail_smem = (int)bytes;
        }
        if (mg.tail_smem > 0) break;
    }
    if (mg.tail_smem > 0) {
        const int blocks = mg.tail_first < last ? mg.tail->ctas : 1;
        int* cur = nullptr;
        MG_ALLOCB(mg.tail_img, (size_t)blocks * mg.tail->image);
        MG_ALLOC(cur, blocks * IBM_MG_MAXLEV);
        cudaError_t e = cudaMemset(cur, 0, sizeof(int) * blocks * IBM_MG_MAXLEV);
        if (e == cudaSuccess) e = cudaMemset(mg.tail_img, 0, (size_t)blocks * mg.tail->image);
        if (e == cudaSuccess) {
            mg.tail->img = (const uint4*)mg.tail_img;
            if (sb == 8) k_tail_image<double><<<blocks, 256>>>(*mg.tail, (unsigned char*)mg.tail_img, cur);
            else k_tail_image<float><<<blocks, 256>>>(*mg.tail, (unsigned char*)mg.tail_img, cur);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
        cudaFree(cur);
        if (e != cudaSuccess) return ibm_cuda_check(e, "multigrid set-up: tail");
    }
    return IBM_OK;
}

// Whether a level's periodic axes join positions of one colour.
int odd_level(const Dom& D, int px, int py, int pz) {
    const int n[3] = {px, py, pz};
    for (int a = 0; a < 3; ++a)
        if (D.bc[2 * a] == IBM_BC_PERIODIC && n[a] > 1 && n[a] % 2 == 1) return 1;
    return 0;
}

int build_level1(const LesCtx& c, MGLev& L, int sb, SetupTmp& t) {
    const Dom& D = c.D;
    L.px = (D.nx + 1) / 2;
    L.py = (D.ny + 1) / 2;
    L.pz = (D.nz + 1) / 2;
    L.P = (long long)L.px * L.py * L.pz;
    L.odd = odd_level(D, L.px, L.py, L.pz);
    MG_ALLOC(L.off, L.P);
    MG_ALLOC(L.cnt, L.P);
    k_parts1<<<lin_blocks(L.P), 256>>>(D, L, t.sub0);
    IBM_LAUNCHED("k_parts1");
    int rc = number_unknowns(L, t);
    if (rc) return rc;
    MG_ALLOC(L.pos, L.M);
    MG_ALLOC(L.rp, L.M + 1);
    MG_ALLOC(L.d, L.M);
    MG_ALLOC(L.invdg, L.M);
    MG_ALLOC(L.parent, L.M);
    MG_ALLOCB(L.b, L.M * sb);
    MG_ALLOCB(L.x, L.M * sb);
    if (L.odd) MG_ALLOCB(L.y, L.M * sb);
    IBM_CUDA(cudaMemset(t.ovf, 0, sizeof(int)));
    k_links1<<<lin_blocks(L.P), 256>>>(D, L, t.sub0, 0, t.ovf);
    IBM_LAUNCHED("k_links1");
    if ((rc = scan_in_place(L.rp, L.M, t, &L.nnz))) return rc;
    MG_ALLOC(L.col, L.nnz);
    MG_ALLOC(L.g, L.nnz);
    k_links1<<<lin_blocks(L.P), 256>>>(D, L, t.sub0, 1, t.ovf);
    IBM_LAUNCHED("k_links1");
    IBM_CUDA(cudaDeviceSynchronize());
    int h = 0;
    IBM_CUDA(cudaMemcpy(&h, t.ovf, sizeof(int), cudaMemcpyDeviceToHost));
    if (h) return ibm_fail(IBM_E_INVALID, "multigrid set-up: a level-1 block has too many links");
    MG_ALLOC(t.lab, L.M);           // the largest level: reused by the others
    MG_ALLOC(t.num, L.M);
    return build_ell(L, t);
}

// Level C from level F; returns 1 (and leaves C empty) when the level would not shrink enough or
// a row would not fit, 0 when built, < 0 on error (negated status).
int build_next(const Dom& D, MGLev& F, MGLev& C, int sb, SetupTmp& t) {
    C.px = (F.px + 1) / 2;
    C.py = (F.py + 1) / 2;
    C.pz = (F.pz + 1) / 2;
    C.P = (long long)C.px * C.py * C.pz;
    C.odd = odd_level(D, C.px, C.py, C.pz);
    MG_ALLOC(C.off, C.P);
    MG_ALLOC(C.cnt, C.P);
    k_uf_init<<<lin_blocks(F.M), 256>>>(F.M, t.lab, t.num);
    k_uf_union<<<lin_blocks(F.M), 256>>>(F, t.lab);
    k_parts_next<<<lin_blocks(C.P), 256>>>(F, C, t.lab, t.num);
    IBM_LAUNCHED("k_parts_next");
    int rc = number_unknowns(C, t);
    if (rc) return -rc;
    if (C.M > (F.M * 4) / 5) {
        free_level(C);
        return 1;
    }
    k_parent_next<<<lin_blocks(F.M), 256>>>(F, C);
    IBM_LAUNCHED("k_parent_next");
    MG_ALLOC(C.pos, C.M);
    MG_ALLOC(C.rp, C.M + 1);
    MG_ALLOC(C.cp, C.M + 1);
    const int all = sb == 8 || F.odd;
    const long long nchild = all ? F.M : F.M0;
    MG_ALLOC(C.ch, nchild);
    MG_ALLOC(C.d, C.M);
    MG_ALLOC(C.invdg, C.M);
    MG_ALLOC(C.parent, C.M);
    MG_ALLOCB(C.b, C.M * sb);
    MG_ALLOCB(C.x, C.M * sb);
    if (C.odd) MG_ALLOCB(C.y, C.M * sb);
    IBM_CUDA(cudaMemset(t.ovf, 0, sizeof(int)));
    k_links_next<<<lin_blocks(C.P), 256>>>(F, C, 0, all, t.ovf);
    IBM_LAUNCHED("k_links_next");
    IBM_CUDA(cudaDeviceSynchronize());
    int h = 0;
    IBM_CUDA(cudaMemcpy(&h, t.ovf, sizeof(int), cudaMemcpyDeviceToHost));
    if (h) {
        free_level(C);
        return 1;
    }
    long long nch = 0;
    if ((rc = scan_in_place(C.rp, C.M, t, &C.nnz))) return -rc;
    if ((rc = scan_in_place(C.cp, C.M, t, &nch))) return -rc;
    if (nch != nchild) return -ibm_fail(IBM_E_INVALID, "multigrid set-up: children do not cover the level");
    MG_ALLOC(C.col, C.nnz);
    MG_ALLOC(C.g, C.nnz);
    k_links_next<<<lin_blocks(C.P), 256>>>(F, C, 1, all, t.ovf);
    IBM_LAUNCHED("k_links_next");
    if ((rc = build_ell(C, t))) return -rc;
    IBM_CUDA(cudaDeviceSynchronize());
    return 0;
}

}  // namespace

// Level l with x as its passes left it (an odd level's separate ones end in y).
static MGLev solved(const MG& mg, int l) {
    MGLev L = mg.lev[l];
    if (L.odd && l < mg.tail_first) L.x = L.y;
    return L;
}

// Coarse levels of a V-cycle (level 1 holds the restricted residual and its first half-sweep; on return level 1
// holds the coarse correction): descent, coarsest solve and ascent, as separate kernels on the large levels
// and one cluster launch for the small ones (and always for the coarsest).
template <class T>
static int coarse_levels(const LesCtx& c, const MG& mg, SolveScal* sc, cudaStream_t s, int& launches) {
    const T om = (T)mg.omega;
    const int last = mg.nlev - 1, tf = mg.tail_first;
    for (int l = 1; l < tf; ++l) {
        const MGLev &L = mg.lev[l], &C = mg.lev[l + 1];
        if (L.odd) k_godd<T><<<lin_blocks(L.M - L.M0), 256, 0, s>>>(L, C, om, 0, sc);
        else k_gsmooth<T><<<lin_blocks(L.M - L.M0), 256, 0, s>>>(L, 1, sc);
        const unsigned nb = lin_blocks(4 * C.M);
        if constexpr (sizeof(T) == 8) k_grestrict<T, true><<<nb, 256, 0, s>>>(L, C, sc);
        else if (L.odd) k_grestrict<T, true><<<nb, 256, 0, s>>>(L, C, sc);
        else k_grestrict<T, false><<<nb, 256, 0, s>>>(L, C, sc);
        launches += 2;
    }
    if (mg.tail_smem > 0) {
        cudaLaunchAttribute at[1];
        cudaLaunchConfig_t cfg = tail_config(tf < last ? mg.tail->ctas : 1, mg.tail_smem, at);
        cfg.stream = s;
        IBM_CUDA(cudaLaunchKernelEx(&cfg, tail_kernel<T>(mg.tail_odd), *mg.tail, (const SolveScal*)sc));
    } else {
        k_gcoarsest<T><<<1, 1024, 0, s>>>(mg.lev[last], mg.coarse_sweeps, sc);
    }
    ++launches;
    for (int l = tf - 1; l >= 1; --l) {
        const MGLev& L = mg.lev[l];
        const MGLev C = solved(mg, l + 1);
        if (L.odd) {
            k_godd<T><<<lin_blocks(L.M - L.M0), 256, 0, s>>>(L, C, om, 1, sc);
            k_godd<T><<<lin_blocks(L.M0), 256, 0, s>>>(L, C, om, 2, sc);
        } else {
            k_gup<T><<<lin_blocks(L.M - L.M0), 256, 0, s>>>(L, C, om, sc);
            k_gsmooth<T><<<lin_blocks(L.M0), 256, 0, s>>>(L, 0, sc);
        }
        launches += 2;
    }
    return IBM_OK;
}

// Calls f(quads along x of a tile, values per row of a column) with the plan's constants.
template <class Fn>
static void fused_dispatch(const LesCtx& c, const MG& mg, Fn f) {
    using std::integral_constant;
    const bool vec = x4_ok(c);
    if (mg.flx == 16) vec ? f(integral_constant<int, 16>{}, integral_constant<int, 3>{}) : f(integral_constant<int, 16>{}, integral_constant<int, 4>{});
    else vec ? f(integral_constant<int, 32>{}, integral_constant<int, 3>{}) : f(integral_constant<int, 32>{}, integral_constant<int, 4>{});
}

// V-cycle with the fused fine-grid passes: pre-smoothing + restriction, the coarse levels,
// prolongation, post-smoothing + (r, z).
static int vcycle_fused(const LesCtx& c, const MG& mg, const float* r, float* z, SolveScal* sc, cudaStream_t s) {
    float* z2 = (float*)mg.z2;
    const float scale = (float)(c.D.dx * c.D.dx);
    const MGLev& L1 = mg.lev[1];
    int launches = 0;
    prof_begin(c.prof, PS_MG_FINE, s);
    auto pre = [&](auto lx, auto ni) {
        constexpr int LX = decltype(lx)::value, NI = decltype(ni)::value;
        k_mg_pre_fused<LX, NI><<<mg.fz_items, FTP_NT, FTile<LX>::smem(), s>>>(c.D, r, z2, scale, L1, mg.fz, mg.fz_tx, mg.fz_ty, sc);
    };
    fused_dispatch(c, mg, pre);
    prof_end(c.prof, PS_MG_FINE, s);
    ++launches;
    prof_begin(c.prof, PS_MG_COARSE, s);
    int rc = coarse_levels<float>(c, mg, sc, s, launches);
    if (rc) return rc;
    prof_end(c.prof, PS_MG_COARSE, s);
    prof_begin(c.prof, PS_MG_TRANSFER, s);
    if (x4_ok(c)) k_mg_prolong0_x4<<<lin_blocks((c.D.nx / 4) * (long long)L1.py * L1.pz), 256, 0, s>>>(c.D, z2, L1, (float)mg.omega, sc);
    else k_mg_prolong0<float><<<lin_blocks(L1.P), 256, 0, s>>>(c.D, z2, L1, (float)mg.omega, sc);
    prof_end(c.prof, PS_MG_TRANSFER, s);
    ++launches;
    prof_begin(c.prof, PS_MG_FINE, s);
    auto post = [&](auto lx, auto ni) {
        constexpr int LX = decltype(lx)::value, NI = decltype(ni)::value;
        k_mg_post_fused<LX, NI><<<mg.fz_items, FTP_NT, FTile<LX>::smem(), s>>>(c.D, r, z2, z, scale, mg.fz, mg.fz_tx, mg.fz_ty, sc, c.partials, c.counter);
    };
    fused_dispatch(c, mg, post);
    prof_end(c.prof, PS_MG_FINE, s);
    ++launches;
    IBM_LAUNCHED("mg_vcycle (fused)");
    IBM_COUNT(c, launches);
    return IBM_OK;
}

void mg_free(MG& mg) {
    for (int l = 1; l < IBM_MG_MAXLEV; ++l) free_level(mg.lev[l]);
    cudaFree(mg.z2);
    cudaFree(mg.fz);
    mg.fz = nullptr;
    cudaFree(mg.tail_img);
    mg.tail_img = nullptr;
    free(mg.tail);
    mg.tail = nullptr;
    mg.z2 = nullptr;
    mg.nlev = 1;
}

int mg_setup(const LesCtx& c, MG& mg, int sb) {
    for (int l = 0; l < IBM_MG_MAXLEV; ++l) memset(&mg.lev[l], 0, sizeof(MGLev));
    mg.fused = 0;
    MGLev& L0 = mg.lev[0];
    L0.px = c.D.nx;
    L0.py = c.D.ny;
    L0.pz = c.D.nz;
    L0.P = L0.M = c.D.N;
    mg.nlev = 1;
    mg.odd = odd_level(c.D, c.D.nx, c.D.ny, c.D.nz);
    if (mg.odd) MG_ALLOCB(mg.z2, c.D.N * sb);
    if (c.D.N <= MG_COARSE_TARGET) return IBM_OK;      // fine smoothing alone
    SetupTmp t;
    t.nt = scan_tiles(c.D.N);
    MG_ALLOC(t.tiles, t.nt + 4);
    MG_ALLOC(t.ovf, 1);
    MG_ALLOC(t.sub0, c.D.N);
    int rc = build_level1(c, mg.lev[1], sb, t);
    if (rc) return rc;
    mg.nlev = 2;
    for (int l = 1; l + 1 < IBM_MG_MAXLEV; ++l) {
        MGLev& F = mg.lev[l];
        if (F.M <= MG_COARSE_TARGET || F.P == 1) break;
        const int r2 = build_next(c.D, F, mg.lev[l + 1], sb, t);
        if (r2 < 0) return -r2;
        if (r2 > 0) break;
        mg.nlev = l + 2;
    }
    if ((rc = tail_plan(mg, sb))) return rc;
    if ((rc = fused_plan(c, mg, sb))) return rc;
    if (mg.fused) {
        MG_ALLOCB(mg.z2, c.D.N * 4);
        cudaError_t e = cudaSuccess;
        auto attr = [&](auto lx, auto ni) {
            constexpr int LX = decltype(lx)::value, NI = decltype(ni)::value;
            e = cudaFuncSetAttribute(k_mg_pre_fused<LX, NI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FTile<LX>::smem());
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k_mg_post_fused<LX, NI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FTile<LX>::smem());
        };
        fused_dispatch(c, mg, attr);
        if (e != cudaSuccess) return ibm_cuda_check(e, "multigrid set-up: fused passes");
    }
    return IBM_OK;
}

// z = V-cycle(r); the last kernel stores rz_old = rz, rz = (r, z).
template <class T>
int mg_vcycle(const LesCtx& c, const MG& mg, const T* r, T* z, SolveScal* sc, cudaStream_t s) {
    const T scale = (T)(c.D.dx * c.D.dx);
    const T om = (T)mg.omega;
    const int S = mg.sweeps;
    const CellGrid& g = c.cg;
    int launches = 0;
    bool vec = false;
    if constexpr (std::is_same<T, float>::value) vec = x4_ok(c);
    if constexpr (std::is_same<T, float>::value) {
        if (mg.fused) return vcycle_fused(c, mg, r, z, sc, s);
    }
    // one pair of planes per thread where four would leave SMs idle
    const bool few = (long long)c.cgrid.x * c.cgrid.y * c.cgrid.z < 4 * IBM_NSM;
    auto pairs = [&](auto f) {
        if (few) f(std::integral_constant<int, 1>{}, flat_grid(c.D.nx, c.D.ny, c.D.nz, 2));
        else f(std::integral_constant<int, IBM_KU>{}, c.cgrid);
    };
    // an odd grid's passes read a copy of the iterate
    const T* zin = mg.odd ? (const T*)mg.z2 : z;
    cudaError_t kept = cudaSuccess;
    auto keep = [&]() { return mg.odd ? cudaMemcpyAsync(mg.z2, z, sizeof(T) * c.D.N, cudaMemcpyDeviceToDevice, s) : cudaSuccess; };
    auto fine = [&](int col, int zero) {
        auto smooth = [&](auto ku, dim3 grid) {
            k_mg_smooth0<T, decltype(ku)::value><<<grid, g.block, 0, s>>>(c.D, r, z, zin, scale, col, zero, sc);
        };
        prof_begin(c.prof, PS_MG_FINE, s);
        if (!zero && kept == cudaSuccess) kept = keep();
        if constexpr (std::is_same<T, float>::value) {
            if (vec) launch_mg_smooth0_x4(c, r, z, zin, scale, col, zero, 0, sc, s);
            else pairs(smooth);
        } else {
            pairs(smooth);
        }
        prof_end(c.prof, PS_MG_FINE, s);
        ++launches;
    };
    for (int q = 0; q < S; ++q) {
        fine(0, q == 0);
        fine(1, 0);
    }
    if (mg.nlev > 1) {
        const MGLev &L1 = mg.lev[1], X1 = solved(mg, 1);
        prof_begin(c.prof, PS_MG_TRANSFER, s);
        if constexpr (std::is_same<T, float>::value) {
            if (vec) k_mg_restrict0_x4<<<lin_blocks((c.D.nx / 4) * (long long)L1.py * L1.pz), 256, 0, s>>>(c.D, r, z, scale, L1, sc);
            else k_mg_restrict0<T><<<lin_blocks(8 * L1.P), 256, 0, s>>>(c.D, r, z, scale, L1, sc);
        } else {
            k_mg_restrict0<T><<<lin_blocks(8 * L1.P), 256, 0, s>>>(c.D, r, z, scale, L1, sc);
        }
        prof_end(c.prof, PS_MG_TRANSFER, s);
        ++launches;
        prof_begin(c.prof, PS_MG_COARSE, s);
        int rc = coarse_levels<T>(c, mg, sc, s, launches);
        if (rc) return rc;
        prof_end(c.prof, PS_MG_COARSE, s);
        prof_begin(c.prof, PS_MG_TRANSFER, s);
        if constexpr (std::is_same<T, float>::value) {
            if (vec) k_mg_prolong0_x4<<<lin_blocks((c.D.nx / 4) * (long long)L1.py * L1.pz), 256, 0, s>>>(c.D, z, X1, om, sc);
            else k_mg_prolong0<T><<<lin_blocks(L1.P), 256, 0, s>>>(c.D, z, X1, om, sc);
        } else {
            k_mg_prolong0<T><<<lin_blocks(L1.P), 256, 0, s>>>(c.D, z, X1, om, sc);
        }
        prof_end(c.prof, PS_MG_TRANSFER, s);
        ++launches;
    }
    for (int q = 0; q < S; ++q) {
        fine(1, 0);
        if (q + 1 < S) fine(0, 0);
    }
    auto final = [&](auto ku, dim3 grid) {
        k_mg_final0<T, decltype(ku)::value><<<grid, g.block, 0, s>>>(c.D, r, z, zin, scale, sc, c.partials, c.counter);
    };
    prof_begin(c.prof, PS_MG_FINE, s);
    if (kept == cudaSuccess) kept = keep();
    if (kept != cudaSuccess) return ibm_cuda_check(kept, "mg_vcycle");
    if constexpr (std::is_same<T, float>::value) {
        if (vec) launch_mg_smooth0_x4(c, r, z, zin, scale, 0, 0, 1, sc, s);
        else pairs(final);
    } else {
        pairs(final);
    }
    prof_end(c.prof, PS_MG_FINE, s);
    ++launches;
    IBM_LAUNCHED("mg_vcycle");
    IBM_COUNT(c, launches);
    return IBM_OK;
}

template int mg_vcycle<float>(const LesCtx&, const MG&, const float*, float*, SolveScal*, cudaStream_t);
template int mg_vcycle<double>(const LesCtx&, const MG&, const double*, double*, SolveScal*, cudaStream_t);
