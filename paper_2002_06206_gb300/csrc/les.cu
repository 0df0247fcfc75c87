// les.cu -- the per-step stencil kernels of the immersed-boundary LES (Sec. 2.1-2.4): CSM eddy
// viscosity, the momentum flux with the QUICK hybrid and its two predictors (Crank-Nicolson with a
// BiCGStab momentum solve, Adams-Bashforth 2), distributed direct forcing, face velocities, Poisson
// right-hand side, velocity correction, and the Shepard surface and viscous forces.
//
// Cell kernels use a 32 x 8 thread tile over (x, y) so that consecutive threads touch consecutive
// cells (coalesced rows); the momentum flux walks z-marching tiles staged in shared memory, with the
// cells next to cut links in a separate general kernel.
#include <type_traits>

#include "scan.cuh"
#include "solver.cuh"

#ifndef IBM_FLUX_GEN_MINB
#define IBM_FLUX_GEN_MINB 5
#endif
#ifndef IBM_FLUX_MINB
#define IBM_FLUX_MINB 3
#endif

namespace {

template <class T>
__device__ __forceinline__ void grad_at(const Dom& D, const T* __restrict__ u, long long P, const int x[3],
                                        unsigned fl, T inv2dx, T G[3][3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const T up = vel_across(D, u, b, P, x[a], fl, a, +1);
            const T um = vel_across(D, u, b, P, x[a], fl, a, -1);
            G[a][b] = (up - um) * inv2dx;
        }
}

__device__ __forceinline__ unsigned flags_at(const Dom& D, long long P) { return D.flags ? (unsigned)D.flags[P] : 0u; }

// Domain-boundary ghost of component c across face (a, s) of the cell holding v (vel_across's rules).
template <class T>
__device__ __forceinline__ T bc_ghost(const Dom& D, int a, int s, int c, T v) {
    switch (D.bc[2 * a + (s > 0)]) {
        case IBM_BC_INFLOW: return (D.hom ? (T)0 : (T)2 * (T)D.u_in[c]) - v;
        case IBM_BC_OUTFLOW: return v;
        case IBM_BC_SLIP: return c == a ? -v : v;
        default: return -v;
    }
}

// base is the same for the whole block, the byte offset within a plane fixed per thread (a plane has less
// than 2^31/3 cells: 32 bits for FP32): one add per access.
template <class T>
using Off = std::conditional_t<sizeof(T) == 4, unsigned, unsigned long long>;

template <class T>
__device__ __forceinline__ T at_off(const T* base, Off<T> off) {
    return *reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + off);
}

template <class T>
__device__ __forceinline__ void to_off(T* base, Off<T> off, T v) {
    *reinterpret_cast<T*>(reinterpret_cast<char*>(base) + off) = v;
}

// Eq. Smagorinsky with the coherent-structure coefficient of Eq. Q / Eq. FCS.
//
// A thread marches through kz planes of one (x, y) column with the velocity of three planes in registers; the x
// neighbours come by shuffle, the rows above and below from L1.  Cells on a domain face take the boundary's ghosts
// in place; only cells with a cut link go through vel_across.  With g = the undivided central differences,
// 4 dx^2 S:S = A + B / 2 and 4 dx^2 W:W = C / 2 for A = sum g_aa^2, B = sum (g_ab + g_ba)^2, C = sum (g_ab - g_ba)^2.
// Bound by issue (87 %): 270 instructions per cell, addresses mostly; 266 us at 512 x 256 x 256 in FP32 (its 16 bytes per
// cell would take 80), 338 us with one thread per cell and 18 loads.
template <class T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 6 : 3) k_csm(Dom D, const T* __restrict__ u, T* __restrict__ nut, int kz) {
    const int i0 = blockIdx.x * IBM_TX + threadIdx.x, j0 = blockIdx.y * IBM_TY + threadIdx.y;
    const bool active = i0 < D.nx && j0 < D.ny;
    const int i = min(i0, D.nx - 1), j = min(j0, D.ny - 1);
    const int k0 = blockIdx.z * kz, k1 = min(k0 + kz, D.nz);
    const T scale = (T)(1.0 / 40.0) * dom_dx<T>(D);              // C / F^(3/2), dx^2 and 1 / (2 dx)
    long long xl = 0, xh = 0, yl = 0, yh = 0, zo = 0;
    const bool hxl = nb_offset(D, 0, -1, i, xl), hxh = nb_offset(D, 0, 1, i, xh);
    const bool hyl = nb_offset(D, 1, -1, j, yl), hyh = nb_offset(D, 1, 1, j, yh);
    const bool endl = threadIdx.x == 0 || i == 0, endh = threadIdx.x == 31 || i == D.nx - 1, both = endl && endh;
    // byte offsets within a plane: the cell, its y neighbours, the x neighbour a warp's end needs (the cell itself
    // where there is none)
    const int p = i + D.sy * j;
    const Off<T> o = (Off<T>)p * sizeof(T), oyl = (Off<T>)(p + (int)yl) * sizeof(T), oyh = (Off<T>)(p + (int)yh) * sizeof(T),
                 oe = (Off<T>)(p + (int)(endl ? xl : xh)) * sizeof(T), oh = (Off<T>)(p + (int)xh) * sizeof(T);
    const bool hx = hxl && hxh && hyl && hyh;
    const T* U0 = u + D.sz * k0;
    T m[3], v[3], n[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) v[c] = at_off(U0 + c * D.N, o);
    const bool hzl = nb_offset(D, 2, -1, k0, zo);
#pragma unroll
    for (int c = 0; c < 3; ++c) m[c] = hzl ? at_off(U0 + c * D.N + zo, o) : bc_ghost(D, 2, -1, c, v[c]);
    for (int k = k0; k < k1; ++k) {
        zo = 0;
        const bool hzh = nb_offset(D, 2, 1, k, zo);
        const T* Uk = u + D.sz * k;
        T gx[3], gy[3], gz[3], b[3], t[3], e[3] = {}, g[3] = {};
        // loads first, from the cell itself where there is no neighbour
#pragma unroll
        for (int c = 0; c < 3; ++c) n[c] = at_off(Uk + c * D.N + zo, o);
#pragma unroll
        for (int c = 0; c < 3; ++c) b[c] = at_off(Uk + c * D.N, oyl);
#pragma unroll
        for (int c = 0; c < 3; ++c) t[c] = at_off(Uk + c * D.N, oyh);
        if (endl || endh) {
#pragma unroll
            for (int c = 0; c < 3; ++c) e[c] = at_off(Uk + c * D.N, oe);
        }
        if (both) {
#pragma unroll
            for (int c = 0; c < 3; ++c) g[c] = at_off(Uk + c * D.N, oh);
        }
        const unsigned fl = D.flags ? (D.flags + D.sz * k)[(unsigned)p] & 63u : 0u;
        T l[3], h[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            l[c] = __shfl_up_sync(0xffffffffu, v[c], 1);
            h[c] = __shfl_down_sync(0xffffffffu, v[c], 1);
            if (endl) l[c] = e[c];
            if (endh) h[c] = both ? g[c] : e[c];
        }
        if (__any_sync(0xffffffffu, !(hx && hzh))) {    // ghosts of the domain faces
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                if (!hxl) l[c] = bc_ghost(D, 0, -1, c, v[c]);
                if (!hxh) h[c] = bc_ghost(D, 0, 1, c, v[c]);
                if (!hyl) b[c] = bc_ghost(D, 1, -1, c, v[c]);
                if (!hyh) t[c] = bc_ghost(D, 1, 1, c, v[c]);
                if (!hzh) n[c] = bc_ghost(D, 2, 1, c, v[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            gx[c] = h[c] - l[c];
            gy[c] = t[c] - b[c];
            gz[c] = n[c] - m[c];
        }
        if (__any_sync(0xffffffffu, fl != 0u) && fl != 0u) {
            const int x[3] = {i, j, k};
            T G[3][3];
            grad_at(D, u, p + D.sz * k, x, fl, (T)1, G);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                gx[c] = G[0][c];
                gy[c] = G[1][c];
                gz[c] = G[2][c];
            }
        }
        const T s0 = gx[1] + gy[0], s1 = gx[2] + gz[0], s2 = gy[2] + gz[1];
        const T w0 = gx[1] - gy[0], w1 = gx[2] - gz[0], w2 = gy[2] - gz[1];
        const T A = gx[0] * gx[0] + gy[1] * gy[1] + gz[2] * gz[2];
        const T SS = A + (T)0.5 * (s0 * s0 + s1 * s1 + s2 * s2), WW = (T)0.5 * (w0 * w0 + w1 * w1 + w2 * w2);
        const T E = WW + SS;
        const T F = E > (T)0 ? (WW - SS) / E : (T)0;
        const T aF = F < (T)0 ? -F : F;
        if (active) to_off(nut + D.sz * k, o, scale * (aF * sqrt(aF * SS)));
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            m[c] = v[c];
            v[c] = n[c];
        }
    }
}

// L(u) of a cell per unit volume: flux-form advection with the face velocity U, diffusion with nu + nu_t, the
// transpose part of the SGS stress divergence.  The advected value is the central one blended with a fraction gam
// of QUICK, (6 upwind + 3 downwind - far upwind) / 8, the far upwind value read across the upwind cell's outer
// link; cut faces and domain faces keep the central value.  flux_axis applies the ghost and boundary rules of
// vel_across on every link; the tiled fast path evaluates the same formulas for a cell where they reduce to direct
// reads (fast_cell).  With D.hom set the ghost values lose their wall and inflow velocities, which gives the linear
// part of L.

// The cell and its six neighbours (across periodic seams too) have no cut link: its flux then needs
// only neighbour values and the domain-boundary ghosts, which the tiles below hold.
__device__ __forceinline__ bool fast_cell(const Dom& D, long long P, int i, int j, int k) {
    if (!D.flags) return true;
    const uint8_t* f = D.flags;
    unsigned m = f[P];
    const int x[3] = {i, j, k};
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int s = -1; s <= 1; s += 2) {
            long long off;
            if (nb_offset(D, a, s, x[a], off)) m |= f[P + off];
        }
    return (m & 63u) == 0u;
}

// Fast cells run in z-marching tiles: a block of 32 x 8 threads owns an (x, y) tile and walks D.tile_z planes.  u
// (three components) and nu_t of the planes k-1 .. k+2 over the tile plus a two-cell halo sit in a ring in shared
// memory; a thread holds its own column in registers.  Halo positions across a periodic
// seam hold the wrapped cell; one cell beyond a non-periodic domain face they hold the boundary ghost of
// vel_across (a function of the cell across that face alone), so cells on the domain faces are fast too.
// A domain face takes the near cell's nu_t and cross derivative and the central advected value: weights
// (0, 2) or (2, 0) in place of (1, 1) and no QUICK share, so every face runs the same instructions.  Cells
// that are not fast_cell are skipped (the general kernel takes them).
//
// The flux form is conservative: the face between L and R = L + e_a gives L the term Phi and R the
// term -Phi, so the march evaluates every face once.  Each thread takes its cell's -x, -y and +z
// faces (two warps add the tile's last x column and y row); the x and y faces meet in shared memory,
// the z face stays in registers for the next plane.  A plane's sums run one step later, so a single
// barrier per plane orders both the face buffers (two of them, by plane parity) and the ring.
//
// Bound by instruction issue (65 %) and the latency of its barriers.  Per face and component the advected value is
// c_L u_L + c_R u_R - kq u_far with coefficients chosen once per face by the sign of its velocity, the scale factors of
// the differences are taken out of the components, and addresses are a block-uniform plane plus a fixed thread offset.
// 512x256x256 FP32, Crank-Nicolson operator: 660 us (490 thread instructions per cell; its 41 bytes per cell would take
// 205 us), 1540 us with per-component face forms, 64-bit face indexes and velocities loaded where they are used.  FP64:
// 183 us at 128x64x64, three quarters of the FP64 rate.
#define FT_X 32
#define FT_Y 8
#define FT_H 2
#define FT_SX (FT_X + 2 * FT_H)
#define FT_NV 4
#define FT_RING 5
#define FT_SY (FT_Y + 2 * FT_H)
#define FT_PL (FT_SX * FT_SY)          // halo-tile positions of a plane
#define FT_NT (FT_X * FT_Y)
#define FT_FXN (FT_Y * (FT_X + 1))     // x faces of a tile plane, per component
#define FT_FYN ((FT_Y + 1) * FT_X)     // y faces

// Coefficients of the faces of one axis at one place.
template <class T>
struct FaceW {
    T cu, cd, kq;  // the advected value is cu u_up + cd u_down - kq u_far
    T wl, wr;      // FP32: weights of the two cells in the cross derivatives (sum 2)
    bool lo, hi;   // domain face below, above: only the cell inside counts
    // wl a + wr b; by selection in FP64, where an operation costs more than four integer ones
    __device__ __forceinline__ T cross(T a, T b) const {
        if constexpr (sizeof(T) == 4) return wl * a + wr * b;
        else return (lo ? b : a) + (hi ? a : b);
    }
};

template <class T>
struct FaceK {
    T cu, cd, kq;          // interior faces
    T nui, h, e;           // nu / dx, 1 / (2 dx), 1 / (8 dx)
};

template <class T>
__device__ __forceinline__ FaceW<T> face_w(const FaceK<T>& K, bool dlo, bool dhi) {
    FaceW<T> w;
    w.wl = dlo ? (T)0 : (dhi ? (T)2 : (T)1);
    w.wr = dlo ? (T)2 : (dhi ? (T)0 : (T)1);
    w.lo = dlo;
    w.hi = dhi;
    w.cu = dlo || dhi ? (T)0.5 : K.cu;
    w.cd = dlo || dhi ? (T)0.5 : K.cd;
    w.kq = dlo || dhi ? (T)0 : K.kq;
    return w;
}

// Phi of the face between L = R - e_A and R, per component: the term of L's flux sum (R takes -Phi).
// far: the cell beyond the upwind one; d0, d1: wl dL + wr dR of the undivided central differences of u_A along
// the other two axes (in axis order); nn: nu_t of both cells, summed (a ghost holds the near cell's); Uf: the
// face velocity.
template <class T, int A>
__device__ __forceinline__ void face_phi(const FaceW<T>& w, const FaceK<T>& K, T Uf, const T (&l)[3], const T (&r)[3],
                                         const T (&far)[3], T d0, T d1, T nn, T (&phi)[3]) {
    const T a = K.nui + K.h * nn, x = K.e * nn, aa = a + K.h * nn;
    const bool up = Uf >= (T)0;
    const T cl = Uf * (up ? w.cu : w.cd), cr = Uf * (up ? w.cd : w.cu), cf = Uf * w.kq;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        T v = (c == A ? aa : a) * (r[c] - l[c]) + cf * far[c];
        v -= cl * l[c];
        v -= cr * r[c];
        if (c != A) v += x * (c == (A == 0 ? 1 : 0) ? d0 : d1);
        phi[c] = v;
    }
}

// The x (A = 0) or y (A = 1) face between ring position q - e_A and q of plane k.  S0: plane k, Sm, Sp: its
// neighbours; r: u at q; dz: undivided z difference of u_A at q.
template <class T, int A>
__device__ __forceinline__ void face_inplane(const FaceW<T>& w, const FaceK<T>& K, T Uf, const T* S0, const T* Sm,
                                             const T* Sp, int q, const T (&r)[3], T nr, T dz, T (&phi)[3]) {
    constexpr int E = A == 0 ? 1 : FT_SX, B = A == 0 ? FT_SX : 1;
    T l[3], far[3];
    const T* sf = S0 + q + (Uf >= (T)0 ? -2 * E : E);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        l[c] = S0[c * FT_PL + q - E];
        far[c] = sf[c * FT_PL];
    }
    const T* s = S0 + A * FT_PL + q;
    const T db = w.cross(s[B - E] - s[-B - E], s[B] - s[-B]);
    const T dzs = w.cross(Sp[A * FT_PL + q - E] - Sm[A * FT_PL + q - E], dz);
    face_phi<T, A>(w, K, Uf, l, r, far, db, dzs, S0[3 * FT_PL + q - E] + nr, phi);
}

// Calls epi(plane, off, h, u, w) for the fast cells: the cell is plane + off / sizeof(T), plane uniform; w holds
// the three values of `wv` at the cell (loaded a step ahead; unset where wv is null).
template <class T, class Epi>
__device__ __forceinline__ void fast_tile_march(const Dom& D, const FaceLayout& F, const T* __restrict__ u,
                                                const T* __restrict__ U, const T* __restrict__ nut, T nu, T gam,
                                                const T* wv, Epi epi) {
    extern __shared__ __align__(16) unsigned char ft_raw[];
    T* sm = reinterpret_cast<T*>(ft_raw);
    const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + FT_X * ty;
    const T invdx = dom_idx<T>(D);
    FaceK<T> K;
    K.kq = gam * (T)0.125;
    K.cd = (T)0.5 * ((T)1 - gam) + (T)3 * K.kq;
    K.cu = K.cd + (T)3 * K.kq;
    K.nui = nu * invdx;
    K.h = (T)0.5 * invdx;
    K.e = (T)0.125 * invdx;
    const int n[3] = {D.nx, D.ny, D.nz};
    const unsigned gx = (D.nx + FT_X - 1) / FT_X, gy = (D.ny + FT_Y - 1) / FT_Y, gz = (D.nz + D.tile_z - 1) / D.tile_z;
    const long long items = (long long)gx * gy * gz;
    // the planes' values a thread stages: two halo-tile positions (the second only where it exists), where they
    // are read from (byte offset within a plane: the wrapped cell across a periodic seam, the cell at the
    // face beyond a domain face) and what becomes of them: 0 as read, 1 + face: the ghost beyond that face, 7:
    // zero (corners and second ghost layers, which no fast cell reads)
    T pf[2][FT_NV];
    int x0 = 0, y0 = 0;
    Off<T> eo[2];
    unsigned kind = 0;
    const bool has1 = tid + FT_NT < FT_PL;
    // domain position along axis a of a coordinate beyond it
    auto beyond = [&](int a, int& g) -> unsigned {
        if (g >= 0 && g < n[a]) return 0u;
        if (D.bc[2 * a] == IBM_BC_PERIODIC) {
            g = ((g % n[a]) + n[a]) % n[a];
            return 0u;
        }
        const unsigned k = g == -1 ? 1u + 2 * a : (g == n[a] ? 2u + 2 * a : 7u);
        g = g < 0 ? 0 : n[a] - 1;
        return k;
    };
    auto places = [&]() {
        kind = 0;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int e = tid + t * FT_NT;
            int i = x0 + e % FT_SX - FT_H, j = y0 + e / FT_SX - FT_H;
            const unsigned kx = beyond(0, i), ky = beyond(1, j);
            kind |= (kx && ky ? 7u : kx | ky) << (4 * t);
            eo[t] = ((Off<T>)i + (Off<T>)D.sy * j) * sizeof(T);
        }
    };
    auto fetch = [&](int kk) {
        const unsigned kz = beyond(2, kk);
        const long long base = D.sz * kk;
        const T *b0 = u + base, *b1 = b0 + D.N, *b2 = b1 + D.N, *b3 = nut + base;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            if (t == 1 && !has1) break;
            pf[t][0] = at_off(b0, eo[t]);
            pf[t][1] = at_off(b1, eo[t]);
            pf[t][2] = at_off(b2, eo[t]);
            pf[t][3] = at_off(b3, eo[t]);
        }
        if (kind | kz) {
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const unsigned kt = (kind >> (4 * t)) & 7u;
                const unsigned k = kt && kz ? 7u : kt | kz;
                if (k == 0u) continue;
#pragma unroll
                for (int c = 0; c < 3; ++c) pf[t][c] = k == 7u ? (T)0 : bc_ghost(D, (int)(k - 1) >> 1, (k & 1u) ? -1 : 1, c, pf[t][c]);
                if (k == 7u) pf[t][3] = (T)0;
            }
        }
    };
    auto commit = [&](T* dst) {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            if (t == 1 && !has1) break;
#pragma unroll
            for (int v = 0; v < FT_NV; ++v) dst[v * FT_PL + tid + t * FT_NT] = pf[t][v];
        }
    };
    const int cidx = (ty + FT_H) * FT_SX + (tx + FT_H);
    T* const fxs = sm + FT_RING * FT_NV * FT_PL;                // [parity][component][FT_Y][FT_X + 1]
    T* const fys = fxs + 2 * 3 * FT_FXN;                        // [parity][component][FT_Y + 1][FT_X]
    const bool per0 = D.bc[0] == IBM_BC_PERIODIC, per1 = D.bc[2] == IBM_BC_PERIODIC, per2 = D.bc[4] == IBM_BC_PERIODIC;
    const long long sUx = (long long)F.dim[0][0] * F.dim[0][1], sUy = (long long)F.dim[1][0] * F.dim[1][1];
    const Off<T> row = (Off<T>)D.sy, rowx = (Off<T>)F.dim[0][0];
    for (long long item = blockIdx.x; item < items; item += gridDim.x) {
        // tiles of a grid of < 2^31 cells; a row of tiles starts one further along than the last, so that a
        // block does not come back to the same (slower) tiles at the domain faces
        const unsigned it = (unsigned)item, itx = it / gx;
        x0 = (int)((it + itx) % gx) * FT_X;
        y0 = (int)(itx % gy) * FT_Y;
        places();
        const int z0 = (int)(itx / gy) * D.tile_z;
        const int z1 = min(z0 + D.tile_z, D.nz);
        // ring planes of step k: k - 2 (then k + 3), k - 1, k, k + 1, k + 2
        T *Sa = sm, *Sm = sm + FT_NV * FT_PL, *S0 = sm + 2 * FT_NV * FT_PL, *Sp = sm + 3 * FT_NV * FT_PL, *Sq = sm + 4 * FT_NV * FT_PL;
        for (int q = 0; q < 5; ++q) {
            fetch(z0 - 2 + q);
            commit(sm + q * (FT_NV * FT_PL));
        }
        if (z0 + 3 <= z1 + 1) fetch(z0 + 3);
        __syncthreads();
        // faces of the thread: -x and -y of its cell (also of the first cell beyond the domain), +z; and the
        // face of the tile's last row (warp 0) or column (warp 1) it adds
        const int i = x0 + tx, j = y0 + ty;
        const bool in = i < D.nx && j < D.ny;
        const FaceW<T> wx = face_w(K, !per0 && i == 0, !per0 && i == D.nx), wy = face_w(K, !per1 && j == 0, !per1 && j == D.ny);
        // byte offsets from the tile's origin of a plane; places outside the domain read the origin (unused)
        const Off<T> oP = in ? (tx + row * ty) * sizeof(T) : 0;
        const Off<T> oUx = i <= D.nx && j < D.ny ? (tx + rowx * ty) * sizeof(T) : 0;
        const Off<T> oUy = i < D.nx && j <= D.ny ? (tx + row * ty) * sizeof(T) : 0;
        const bool exrow = ty == 0, excol = ty == 1 && tx < FT_Y;
        const int ei = x0 + FT_X, ej = exrow ? y0 + FT_Y : y0 + tx;
        const bool exin = exrow ? (i < D.nx && ej <= D.ny) : (excol && ei <= D.nx && ej < D.ny);
        const FaceW<T> we = exrow ? face_w(K, false, !per1 && ej == D.ny) : face_w(K, false, !per0 && ei == D.nx);
        const int eidx = exrow ? (FT_Y + FT_H) * FT_SX + tx + FT_H : (tx + FT_H) * FT_SX + FT_X + FT_H;
        const Off<T> oUe = exin ? (exrow ? tx + row * FT_Y : FT_X + rowx * tx) * sizeof(T) : 0;
        const T* Ux = U + F.index(0, x0, y0, z0);
        const T* Uy = U + F.index(1, x0, y0, z0);
        const T* Uz = U + F.index(2, x0, y0, z0);
        long long P = x0 + (long long)D.sy * y0 + D.sz * z0;
        // the thread's column: u of the planes k - 1 .. k + 1, nu_t of k, undivided in-plane differences of
        // u_z on plane k
        T um[3], uc[3], up[3], zlo[3], zhi[3] = {0, 0, 0}, nc, ex, ey;
        {
            const FaceW<T> wz = face_w(K, !per2 && z0 == 0, false);
            T far[3];
            const T Uf = at_off(Uz, oP);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                um[c] = Sm[c * FT_PL + cidx];
                uc[c] = S0[c * FT_PL + cidx];
                up[c] = Sp[c * FT_PL + cidx];
                far[c] = Uf >= (T)0 ? Sa[c * FT_PL + cidx] : up[c];
            }
            nc = S0[3 * FT_PL + cidx];
            const T *m = Sm + 2 * FT_PL + cidx, *o = S0 + 2 * FT_PL + cidx;
            ex = o[1] - o[-1];
            ey = o[FT_SX] - o[-FT_SX];
            face_phi<T, 2>(wz, K, Uf, um, uc, far, wz.cross(m[1] - m[-1], ex),
                           wz.cross(m[FT_SX] - m[-FT_SX], ey), Sm[3 * FT_PL + cidx] + nc, zlo);
        }
        // face velocities of the step's faces, loaded a step ahead
        T Ufx, Ufy, Ufz, Ufe;
        auto faces = [&]() {
            Ufx = at_off(Ux, oUx);
            Ufy = at_off(Uy, oUy);
            Ufz = at_off(Uz + D.sz, oP);
            Ufe = at_off(exrow ? Uy : Ux, oUe);
            Ux += sUx;
            Uy += sUy;
            Uz += D.sz;
        };
        faces();
        __syncthreads();                // the ring slot of plane z0 - 2 is free
        bool fast = false;
        T wq[3] = {};
        for (int k = z0; k <= z1; ++k, P += D.sz) {
            // plane k + 3, fetched into registers during the previous step, goes into the ring slot that
            // plane k - 2 left (the previous barrier ended every read of it); then plane k + 4 is fetched,
            // so each load has a whole step and a barrier to land.  The barrier at the end of the step
            // publishes plane k + 3.
            if (k < z1 && k + 3 <= z1 + 1) {
                commit(Sa);
                if (k + 4 <= z1 + 1) fetch(k + 4);
            }
            if (k > z0) {
                // sums of plane k - 1, whose faces the previous step wrote
                if (fast) {
                    const int pb = (k - 1) & 1;
                    const T* fx = fxs + pb * 3 * FT_FXN + ty * (FT_X + 1) + tx;
                    const T* fy = fys + pb * 3 * FT_FYN + ty * FT_X + tx;
                    T h[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        h[c] = ((fx[c * FT_FXN + 1] - fx[c * FT_FXN]) + (fy[c * FT_FYN + FT_X] - fy[c * FT_FYN]) +
                                (zhi[c] - zlo[c])) * invdx;
                    epi(P - D.sz, oP, h, um, wq);
                }
#pragma unroll
                for (int c = 0; c < 3; ++c) zlo[c] = zhi[c];
            }
            if (k == z1) break;
            fast = in && (D.fast ? D.fast[P + oP / sizeof(T)] != 0 : fast_cell(D, P + oP / sizeof(T), i, j, k));
            const int b = k & 1;
            T* fx = fxs + b * 3 * FT_FXN + ty * (FT_X + 1) + tx;
            T* fy = fys + b * 3 * FT_FYN + ty * FT_X + tx;
            T ph[3];
            face_inplane<T, 0>(wx, K, Ufx, S0, Sm, Sp, cidx, uc, nc, up[0] - um[0], ph);
#pragma unroll
            for (int c = 0; c < 3; ++c) fx[c * FT_FXN] = ph[c];
            face_inplane<T, 1>(wy, K, Ufy, S0, Sm, Sp, cidx, uc, nc, up[1] - um[1], ph);
#pragma unroll
            for (int c = 0; c < 3; ++c) fy[c * FT_FYN] = ph[c];
            {
                // the +z face
                const FaceW<T> wz = face_w(K, false, !per2 && k + 1 == D.nz);
                T uq[3], far[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    uq[c] = Sq[c * FT_PL + cidx];
                    far[c] = Ufz >= (T)0 ? um[c] : uq[c];
                }
                const T np = Sp[3 * FT_PL + cidx];
                const T* o = Sp + 2 * FT_PL + cidx;
                const T nx_ = o[1] - o[-1], ny_ = o[FT_SX] - o[-FT_SX];
                face_phi<T, 2>(wz, K, Ufz, uc, up, far, wz.cross(ex, nx_), wz.cross(ey, ny_), nc + np, zhi);
                ex = nx_;
                ey = ny_;
                nc = np;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    um[c] = uc[c];
                    uc[c] = up[c];
                    up[c] = uq[c];
                }
            }
            if (ty < 2) {
                // the +y faces of the tile's last row (ty = 0), the +x faces of its last column (ty = 1, row tx)
                T r[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) r[c] = S0[c * FT_PL + eidx];
                if (exrow) {
                    face_inplane<T, 1>(we, K, Ufe, S0, Sm, Sp, eidx, r, S0[3 * FT_PL + eidx], Sp[FT_PL + eidx] - Sm[FT_PL + eidx], ph);
#pragma unroll
                    for (int c = 0; c < 3; ++c) fy[c * FT_FYN + FT_Y * FT_X] = ph[c];
                } else if (excol) {
                    face_inplane<T, 0>(we, K, Ufe, S0, Sm, Sp, eidx, r, S0[3 * FT_PL + eidx], Sp[eidx] - Sm[eidx], ph);
                    T* fe = fxs + b * 3 * FT_FXN + tx * (FT_X + 1) + FT_X;
#pragma unroll
                    for (int c = 0; c < 3; ++c) fe[c * FT_FXN] = ph[c];
                }
            }
            if (k + 1 < z1) faces();
            if (wv) {
#pragma unroll
                for (int c = 0; c < 3; ++c) wq[c] = at_off(wv + c * D.N + P, oP);
            }
            T* const t = Sa;
            Sa = Sm;
            Sm = S0;
            S0 = Sp;
            Sp = Sq;
            Sq = t;
            __syncthreads();
        }
    }
}

template <class T>
size_t fast_tile_smem() { return (size_t)(FT_RING * FT_NV * FT_PL + 2 * 3 * (FT_FXN + FT_FYN)) * sizeof(T); }

// Values of the components a, a + 1, a + 2 (mod 3) that cell P reads across its link (a, s): vel_across for all
// three, with the kind of the link found once.  v: the cell's own values.
template <class T>
__device__ __forceinline__ void vel3_across(const Dom& D, const T* const (&u)[3], const int (&cm)[3], long long P, int xa,
                                            unsigned fl, int a, int s, const T (&v)[3], T (&o)[3]) {
    const int bit = link_bit(a, s);
    long long off;
    if (fl & (1u << bit)) {
        const LinkRec& r = link_record(D, P, fl, bit);
        const T cp = (T)r.c_p, ci = D.hom ? (T)0 : (T)r.c_ib, co = r.opp >= 0 ? (T)r.c_o : (T)0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            o[c] = (D.hom ? (T)0 : ci * (T)r.uib[cm[c]]) + cp * v[c];
            if (r.opp >= 0) o[c] = o[c] + co * u[c][r.opp];
        }
    } else if (nb_offset(D, a, s, xa, off)) {
#pragma unroll
        for (int c = 0; c < 3; ++c) o[c] = u[c][P + off];
    } else {
        const int k = D.bc[bit];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (k == IBM_BC_INFLOW) o[c] = (D.hom ? (T)0 : (T)2 * (T)D.u_in[cm[c]]) - v[c];
            else if (k == IBM_BC_OUTFLOW) o[c] = v[c];
            else o[c] = k == IBM_BC_SLIP && c > 0 ? v[c] : -v[c];
        }
    }
}

// Both faces of cell P along axis a, any links: contributions to the components a, a + 1, a + 2 (mod 3), which
// uP receives at the cell.
template <class T>
__device__ __forceinline__ void flux_axis(const Dom& D, const FaceLayout& F, const T* __restrict__ u,
                                          const T* __restrict__ U, const T* __restrict__ nut, long long P,
                                          const int (&x)[3], int a, T nu, T gam, T (&h)[3], T (&uP)[3]) {
    const T inv2dx = (T)0.5 * dom_idx<T>(D), invdx = dom_idx<T>(D);
    const int b = a == 2 ? 0 : a + 1, d = b == 2 ? 0 : b + 1, cm[3] = {a, b, d};
    const T* const uc[3] = {u + a * D.N, u + b * D.N, u + d * D.N};
    const int xa = a == 0 ? x[0] : (a == 1 ? x[1] : x[2]), xb = a == 0 ? x[1] : (a == 1 ? x[2] : x[0]),
              xd = a == 0 ? x[2] : (a == 1 ? x[0] : x[1]), na = a == 0 ? D.nx : (a == 1 ? D.ny : D.nz);
    const unsigned fl = flags_at(D, P);
    const T nutP = nut[P];
    const long long f0 = F.index(a, x[0], x[1], x[2]);
    const long long fs = a == 0 ? 1 : (a == 1 ? F.dim[1][0] : (long long)F.dim[2][0] * F.dim[2][1]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        uP[c] = uc[c][P];
        h[c] = (T)0;
    }
    // d u_a / d b and d u_a / d d at a cell with coordinates (.., xb, xd)
    auto cross = [&](long long Q, unsigned f, T& gb, T& gd) {
        gb = (vel_across(D, u, a, Q, xb, f, b, +1) - vel_across(D, u, a, Q, xb, f, b, -1)) * inv2dx;
        gd = (vel_across(D, u, a, Q, xd, f, d, +1) - vel_across(D, u, a, Q, xd, f, d, -1)) * inv2dx;
    };
    T GP[2];
    cross(P, fl, GP[0], GP[1]);
#pragma unroll 1
    for (int s = -1; s <= 1; s += 2) {
        const T Uf = U[f0 + (s > 0 ? fs : 0)], sg = (T)s;
        long long off = 0;
        const bool interior = !(fl & (1u << link_bit(a, s))) && nb_offset(D, a, s, xa, off);
        T uN[3], tt[2] = {sg * GP[0], sg * GP[1]}, nutf = nutP;
        vel3_across(D, uc, cm, P, xa, fl, a, s, uP, uN);
        T adv[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) adv[c] = (T)0.5 * (uP[c] + uN[c]);
        if (interior) {
            const long long Q = P + off;
            const unsigned fn = flags_at(D, Q);
            nutf = (T)0.5 * (nutP + nut[Q]);
            T GN[2];
            cross(Q, fn, GN[0], GN[1]);
#pragma unroll
            for (int c = 0; c < 2; ++c) tt[c] = sg * (T)0.5 * (GP[c] + GN[c]);
            if (gam != (T)0) {
                // far upwind value: across the outer link of the upwind cell
                const bool up = (Uf >= (T)0) == (s > 0);        // P is the upwind cell
                const int xn = xa + s < 0 ? na - 1 : (xa + s >= na ? 0 : xa + s);
                T v[3], w[3], far[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    v[c] = up ? uP[c] : uN[c];
                    w[c] = up ? uN[c] : uP[c];
                }
                vel3_across(D, uc, cm, up ? P : Q, up ? xa : xn, up ? fl : fn, a, up ? -s : s, v, far);
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    adv[c] = ((T)1 - gam) * adv[c] + gam * (((T)6 * v[c] + (T)3 * w[c] - far[c]) * (T)0.125);
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T D1 = (uN[c] - uP[c]) * invdx;
            h[c] += (nu + nutf) * D1 + nutf * (c == 0 ? D1 : tt[c > 0 ? c - 1 : 0]) - sg * Uf * adv[c];
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) h[c] *= invdx;
}

// (grids hold fewer than 2^31 cells: 32-bit division)
__device__ __forceinline__ void cell_coords(const Dom& D, long long P, int& i, int& j, int& k) {
    const unsigned u = (unsigned)P, sy = (unsigned)D.sy, sz = (unsigned)D.sz;
    const unsigned kk = u / sz, r = u - kk * sz, jj = r / sy;
    k = (int)kk;
    j = (int)jj;
    i = (int)(r - jj * sy);
}

// Cells that are not fast_cell, from their list.  A warp takes one axis of 32 cells, so that what depends on the axis
// is uniform in it, and three warps make up the cells: they leave their shares of the three components in shared
// memory and each finishes one component.  Bound by the latency of the scattered reads.  1024 x 512 x 384 around a
// vehicle, Crank-Nicolson operator: 1.8 ms; 3.9 ms with one thread per cell and all six faces unrolled, which waited for
// instructions (a thousand per face) and spilled.
#define FG_CELLS 64
#define FG_NT (3 * FG_CELLS)

template <class T, class Epi>
__device__ __forceinline__ void general_march(const Dom& D, const FaceLayout& F, const T* __restrict__ u,
                                              const T* __restrict__ U, const T* __restrict__ nut, T nu, T gam,
                                              const int32_t* __restrict__ list, long long nlist, const T* wv, Epi epi) {
    __shared__ T part[2][3][3][FG_CELLS];           // [parity][axis][component][cell]
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), a = warp % 3;
    const int cell = 32 * (warp / 3) + (threadIdx.x & 31);
    int buf = 0;
    for (long long q0 = blockIdx.x * (long long)FG_CELLS; q0 < nlist; q0 += (long long)gridDim.x * FG_CELLS) {
        const bool on = q0 + cell < nlist;
        const long long P = on ? list[q0 + cell] : 0;
        T uP[3] = {}, w = (T)0;
        if (on) {
            int x[3];
            cell_coords(D, P, x[0], x[1], x[2]);
            if (wv) w = wv[a * D.N + P];
            T h[3];
            flux_axis(D, F, u, U, nut, P, x, a, nu, gam, h, uP);
#pragma unroll
            for (int c = 0; c < 3; ++c) part[buf][a][a + c < 3 ? a + c : a + c - 3][cell] = h[c];
        }
        __syncthreads();
        if (on) epi(a * D.N + P, 0, (part[buf][0][a][cell] + part[buf][1][a][cell]) + part[buf][2][a][cell], uP[0], w);
        buf ^= 1;
    }
}

// Runs epi(q, off, h, u, w) for every component of the kernel's cells (value q + off / sizeof(T) of the stacked
// components, w = wv there): z-marching shared-memory tiles of fast cells, or the general list.
template <bool GENERAL, class T, class Epi>
__device__ __forceinline__ void flux_cells(const Dom& D, const FaceLayout& F, const T* __restrict__ u,
                                           const T* __restrict__ U, const T* __restrict__ nut, T nu, T gam,
                                           const int32_t* __restrict__ list, long long nlist, const T* wv, Epi epi) {
    if constexpr (GENERAL) {
        general_march<T>(D, F, u, U, nut, nu, gam, list, nlist, wv, epi);
    } else {
        fast_tile_march<T>(D, F, u, U, nut, nu, gam, wv,
                           [&](long long P, Off<T> o, const T (&h)[3], const T (&uc)[3], const T (&w)[3]) {
#pragma unroll
            for (int c = 0; c < 3; ++c) epi(c * D.N + P, o, h[c], uc[c], w[c]);
        });
    }
}

// Resident blocks per SM the flux kernels are compiled for (register cap), and their threads.
template <class T, bool GENERAL>
struct FluxOcc {
    static constexpr int value = sizeof(T) == 4 ? (GENERAL ? IBM_FLUX_GEN_MINB : IBM_FLUX_MINB) : (GENERAL ? 2 : 1);
    static constexpr int threads = GENERAL ? FG_NT : 256;
};

// Momentum predictor, Adams-Bashforth 2 in time (Euler on the first step).
template <bool GENERAL, class T>
__global__ void __launch_bounds__((FluxOcc<T, GENERAL>::threads), (FluxOcc<T, GENERAL>::value)) k_predict(Dom D, FaceLayout F, const T* __restrict__ u, const T* __restrict__ U,
                                                 const T* __restrict__ nut, const T* Hprev, T* H,
                                                 T* __restrict__ ustar, T nu, T dt, int first, T gam,
                                                 const int32_t* __restrict__ list, long long nlist) {
    flux_cells<GENERAL, T>(D, F, u, U, nut, nu, gam, list, nlist, first ? nullptr : Hprev,
                           [&](long long q, Off<T> o, T h, T uc, T w) {
        to_off(H + q, o, h);
        to_off(ustar + q, o, first ? uc + dt * h : uc + dt * ((T)1.5 * h - (T)0.5 * w));
    });
}

// Distributed direct forcing (Eq. forcing_term, Eq. discrete_forcing_term), gathered per Omega_inc
// cell over its own link records: the velocity at the wall point X is interpolated between the cell
// and the cell behind the wall, the force (u_IB - u_X)/dt is spread to the cell with the ghost branch
// (dx - d)/(dx + d) of Eq. distribution_function (the cell is a ghost of the stencil across the wall;
// weight 1 at d = 0 puts it on u_IB), and a cell whose weights add up to more than 1 takes their
// normalised sum.  All reads use the unforced u*, so the result does not depend on thread order.
template <class T>
__global__ void __launch_bounds__(256) k_forcing_gather(Dom D, const int32_t* __restrict__ inc, long long n_inc,
                                                        const T* __restrict__ us, double* __restrict__ delta, T dt,
                                                        int deadend_on, double vol, double* partials,
                                                        unsigned* counter, double* fscal) {
    double acc[3] = {0.0, 0.0, 0.0};
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n_inc; q += (long long)gridDim.x * blockDim.x) {
        const long long X = inc[q];
        const unsigned fl = D.flags[X];
        T d3[3] = {0, 0, 0};
        T wsum = 0;
        const bool dead = deadend_on && __popc(fl & 63u) >= 5;
        if (!dead) {
            for (int bit = 0; bit < 6; ++bit) {
                if (!((fl >> bit) & 1u)) continue;
                const LinkRec& r = link_record(D, X, fl, bit);
                const long long G = r.far;
                const T d = (T)r.d, wn = (T)r.w_ghost;
                wsum += wn;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const T uX = ((T)1 - d) * us[c * D.N + X] + d * us[c * D.N + G];
                    const T Fc = ((T)r.uib[c] - uX) / dt;
                    d3[c] += dt * wn * Fc;
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T dc = wsum > (T)1 ? d3[c] / wsum : d3[c];
            delta[3 * q + c] = (double)dc;
            acc[c] += (double)dc * vol;
        }
    }
    grid_reduce<3>(acc, partials, counter, [&](double* tot) {
        fscal[0] = tot[0];
        fscal[1] = tot[1];
        fscal[2] = tot[2];
    });
}

template <class T>
__global__ void k_forcing_apply(Dom D, const int32_t* __restrict__ inc, long long n_inc, const double* __restrict__ delta,
                                T* __restrict__ us) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n_inc; q += (long long)gridDim.x * blockDim.x) {
        const long long X = inc[q];
#pragma unroll
        for (int c = 0; c < 3; ++c) us[c * D.N + X] = us[c * D.N + X] + (T)delta[3 * q + c];
    }
}

// Normal velocity of the wall on a cut face between cells L and R along a: the mean of u_IB.e_a over
// the face's link records (L's +a record and, when present, R's -a record), in FP64.
__device__ __forceinline__ double cut_face_velocity(const Dom& D, long long L, long long R, int a) {
    const unsigned fL = D.flags[L], fR = D.flags[R];
    double sum = link_record(D, L, fL, 2 * a + 1).uib[a];
    double n = 1.0;
    if ((fR >> (2 * a)) & 1u) {
        sum += link_record(D, R, fR, 2 * a).uib[a];
        n = 2.0;
    }
    return sum / n;
}

// A thread of the face and correction kernels takes one (x, y) column of `kz` planes, so the z neighbour
// of a plane is the register of the next; kz falls to 1 on grids that would give fewer than `least` blocks.
inline dim3 column_grid(const Dom& D, int& kz, long long least = 8LL * IBM_NSM) {
    const long long bxy = (long long)((D.nx + IBM_TX - 1) / IBM_TX) * ((D.ny + IBM_TY - 1) / IBM_TY);
    kz = 8;
    while (kz > 1 && bxy * ((D.nz + kz - 1) / kz) < least) kz >>= 1;
    return flat_grid(D.nx, D.ny, D.nz, kz);
}

// Value of the face (a, s) of a cell on a domain side: `in` is the cell's own value, ua[wrap] that of the cell
// across a periodic seam.
template <class T>
__device__ __forceinline__ T domain_face(const Dom& D, int a, int s, T in, const T* __restrict__ ua, long long wrap) {
    switch (D.bc[2 * a + (s > 0)]) {
        case IBM_BC_PERIODIC: return (T)0.5 * (s < 0 ? ua[wrap] + in : in + ua[wrap]);
        case IBM_BC_INFLOW: return (T)D.u_in[a];
        case IBM_BC_OUTFLOW: return in;
        default: return (T)0;
    }
}

// Face velocity of the intermediate field: the mean of the two cell values on uncut interior faces, the
// wall's normal velocity on cut faces (zero for a stationary body), the boundary value on domain faces.
// One thread per cell writes its three lower faces (and the upper one of the last cell of an axis), so the
// three components are read once and no face index has to be taken apart.  A cell knows a cut lower face
// from its own flags: ibm_setup accepts only flags in which both cells of a face agree.  512x256x256 FP32:
// 181 us (4.6 TB/s of the 25 bytes per cell; bound by latency: six blocks per SM and two planes in flight; four planes
// at three blocks took 260), 660 us as one grid-stride kernel per axis with 64-bit divisions.
template <class T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 6 : 3) k_faces(Dom D, FaceLayout F, const T* __restrict__ us, T* __restrict__ Us, int kz) {
    const int i = blockIdx.x * IBM_TX + threadIdx.x, j = blockIdx.y * IBM_TY + threadIdx.y;
    const int k0 = blockIdx.z * kz, k1 = min(k0 + kz, D.nz);
    if (i >= D.nx || j >= D.ny) return;
    const long long P0 = i + (long long)D.sy * j + D.sz * k0;
    const T* __restrict__ u0 = us + P0;
    const T* __restrict__ u1 = us + D.N + P0;
    const T* __restrict__ u2 = us + 2 * D.N + P0;
    T* __restrict__ X = Us + F.index(0, i, j, k0);
    T* __restrict__ Y = Us + F.index(1, i, j, k0);
    T* __restrict__ Z = Us + F.index(2, i, j, k0);
    const long long sfx = (long long)F.dim[0][0] * F.dim[0][1], sfy = (long long)F.dim[1][0] * F.dim[1][1];
    // the cell across the lower x and y face; at a domain face the cell itself (replaced below)
    const int ox = i > 0 ? -1 : 0, oy = j > 0 ? -D.sy : 0;
    const bool edge = i == 0 || j == 0 || i == D.nx - 1 || j == D.ny - 1;
    T zm = k0 > 0 ? u2[-D.sz] : (T)0;
    const int nk = k1 - k0;
#pragma unroll 2
    for (int q = 0; q < nk; ++q) {
        const long long o = q * D.sz;
        const unsigned fl = D.flags ? (unsigned)D.flags[P0 + o] : 0u;
        const T cx = u0[o], cy = u1[o], cz = u2[o];
        T vx = (T)0.5 * (u0[o + ox] + cx), vy = (T)0.5 * (u1[o + oy] + cy), vz = (T)0.5 * (zm + cz);
        if (fl & 21u) {
            const long long P = P0 + o;
            if (fl & 1u) vx = (T)cut_face_velocity(D, P - 1, P, 0);
            if (fl & 4u) vy = (T)cut_face_velocity(D, P - D.sy, P, 1);
            if (fl & 16u) vz = (T)cut_face_velocity(D, P - D.sz, P, 2);
        }
        const int k = k0 + q;
        if (edge || k == 0 || k == D.nz - 1) {
            if (i == 0) vx = domain_face(D, 0, -1, cx, u0 + o, (long long)D.nx - 1);
            if (j == 0) vy = domain_face(D, 1, -1, cy, u1 + o, (long long)(D.ny - 1) * D.sy);
            if (k == 0) vz = domain_face(D, 2, -1, cz, u2 + o, (long long)(D.nz - 1) * D.sz);
            if (i == D.nx - 1) X[q * sfx + 1] = domain_face(D, 0, 1, cx, u0 + o, -(long long)i);
            if (j == D.ny - 1) Y[q * sfy + D.nx] = domain_face(D, 1, 1, cy, u1 + o, -(long long)j * D.sy);
            if (k == D.nz - 1) Z[o + D.sz] = domain_face(D, 2, 1, cz, u2 + o, -(long long)k * D.sz);
        }
        X[q * sfx] = vx;
        Y[q * sfy] = vy;
        Z[o] = vz;
        zm = cz;
    }
}

// Net boundary flux: fscal[3] = outward flux of inflow faces, fscal[4] = of outflow faces,
// fscal[5] = number of outflow faces.  Only the planes of these two types are walked.
template <class T>
__global__ void __launch_bounds__(256) k_boundary_flux(Dom D, FaceLayout F, const T* __restrict__ Us, double* partials,
                                                       unsigned* counter, double* fscal) {
    const int n[3] = {D.nx, D.ny, D.nz};
    double acc[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int p = 0; p < 6; ++p) {
        const int bc = D.bc[p];
        if (bc != IBM_BC_INFLOW && bc != IBM_BC_OUTFLOW) continue;
        const int a = p >> 1, s = (p & 1) ? 1 : -1;
        const int b = a == 0 ? 1 : 0, c = a == 2 ? 1 : 2;         // the plane's axes, the faster one first
        const unsigned np = (unsigned)n[b] * (unsigned)n[c];      // a plane of a grid of < 2^31 cells
        for (unsigned r = blockIdx.x * blockDim.x + threadIdx.x; r < np; r += gridDim.x * blockDim.x) {
            int x[3];
            x[c] = (int)(r / (unsigned)n[b]);
            x[b] = (int)(r - (unsigned)x[c] * (unsigned)n[b]);
            x[a] = s < 0 ? 0 : n[a];
            const double v = (double)Us[F.index(a, x[0], x[1], x[2])];
            if (bc == IBM_BC_INFLOW) acc[0] += s * v;
            else { acc[1] += s * v; acc[2] += 1.0; }
        }
    }
    grid_reduce<3>(acc, partials, counter, [&](double* t) {
        fscal[3] = t[0];
        fscal[4] = t[1];
        fscal[5] = t[2];
    });
}

template <class T>
__global__ void k_outflow_shift(Dom D, FaceLayout F, T* __restrict__ Us, const double* __restrict__ fscal) {
    const double nout = fscal[5];
    if (nout == 0.0) return;
    const double shift = (-fscal[3] - fscal[4]) / nout;
    const int n[3] = {D.nx, D.ny, D.nz};
    for (int p = 0; p < 6; ++p) {
        if (D.bc[p] != IBM_BC_OUTFLOW) continue;
        const int a = p >> 1, s = (p & 1) ? 1 : -1;
        const int b = a == 0 ? 1 : 0, c = a == 2 ? 1 : 2;
        const unsigned np = (unsigned)n[b] * (unsigned)n[c];
        for (unsigned r = blockIdx.x * blockDim.x + threadIdx.x; r < np; r += gridDim.x * blockDim.x) {
            int x[3];
            x[c] = (int)(r / (unsigned)n[b]);
            x[b] = (int)(r - (unsigned)x[c] * (unsigned)n[b]);
            x[a] = s < 0 ? 0 : n[a];
            const long long fi = F.index(a, x[0], x[1], x[2]);
            Us[fi] = (T)((double)Us[fi] + s * shift);
        }
    }
}

// Eq. poisson right-hand side: b = div(U*) / dt, evaluated in the working precision and stored in
// FP64 (the pressure solve's FP64 residual b - A p starts from it).  A thread marches a column and keeps the z face
// it shares with the next cell.  512x256x256 FP32: 110 us (20 bytes per cell would take 99), 157 us with one thread
// per cell and a 64-bit index for each of its six faces.
template <class T>
__global__ void __launch_bounds__(256, 8) k_rhs(Dom D, FaceLayout F, const T* __restrict__ Us, double* __restrict__ b,
                                                double inv_dxdt, int kz) {
    const int i = blockIdx.x * IBM_TX + threadIdx.x, j = blockIdx.y * IBM_TY + threadIdx.y;
    const int k0 = blockIdx.z * kz, nk = min(kz, D.nz - k0);
    if (i >= D.nx || j >= D.ny) return;
    const T inv = (T)inv_dxdt;
    const T* __restrict__ X = Us + F.index(0, i, j, k0);
    const T* __restrict__ Y = Us + F.index(1, i, j, k0);
    const T* __restrict__ Z = Us + F.index(2, i, j, k0);
    double* __restrict__ o = b + i + (long long)D.sy * j + D.sz * k0;
    const long long sfx = (long long)F.dim[0][0] * F.dim[0][1], sfy = (long long)F.dim[1][0] * F.dim[1][1];
    T z = Z[0];
#pragma unroll 4
    for (int q = 0; q < nk; ++q, X += sfx, Y += sfy, Z += D.sz, o += D.sz) {
        const T x0 = X[0], x1 = X[1], y0 = Y[0], y1 = Y[D.nx], z1 = Z[D.sz];
        *o = (double)((((x1 - x0) + (y1 - y0)) + (z1 - z)) * inv);
        z = z1;
    }
}

// A pressure held for differences that are rounded to the working precision.  FP64 mode: the double itself.
// FP32 mode: hi + mid + lo, the double's leading 24 bits and the 16 and 13 below them as three floats, all exact,
// taken from its bits: GB300 issues an FP64 subtraction or conversion at 1/70 of the FP32 rate, and six differences
// per cell made the correction FP64 bound.  `minus` keeps the rounding errors of its two large terms, so the result is
// the exact difference rounded once, however much of the two values cancels, as an FP64 subtraction rounded to FP32
// gives it (a tie may round the other way).  Values whose low part leaves the normal range of a float (below 2^-74, above
// 2^126, not finite) set `odd`: the cell then takes FP64 arithmetic.
template <class T> struct PVal;
template <> struct PVal<double> {
    double v;
    __device__ __forceinline__ PVal(double x, bool&) : v(x) {}
    __device__ __forceinline__ PVal neg() const { PVal r(*this); r.v = -v; return r; }
    __device__ __forceinline__ double minus(const PVal& o) const { return v - o.v; }
};
template <> struct PVal<float> {
    float hi, mid, lo;
    __device__ __forceinline__ PVal(double x, bool& odd) {
        const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
        // exponents 949 .. 1148 (and zero): the float's exponent is the low eight bits with the top one flipped
        const unsigned m = h & 0x7fffffffu;
        odd = odd || (m - (949u << 20) > (200u << 20) && (m | l) != 0u);
        const unsigned b = (__funnelshift_l(l, h, 3) ^ 0x40000000u) & 0x7fffffffu;
        const unsigned f = m == 0u ? 0u : b | (h & 0x80000000u), e = f & 0xff800000u;
        hi = __uint_as_float(f);
        // (whole numbers below 2^23 by way of 2^23 + n: conversions run at an eighth of the FP32 rate)
        mid = __uint_as_float(e - (39u << 23)) * (__uint_as_float(0x4b000000u | ((l >> 13) & 0xffffu)) - 8388608.f);
        lo = __uint_as_float(e - (52u << 23)) * (__uint_as_float(0x4b000000u | (l & 0x1fffu)) - 8388608.f);
    }
    __device__ __forceinline__ PVal neg() const {
        PVal r(*this);
        r.hi = -hi;
        r.mid = -mid;
        r.lo = -lo;
        return r;
    }
    __device__ __forceinline__ float minus(const PVal& o) const {
        // the rounding error of the leading difference (any order of the two) ...
        const float d = __fsub_rn(hi, o.hi), t = __fsub_rn(d, hi), e1 = __fsub_rn(__fsub_rn(hi, __fsub_rn(d, t)), __fadd_rn(o.hi, t));
        // ... and of the sum with the middle one, which is exact where that is the larger
        const float m = __fsub_rn(mid, o.mid), s = __fadd_rn(d, m), e2 = __fsub_rn(m, __fsub_rn(s, d));
        return s + ((e1 + e2) + (lo - o.lo));
    }
};

// Eq. correction: cells by the central pressure difference through the link values (c = dt / (2 dx)), faces
// by the compact difference across uncut interior and outflow faces (dtdx = dt / dx).  One thread per cell
// updates the cell, its three lower faces and the upper one of the last cell of an axis, marching a column:
// p, u*, U* and the flags are read once.  The differences along y are left to the FP64 units, which are idle beside
// those of split pressures.  512x256x256 FP32: 416 us (4.6 TB/s of the 57 bytes per cell), 475 us with all differences
// from split pressures; 930 us as one cell and three face kernels in FP64 differences.
template <class T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2) k_correct(Dom D, FaceLayout F, const T* __restrict__ us, const T* __restrict__ Us,
                                                 const double* __restrict__ p, T* __restrict__ u, T* __restrict__ U, T c,
                                                 T dtdx, int kz) {
    const int i = blockIdx.x * IBM_TX + threadIdx.x, j = blockIdx.y * IBM_TY + threadIdx.y;
    const int k0 = blockIdx.z * kz, k1 = min(k0 + kz, D.nz);
    if (i >= D.nx || j >= D.ny) return;
    using V = PVal<T>;
    // The cell across the domain face (a, s): the other end of a periodic axis, else the cell itself (-p at an
    // outflow, p = 0 on the face).  Faces that keep U*: walls and inflow (and, by the flags, cut faces).
    auto outflow = [&](int a, int s) { return D.bc[2 * a + (s > 0)] == IBM_BC_OUTFLOW; };
    auto periodic = [&](int a) { return D.bc[2 * a] == IBM_BC_PERIODIC; };
    auto kept = [&](int a, int s) { return !periodic(a) && !outflow(a, s); };
    const int oxm = i > 0 ? -1 : (periodic(0) ? D.nx - 1 : 0), oxp = i + 1 < D.nx ? 1 : (periodic(0) ? -i : 0);
    const int oym = j > 0 ? -D.sy : (periodic(1) ? (D.ny - 1) * D.sy : 0);
    const int oyp = j + 1 < D.ny ? D.sy : (periodic(1) ? -j * D.sy : 0);
    const bool edge = i == 0 || j == 0 || i == D.nx - 1 || j == D.ny - 1;
    const unsigned keep_xy = (i == 0 && kept(0, -1) ? 1u : 0u) | (j == 0 && kept(1, -1) ? 4u : 0u);
    long long P = i + (long long)D.sy * j + D.sz * k0;
    long long fx = F.index(0, i, j, k0), fy = F.index(1, i, j, k0), fz = F.index(2, i, j, k0);
    const long long sfx = (long long)F.dim[0][0] * F.dim[0][1], sfy = (long long)F.dim[1][0] * F.dim[1][1];
    // the offsets and values of one cell; `odd` of the carried values
    auto zoff = [&](int k, int s) -> long long {
        if (s < 0) return k > 0 ? -D.sz : (periodic(2) ? (long long)(D.nz - 1) * D.sz : 0);
        return k + 1 < D.nz ? D.sz : (periodic(2) ? -(long long)k * D.sz : 0);
    };
    bool odd = false, odd_c = false;
    double q = p[P];
    V pc(q, odd_c), pm(p[P + zoff(k0, -1)], odd);
    for (int k = k0; k < k1; ++k, P += D.sz, fx += sfx, fy += sfy, fz += D.sz) {
        const unsigned fl = D.flags ? (unsigned)D.flags[P] : 0u;
        const T usx = us[P], usy = us[D.N + P], usz = us[2 * D.N + P];
        const T Ux = Us[fx], Uy = Us[fy], Uz = Us[fz];
        const long long oz = zoff(k, 1);
        bool odd_z = false;
        odd = odd || odd_c;
        const double qz = p[P + oz];
        double yl = p[P + oym], yh = p[P + oyp];
        V zp(qz, odd_z);
        V xm(p[P + oxm], odd), xp(p[P + oxp], odd);
        V zm = pm;
        const V zc = zp;
        odd = odd || odd_z;
        unsigned keep = (fl & 21u) | keep_xy;
        const bool side = edge || k == 0 || k == D.nz - 1;
        if (side) {
            if (i == 0 && outflow(0, -1)) xm = pc.neg();
            if (i == D.nx - 1 && outflow(0, 1)) xp = pc.neg();
            if (j == 0 && outflow(1, -1)) yl = -q;
            if (j == D.ny - 1 && outflow(1, 1)) yh = -q;
            if (k == 0 && outflow(2, -1)) zm = pc.neg();
            if (k == D.nz - 1 && outflow(2, 1)) zp = pc.neg();
            if (k == 0 && kept(2, -1)) keep |= 16u;
        }
        // differences: lower, upper and central of each axis; a cut link reads the cell's own pressure
        T lo[3] = {pc.minus(xm), (T)(q - yl), pc.minus(zm)}, up[3] = {(T)0, (T)0, (T)0}, ce[3];
        ce[0] = xp.minus(xm);
        ce[2] = zp.minus(zm);
        if (side) {
            up[0] = xp.minus(pc);
            up[1] = (T)(yh - q);
            up[2] = zp.minus(pc);
        }
        if (fl & 4u) yl = q;
        if (fl & 8u) yh = q;
        ce[1] = (T)(yh - yl);
        if (fl & 51u) {
            if (fl & 3u) ce[0] = ((fl & 2u) ? pc : xp).minus((fl & 1u) ? pc : xm);
            if (fl & 48u) ce[2] = ((fl & 32u) ? pc : zp).minus((fl & 16u) ? pc : zm);
        }
        if (sizeof(T) == 4 && odd) {
            const long long off[2][2] = {{oxm, oxp}, {zoff(k, -1), oz}};
            const int x[2] = {i, k}, n[2] = {D.nx, D.nz};
            for (int h = 0; h < 2; ++h) {
                const int a = 2 * h;
                const double l = x[h] == 0 && outflow(a, -1) ? -q : p[P + off[h][0]];
                const double r = x[h] == n[h] - 1 && outflow(a, 1) ? -q : p[P + off[h][1]];
                lo[a] = (T)(q - l);
                up[a] = (T)(r - q);
                ce[a] = (T)(((fl >> (2 * a + 1)) & 1u ? q : r) - ((fl >> (2 * a)) & 1u ? q : l));
            }
        }
        u[P] = usx - c * ce[0];
        u[D.N + P] = usy - c * ce[1];
        u[2 * D.N + P] = usz - c * ce[2];
        U[fx] = (keep & 1u) ? Ux : Ux - dtdx * lo[0];
        U[fy] = (keep & 4u) ? Uy : Uy - dtdx * lo[1];
        U[fz] = (keep & 16u) ? Uz : Uz - dtdx * lo[2];
        if (side) {
            if (i == D.nx - 1) U[fx + 1] = kept(0, 1) ? Us[fx + 1] : Us[fx + 1] - dtdx * up[0];
            if (j == D.ny - 1) U[fy + D.nx] = kept(1, 1) ? Us[fy + D.nx] : Us[fy + D.nx] - dtdx * up[1];
            if (k == D.nz - 1) U[fz + D.sz] = kept(2, 1) ? Us[fz + D.sz] : Us[fz + D.sz] - dtdx * up[2];
        }
        pm = pc;
        pc = zc;
        q = qz;
        odd = odd_c;
        odd_c = odd_z;
    }
}

// Eq. force: Shepard average of p on each side of every triangle over the 2x2x2 block of cell
// centres around its centroid.
__global__ void k_forces(Dom D, const float* __restrict__ tri, long long ntri, const double* __restrict__ p,
                         double* partials, unsigned* counter, double* out) {
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < ntri; t += (long long)gridDim.x * blockDim.x) {
        double V[3][3];
        bool ok = true;
        for (int q = 0; q < 9; ++q) {
            V[q / 3][q % 3] = (double)tri[9 * t + q];
            ok = ok && isfinite(V[q / 3][q % 3]);
        }
        if (!ok) continue;
        double e1[3], e2[3], nrm[3], X[3];
        for (int d = 0; d < 3; ++d) {
            e1[d] = V[1][d] - V[0][d];
            e2[d] = V[2][d] - V[0][d];
            X[d] = (V[0][d] + V[1][d] + V[2][d]) / 3.0;
        }
        nrm[0] = e1[1] * e2[2] - e1[2] * e2[1];
        nrm[1] = e1[2] * e2[0] - e1[0] * e2[2];
        nrm[2] = e1[0] * e2[1] - e1[1] * e2[0];
        const double len = sqrt(nrm[0] * nrm[0] + nrm[1] * nrm[1] + nrm[2] * nrm[2]);
        if (!(len > 0.0)) continue;
        const double area = 0.5 * len * D.dx * D.dx;
        for (int d = 0; d < 3; ++d) nrm[d] /= len;
        long long base[3];
        for (int d = 0; d < 3; ++d) base[d] = (long long)floor(X[d] - 0.5);
        double sw[2] = {0.0, 0.0}, sp[2] = {0.0, 0.0};
        const long long n[3] = {D.nx, D.ny, D.nz};
        for (int dk = 0; dk < 2; ++dk)
            for (int dj = 0; dj < 2; ++dj)
                for (int di = 0; di < 2; ++di) {
                    const long long x[3] = {base[0] + di, base[1] + dj, base[2] + dk};
                    if (x[0] < 0 || x[1] < 0 || x[2] < 0 || x[0] >= n[0] || x[1] >= n[1] || x[2] >= n[2]) continue;
                    double r2 = 0.0, sd = 0.0;
                    for (int d = 0; d < 3; ++d) {
                        const double r = ((double)x[d] + 0.5) - X[d];
                        r2 += r * r;
                        sd += nrm[d] * r;
                    }
                    if (sd == 0.0) continue;
                    if (r2 < 1e-24) r2 = 1e-24;
                    const double w = 1.0 / r2;
                    const int side = sd > 0.0 ? 0 : 1;
                    sw[side] += w;
                    sp[side] += w * p[x[0] + (long long)D.sy * x[1] + D.sz * x[2]];
                }
        if (sw[0] == 0.0 || sw[1] == 0.0) continue;
        const double pf = sp[0] / sw[0], pb = sp[1] / sw[1];
        for (int d = 0; d < 3; ++d) acc[d] += area * (pb - pf) * nrm[d];
        acc[3] += 1.0;
    }
    grid_reduce<4>(acc, partials, counter, [&](double* t) {
        for (int q = 0; q < 4; ++q) out[q] = t[q];
    });
}

// Viscous force on the body: the molecular diffusive flux nu (u_P - u_G) dx through every cut link,
// u_G the Eq. q_axis ghost value the momentum equation uses there.  One thread per link record.
template <class T>
__global__ void k_viscous_force(Dom D, const T* __restrict__ u, double nu, double* partials, unsigned* counter,
                                double* out) {
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const long long nrec = D.flags ? (long long)D.nrec : 0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nrec; q += (long long)gridDim.x * blockDim.x) {
        const LinkRec& R = D.rec[q];
        const long long P = R.cell;
        const int a = R.axis, sd = R.side;
        const int xa = a == 0 ? (int)(P % D.nx) : (a == 1 ? (int)((P / D.nx) % D.ny) : (int)(P / D.sz));
        const unsigned fl = D.flags[P];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double uG = (double)vel_across(D, u, c, P, xa, fl, a, sd);
            acc[c] += nu * ((double)u[c * D.N + P] - uG) * D.dx;
        }
        acc[3] += 1.0;
    }
    grid_reduce<4>(acc, partials, counter, [&](double* t) {
        for (int q = 0; q < 4; ++q) out[q] = t[q];
    });
}

unsigned lin_blocks(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    long long cap = 16LL * IBM_NSM;
    if (b > cap) b = cap;
    return (unsigned)(b < 1 ? 1 : b);
}


// ---- Crank-Nicolson predictor (Eq. crank-nicolson) -----------------------------------------------
// delta = u* - u^n solves M delta = delta - (dt/2) L_0(delta) = dt L(u^n) over the stacked three
// components; BiCGStab from delta = 0, scalars on the device (the same recurrences as the pressure
// BiCGStab).  Cell kernels loop over a capped grid; per-thread sums run in the working precision and
// the block and grid sums in FP64.

// The fast kernel of a pair leaves its sums in sc->part; the general kernel, launched after it, adds
// its own and finishes (so the totals are formed in a fixed order).
template <class T, bool GENERAL>
__global__ void __launch_bounds__((FluxOcc<T, GENERAL>::threads), (FluxOcc<T, GENERAL>::value)) k_cn_begin(Dom D, FaceLayout F, const T* __restrict__ u, const T* __restrict__ U,
                                                  const T* __restrict__ nut, T* __restrict__ H, T* __restrict__ r,
                                                  T* __restrict__ rh, T* __restrict__ x, T nu, T gam, T dt, double tol2,
                                                  int maxit, int keepx, SolveScal* sc, double* partials, unsigned* counter,
                                                  const int32_t* __restrict__ list, long long nlist) {
    T a0 = 0;
    flux_cells<GENERAL, T>(D, F, u, U, nut, nu, gam, list, nlist, (const T*)nullptr,
                           [&](long long q, Off<T> o, T h, T, T) {
        const T b = dt * h;
        to_off(H + q, o, h);
        to_off(r + q, o, b);
        to_off(rh + q, o, b);
        if (!keepx) to_off(x + q, o, (T)0);
        a0 += b * b;
    });
    T acc[1] = {a0};
    grid_reduce<1>(acc, partials, counter, [&](double* t) {
        if (!GENERAL) {
            sc->part[0] = t[0];
            return;
        }
        const double bb = t[0] + sc->part[0];
        sc->bb = bb;
        sc->rr = bb;
        sc->rho = bb;
        sc->rho_old = 1.0;
        sc->alpha = 1.0;
        sc->omega = 1.0;
        sc->target2 = tol2 * bb;
        sc->iters = 0;
        sc->maxit = maxit;
        sc->restart = 1;
        sc->nonfinite = isfinite(bb) ? 0 : 1;
        sc->done = (bb == 0.0 || !isfinite(bb)) ? 1 : 0;
    });
}

// p = r (first iteration) or r + beta (p - omega v)
template <class T>
__global__ void k_cn_p(long long n, const T* __restrict__ r, T* __restrict__ p, const T* __restrict__ v,
                       const SolveScal* sc) {
    if (sc->done) return;
    const bool rs = sc->restart != 0;
    const T beta = rs ? (T)0 : (T)((sc->rho / sc->rho_old) * (sc->alpha / sc->omega));
    const T om = rs ? (T)0 : (T)sc->omega;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        p[q] = rs ? r[q] : r[q] + beta * (p[q] - om * v[q]);
}

// y = M xin = xin - (dt/2) L_0(xin).  mode 0: (w, y) -> alpha = rho / (r_hat, v).  mode 1 (xin = s):
// (y, s), (y, y) -> omega.  mode 2 (warm start, xin = the previous increment): r = b - M xin with b
// read from and r written to r2, r_hat = r in y, (r, r) -> rr = rho.
template <class T, bool GENERAL, int mode>
__global__ void __launch_bounds__((FluxOcc<T, GENERAL>::threads), (FluxOcc<T, GENERAL>::value)) k_cn_apply(Dom D, FaceLayout F, const T* __restrict__ xin,
                                                  const T* __restrict__ U, const T* __restrict__ nut,
                                                  T* __restrict__ y, const T* __restrict__ w, T* r2, T nu, T gam,
                                                  T hdt, SolveScal* sc, double* partials,
                                                  unsigned* counter, const int32_t* __restrict__ list, long long nlist) {
    if (sc->done) return;
    T a0 = 0, a1 = 0;
    flux_cells<GENERAL, T>(D, F, xin, U, nut, nu, gam, list, nlist, mode == 0 ? w : (mode == 2 ? (const T*)r2 : nullptr),
                           [&](long long q, Off<T> o, T h, T xv, T wq) {
        const T yv = xv - hdt * h;
        if (mode == 2) {
            const T rn = wq - yv;
            to_off(r2 + q, o, rn);
            to_off(y + q, o, rn);
            a0 += rn * rn;
            return;
        }
        to_off(y + q, o, yv);
        if (mode == 0) {
            a0 += wq * yv;
        } else {
            a0 += yv * xv;
            a1 += yv * yv;
        }
    });
    T acc[2] = {a0, a1};
    grid_reduce<2>(acc, partials, counter, [&](double* t) {
        if (!GENERAL) {
            sc->part[0] = t[0];
            sc->part[1] = t[1];
            return;
        }
        const double t0 = t[0] + sc->part[0], t1 = t[1] + sc->part[1];
        if (mode == 2) {
            sc->rr = t0;
            sc->rho = t0;
            if (!isfinite(t0)) sc->nonfinite = 1;
            if (!isfinite(t0) || t0 <= sc->target2) sc->done = 1;
            return;
        }
        if (mode == 0) {
            sc->rv = t0;
            sc->alpha = t0 != 0.0 ? sc->rho / t0 : 0.0;
            if (t0 == 0.0 || !isfinite(t0)) {
                if (!isfinite(t0)) sc->nonfinite = 1;
                sc->done = 1;                                        // breakdown
            }
        } else {
            sc->ts = t0;
            sc->tt = t1;
            sc->omega = t1 > 0.0 ? t0 / t1 : 0.0;
        }
    });
}

// s = r - alpha v
template <class T>
__global__ void k_cn_s(long long n, const T* __restrict__ r, const T* __restrict__ v, T* __restrict__ sv,
                       const SolveScal* sc) {
    if (sc->done) return;
    const T alpha = (T)sc->alpha;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        sv[q] = r[q] - alpha * v[q];
}

// x += alpha p + omega s, r = s - omega t; (r_hat, r), (r, r); convergence test.
template <class T>
__global__ void __launch_bounds__(256) k_cn_xr(long long n, const T* __restrict__ p, const T* __restrict__ sv,
                                               const T* __restrict__ tv, const T* __restrict__ rh, T* __restrict__ x,
                                               T* __restrict__ r, SolveScal* sc, double* partials, unsigned* counter) {
    if (sc->done) return;
    const T alpha = (T)sc->alpha, om = (T)sc->omega;
    T a0 = 0, a1 = 0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        x[q] = x[q] + alpha * p[q] + om * sv[q];
        const T rv = sv[q] - om * tv[q];
        r[q] = rv;
        a0 += rh[q] * rv;
        a1 += rv * rv;
    }
    T acc[2] = {a0, a1};
    grid_reduce<2>(acc, partials, counter, [&](double* t) {
        sc->rho_old = sc->rho;
        sc->rho = t[0];
        sc->rr_old = sc->rr;
        sc->rr = t[1];
        sc->restart = 0;
        sc->iters += 1;
        if (!isfinite(t[1])) {
            sc->nonfinite = 1;
            sc->done = 1;
        } else if (t[1] <= sc->target2 || sc->iters >= sc->maxit || sc->omega == 0.0 || t[0] == 0.0) {
            sc->done = 1;
        }
    });
}

template <class T>
__global__ void k_cn_finish(long long n, const T* __restrict__ u, const T* __restrict__ x, T* __restrict__ ustar) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        ustar[q] = u[q] + x[q];
}

// Persistent launch of the tiled flux kernels: as many blocks as fit on the GPU at once (measured
// for the heaviest of them at set-up), each walking tiles until none is left.
int g_tile_blocks[2] = {2 * IBM_NSM, 2 * IBM_NSM};   // FP32, FP64

template <class T>
dim3 tile_grid(const LesCtx& c) {
    const long long items = (long long)((c.D.nx + FT_X - 1) / FT_X) * ((c.D.ny + FT_Y - 1) / FT_Y) *
                            ((c.D.nz + c.D.tile_z - 1) / c.D.tile_z);
    const long long cap = g_tile_blocks[sizeof(T) == 8];
    return dim3((unsigned)(items < cap ? items : cap));
}

// Planes per tile of the march: the fewest plane steps over all rounds of the persistent blocks (a tile of
// k planes takes about k + 4: five are staged before its first).
template <class T>
int tile_planes(const Dom& D) {
    const long long xy = (long long)((D.nx + FT_X - 1) / FT_X) * ((D.ny + FT_Y - 1) / FT_Y);
    const long long cap = g_tile_blocks[sizeof(T) == 8];
    long long best = -1;
    int best_k = D.nz;
    for (int ch = 1; ch <= D.nz; ++ch) {
        const int k = (D.nz + ch - 1) / ch;
        if ((k < 4 || k > 64) && ch > 1 && best >= 0) { if (k < 4) break; else continue; }
        const long long cost = ((xy * ((D.nz + k - 1) / k) + cap - 1) / cap) * (k + 4);
        if (best < 0 || cost < best || best_k > 64) {
            best = cost;
            best_k = k;
        }
    }
    return best_k;
}

// Blocks of the general-cell kernels: those that fit on the GPU at once, fewer for a short list.
template <class T>
unsigned general_blocks(long long n) {
    const long long b = (n + FG_CELLS - 1) / FG_CELLS, cap = (long long)FluxOcc<T, true>::value * IBM_NSM;
    return (unsigned)(b > cap ? cap : (b < 1 ? 1 : b));
}

template <class T>
int predict_cn_t(const LesCtx& c, const T* u, const T* U, const T* nut, T* H, T* ustar, int* iters, cudaStream_t s) {
    CNWork& w = *c.cn;
    Dom Dh = c.D;
    Dh.hom = 1;
    const long long n3 = 3 * c.D.N;
    const unsigned nbv = lin_blocks(n3, 256);
    T *r = (T*)w.r, *rh = (T*)w.rh, *p = (T*)w.p, *v = (T*)w.v, *sv = (T*)w.sv, *tv = (T*)w.tv, *x = (T*)w.x;
    const T nu = (T)c.nu, gam = (T)c.quick, dt = (T)c.dt, hdt = (T)(0.5 * c.dt);
    const unsigned ngen = general_blocks<T>(c.n_general);
    prof_begin(c.prof, PS_PREDICT, s);
    // warm start from the previous step's increment (the increment changes slowly from step to step)
    const int keepx = w.have_x;
    k_cn_begin<T, false><<<tile_grid<T>(c), dim3(FT_X, FT_Y), fast_tile_smem<T>(), s>>>(c.D, c.F, u, U, nut, H, r, rh, x, nu, gam, dt, w.tol * w.tol,
                                                        w.maxit, keepx, w.sc, c.partials, c.counter, nullptr, 0);
    k_cn_begin<T, true><<<ngen, FG_NT, 0, s>>>(c.D, c.F, u, U, nut, H, r, rh, x, nu, gam, dt, w.tol * w.tol, w.maxit,
                                             keepx, w.sc, c.partials, c.counter, c.general, c.n_general);
    prof_end(c.prof, PS_PREDICT, s);
    IBM_LAUNCHED("k_cn_begin");
    IBM_COUNT(c, 2);
    auto apply = [&](const T* in, T* out, auto m) {
        constexpr int mode = decltype(m)::value;
        const T* wv = mode == 2 ? nullptr : rh;
        T* r2 = mode == 2 ? r : nullptr;
        k_cn_apply<T, false, mode><<<tile_grid<T>(c), dim3(FT_X, FT_Y), fast_tile_smem<T>(), s>>>(
            Dh, c.F, in, U, nut, out, wv, r2, nu, gam, hdt, w.sc, c.partials, c.counter, nullptr, 0);
        k_cn_apply<T, true, mode><<<ngen, FG_NT, 0, s>>>(Dh, c.F, in, U, nut, out, wv, r2, nu, gam, hdt, w.sc, c.partials,
                                                       c.counter, c.general, c.n_general);
    };
    if (keepx) {
        apply(x, rh, std::integral_constant<int, 2>{});
        IBM_COUNT(c, 2);
    }
    for (;;) {
        prof_begin(c.prof, PS_MOMENTUM, s);
        for (int it = 0; it < 4; ++it) {
            k_cn_p<T><<<nbv, 256, 0, s>>>(n3, r, p, v, w.sc);
            apply(p, v, std::integral_constant<int, 0>{});
            k_cn_s<T><<<nbv, 256, 0, s>>>(n3, r, v, sv, w.sc);
            apply(sv, tv, std::integral_constant<int, 1>{});
            k_cn_xr<T><<<nbv, 256, 0, s>>>(n3, p, sv, tv, rh, x, r, w.sc, c.partials, c.counter);
        }
        prof_end(c.prof, PS_MOMENTUM, s);
        IBM_LAUNCHED("crank-nicolson bicgstab");
        IBM_COUNT(c, 28);
        IBM_CUDA(cudaMemcpyAsync(w.hsc, w.sc, sizeof(SolveScal), cudaMemcpyDeviceToHost, s));
        IBM_CUDA(cudaStreamSynchronize(s));
        if (w.hsc->done) break;
    }
    k_cn_finish<T><<<nbv, 256, 0, s>>>(n3, u, x, ustar);
    IBM_LAUNCHED("k_cn_finish");
    IBM_COUNT(c, 1);
    if (iters) *iters = w.hsc->iters;
    w.have_x = !w.hsc->nonfinite && w.hsc->rr <= w.hsc->target2;
    if (w.hsc->nonfinite) return ibm_fail(IBM_E_NONFINITE, "crank-nicolson momentum solve: non-finite residual");
    if (!(w.hsc->rr <= w.hsc->target2))
        return ibm_fail(IBM_E_NOCONV, "crank-nicolson momentum solve: relative residual %.3e after %d iterations",
                        sqrt(w.hsc->rr / (w.hsc->bb > 0 ? w.hsc->bb : 1.0)), w.hsc->iters);
    return IBM_OK;
}

}  // namespace

namespace {
// Order-preserving compaction of the general cells: one block per (y, z) row, ballots over x.
__global__ void k_list_general(Dom D, const unsigned long long* __restrict__ row_off,
                               int32_t* __restrict__ list) {
    const int j = blockIdx.x, k = blockIdx.y;
    __shared__ int base;
    if (threadIdx.x == 0) base = 0;
    __syncthreads();
    const long long row = j + (long long)D.ny * k;
    for (int i0 = 0; i0 < D.nx; i0 += 32) {
        const int i = i0 + threadIdx.x;
        const long long P = i + (long long)D.sy * j + D.sz * k;
        const bool g = i < D.nx && !fast_cell(D, P, i, j, k);
        const unsigned m = __ballot_sync(0xffffffffu, g);
        if (g) list[row_off[row] + base + __popc(m & ((1u << threadIdx.x) - 1u))] = (int32_t)P;
        __syncwarp();
        if (threadIdx.x == 0) base += __popc(m);
        __syncwarp();
    }
}

__global__ void k_row_counts(Dom D, unsigned long long* __restrict__ rc, uint8_t* __restrict__ fast) {
    const int j = blockIdx.x, k = blockIdx.y;
    unsigned n = 0;
    for (int i = threadIdx.x; i < D.nx; i += 32) {
        const long long P = i + (long long)D.sy * j + D.sz * k;
        const bool f = fast_cell(D, P, i, j, k);
        fast[P] = f ? 1 : 0;
        n += !f;
    }
    for (int o = 16; o > 0; o >>= 1) n += __shfl_down_sync(0xffffffffu, n, o);
    if (threadIdx.x == 0) rc[j + (long long)D.ny * k] = n;
}
}  // namespace

int flux_kernels_setup() {
    // the tiles need more than the default 48 KB of dynamic shared memory
    const int bytes = (int)fast_tile_smem<double>(), bytesf = (int)fast_tile_smem<float>();
    IBM_CUDA(cudaFuncSetAttribute(k_predict<false, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    IBM_CUDA(cudaFuncSetAttribute(k_cn_begin<double, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    IBM_CUDA(cudaFuncSetAttribute(k_cn_apply<double, false, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    IBM_CUDA(cudaFuncSetAttribute(k_cn_apply<double, false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    IBM_CUDA(cudaFuncSetAttribute(k_cn_apply<double, false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    IBM_CUDA(cudaFuncSetAttribute(k_predict<false, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytesf));
    IBM_CUDA(cudaFuncSetAttribute(k_cn_begin<float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytesf));
    IBM_CUDA(cudaFuncSetAttribute(k_cn_apply<float, false, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytesf));
    IBM_CUDA(cudaFuncSetAttribute(k_cn_apply<float, false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytesf));
    IBM_CUDA(cudaFuncSetAttribute(k_cn_apply<float, false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytesf));
    int dev = 0, nsm = IBM_NSM, bf = 0, bd = 0;
    IBM_CUDA(cudaGetDevice(&dev));
    IBM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    IBM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bf, k_cn_apply<float, false, 0>, FT_NT,
                                                           fast_tile_smem<float>()));
    IBM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bd, k_cn_apply<double, false, 0>, FT_NT,
                                                           fast_tile_smem<double>()));
    g_tile_blocks[0] = (bf > 0 ? bf : 1) * nsm;
    g_tile_blocks[1] = (bd > 0 ? bd : 1) * nsm;
    return IBM_OK;
}

int build_general_list(LesCtx& c, cudaStream_t s) {
    const long long nrows = (long long)c.D.ny * c.D.nz;
    unsigned long long* rc = nullptr;
    IBM_CUDA(ibm_malloc(&rc, (size_t)(nrows + 1) * sizeof(unsigned long long)));
    dim3 rows((unsigned)c.D.ny, (unsigned)c.D.nz);
    cudaError_t e0 = ibm_malloc(&c.fastmask, (size_t)c.D.N);
    if (e0 != cudaSuccess) {
        cudaFree(rc);
        return ibm_fail(IBM_E_NOMEM, "momentum flux: fast-cell mask (%lld bytes)", (long long)c.D.N);
    }
    k_row_counts<<<rows, 32, 0, s>>>(c.D, rc, c.fastmask);
    k_scan_tile_totals<<<1, IBM_SCAN_NT, 0, s>>>((long long*)rc, nrows, (long long*)rc + nrows);
    unsigned long long total = 0;
    cudaError_t e = cudaMemcpyAsync(&total, rc + nrows, sizeof(total), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = ibm_malloc(&c.general, (size_t)(total > 0 ? total : 1) * sizeof(int32_t));
    if (e == cudaSuccess && total > 0) {
        k_list_general<<<rows, 32, 0, s>>>(c.D, rc, c.general);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(rc);
    if (e != cudaSuccess) return ibm_cuda_check(e, "momentum flux: general-cell list");
    c.n_general = (long long)total;
    c.D.fast = c.fastmask;
    c.D.tile_z = c.prec == IBM_FP64 ? tile_planes<double>(c.D) : tile_planes<float>(c.D);
    return IBM_OK;
}

int launch_csm(const LesCtx& c, const void* u, void* nut, cudaStream_t s) {
    int kz = 1;
    const dim3 g = column_grid(c.D, kz, 24LL * IBM_NSM);        // four rounds of six blocks per SM
    if (c.prec == IBM_FP64) k_csm<double><<<g, c.cg.block, 0, s>>>(c.D, (const double*)u, (double*)nut, kz);
    else k_csm<float><<<g, c.cg.block, 0, s>>>(c.D, (const float*)u, (float*)nut, kz);
    IBM_LAUNCHED("k_csm");
    IBM_COUNT(c, 1);
    return IBM_OK;
}

template <class T>
static void predict_t(const LesCtx& c, const T* u, const T* U, const T* nut, const T* Hprev, T* H, T* ustar, int first,
                      cudaStream_t s) {
    k_predict<false, T><<<tile_grid<T>(c), dim3(FT_X, FT_Y), fast_tile_smem<T>(), s>>>(c.D, c.F, u, U, nut, Hprev, H, ustar, (T)c.nu, (T)c.dt, first,
                                                       (T)c.quick, nullptr, 0);
    if (c.n_general > 0)
        k_predict<true, T><<<general_blocks<T>(c.n_general), FG_NT, 0, s>>>(c.D, c.F, u, U, nut, Hprev, H, ustar,
                                                                         (T)c.nu, (T)c.dt, first, (T)c.quick,
                                                                         c.general, c.n_general);
}

int launch_predict(const LesCtx& c, const void* u, const void* U, const void* nut, const void* Hprev, void* H,
                   void* ustar, int first, cudaStream_t s) {
    if (c.prec == IBM_FP64)
        predict_t<double>(c, (const double*)u, (const double*)U, (const double*)nut, (const double*)Hprev, (double*)H,
                          (double*)ustar, first, s);
    else
        predict_t<float>(c, (const float*)u, (const float*)U, (const float*)nut, (const float*)Hprev, (float*)H,
                         (float*)ustar, first, s);
    IBM_LAUNCHED("k_predict");
    IBM_COUNT(c, c.n_general > 0 ? 2 : 1);
    return IBM_OK;
}

int launch_predict_cn(const LesCtx& c, const void* u, const void* U, const void* nut, void* H, void* ustar,
                      int* iters, cudaStream_t s) {
    if (!c.cn) return ibm_fail(IBM_E_INVALID, "crank-nicolson predictor: state created without integrator = 1");
    if (c.prec == IBM_FP64)
        return predict_cn_t<double>(c, (const double*)u, (const double*)U, (const double*)nut, (double*)H,
                                    (double*)ustar, iters, s);
    return predict_cn_t<float>(c, (const float*)u, (const float*)U, (const float*)nut, (float*)H, (float*)ustar,
                               iters, s);
}

int launch_forcing(const LesCtx& c, void* ustar, cudaStream_t s) {
    if (c.n_inc == 0 || !c.D.flags) {
        IBM_CUDA(cudaMemsetAsync(c.fscal, 0, 3 * sizeof(double), s));
        return IBM_OK;
    }
    const unsigned nb = lin_blocks(c.n_inc, 256);
    const double vol = c.D.dx * c.D.dx * c.D.dx;
    if (c.prec == IBM_FP64) {
        k_forcing_gather<double><<<nb, 256, 0, s>>>(c.D, c.inc, c.n_inc, (const double*)ustar, c.fdelta, c.dt,
                                                    c.deadend_on, vol, c.partials, c.counter, c.fscal);
        k_forcing_apply<double><<<nb, 256, 0, s>>>(c.D, c.inc, c.n_inc, c.fdelta, (double*)ustar);
    } else {
        k_forcing_gather<float><<<nb, 256, 0, s>>>(c.D, c.inc, c.n_inc, (const float*)ustar, c.fdelta, (float)c.dt,
                                                   c.deadend_on, vol, c.partials, c.counter, c.fscal);
        k_forcing_apply<float><<<nb, 256, 0, s>>>(c.D, c.inc, c.n_inc, c.fdelta, (float*)ustar);
    }
    IBM_LAUNCHED("k_forcing");
    IBM_COUNT(c, 2);
    return IBM_OK;
}

template <class T>
static void faces_t(const LesCtx& c, const T* us, T* Us, cudaStream_t s) {
    int kz = 1;
    const dim3 g = column_grid(c.D, kz);
    k_faces<T><<<g, c.cg.block, 0, s>>>(c.D, c.F, us, Us, kz);
    k_boundary_flux<T><<<64, 256, 0, s>>>(c.D, c.F, Us, c.partials, c.counter, c.fscal);
    k_outflow_shift<T><<<64, 256, 0, s>>>(c.D, c.F, Us, c.fscal);
}

int launch_faces(const LesCtx& c, const void* ustar, void* Ustar, cudaStream_t s) {
    if (c.prec == IBM_FP64) faces_t<double>(c, (const double*)ustar, (double*)Ustar, s);
    else faces_t<float>(c, (const float*)ustar, (float*)Ustar, s);
    IBM_LAUNCHED("k_faces");
    IBM_COUNT(c, 3);
    return IBM_OK;
}

int launch_rhs(const LesCtx& c, const void* Ustar, double* b, cudaStream_t s) {
    const double inv = 1.0 / (c.D.dx * c.dt);
    int kz = 1;
    const dim3 g = column_grid(c.D, kz);
    if (c.prec == IBM_FP64) k_rhs<double><<<g, c.cg.block, 0, s>>>(c.D, c.F, (const double*)Ustar, b, inv, kz);
    else k_rhs<float><<<g, c.cg.block, 0, s>>>(c.D, c.F, (const float*)Ustar, b, inv, kz);
    IBM_LAUNCHED("k_rhs");
    IBM_COUNT(c, 1);
    return IBM_OK;
}

template <class T>
static void correct_t(const LesCtx& c, const T* us, const T* Us, const double* p, T* u, T* U, cudaStream_t s) {
    int kz = 1;
    const dim3 g = column_grid(c.D, kz);
    k_correct<T><<<g, c.cg.block, 0, s>>>(c.D, c.F, us, Us, p, u, U, (T)(c.dt / (2.0 * c.D.dx)), (T)(c.dt / c.D.dx), kz);
}

int launch_correct(const LesCtx& c, const void* ustar, const void* Ustar, const double* p, void* u, void* U,
                   cudaStream_t s) {
    if (c.prec == IBM_FP64)
        correct_t<double>(c, (const double*)ustar, (const double*)Ustar, p, (double*)u, (double*)U, s);
    else
        correct_t<float>(c, (const float*)ustar, (const float*)Ustar, p, (float*)u, (float*)U, s);
    IBM_LAUNCHED("k_correct");
    IBM_COUNT(c, 1);
    return IBM_OK;
}

int launch_forces(const LesCtx& c, const float* tri, long long ntri, const double* p, double* d_out4, cudaStream_t s) {
    k_forces<<<lin_blocks(ntri, 128), 128, 0, s>>>(c.D, tri, ntri, p, c.partials, c.counter, d_out4);
    IBM_LAUNCHED("k_forces");
    IBM_COUNT(c, 1);
    return IBM_OK;
}

int launch_viscous_force(const LesCtx& c, const void* u, double* d_out4, cudaStream_t s) {
    const unsigned nb = lin_blocks(c.n_rec > 0 ? c.n_rec : 1, 256);
    if (c.prec == IBM_FP64)
        k_viscous_force<double><<<nb, 256, 0, s>>>(c.D, (const double*)u, c.nu, c.partials, c.counter, d_out4);
    else
        k_viscous_force<float><<<nb, 256, 0, s>>>(c.D, (const float*)u, c.nu, c.partials, c.counter, d_out4);
    IBM_LAUNCHED("k_viscous_force");
    IBM_COUNT(c, 1);
    return IBM_OK;
}
