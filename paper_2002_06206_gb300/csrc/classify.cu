// classify.cu -- per-geometry kernels: exact axis-aligned ray/triangle classification (Sec. 2.4.1)
// and the setup of the link records (Sec. 2.4.1-2.4.2).
//
// Every floating-point operation of the predicate and of the record coefficients is written with an
// explicit IEEE round-to-nearest intrinsic (no FMA contraction), so the result is reproducible bit
// for bit by any FP64 implementation that evaluates the same expressions in the same order.
#include <stdlib.h>

#include <mutex>

#include "scan.cuh"

namespace {

// Candidate lines of a triangle: its projected bounding box widened by this margin (grid units).
// The edge tolerance admits points at most eps_edge * (triangle height) outside the triangle.
constexpr double kLineMargin = 1e-4;
constexpr unsigned long long kEmpty = 0xffffffffffffffffULL;

struct Tri { double v[3][3]; };

__device__ __forceinline__ long long clamp_line(double v, long long n) {
    if (!(v > -1.0)) return -1;
    if (v > (double)n) return n;
    return (long long)v;
}

// [lo, hi] of line indices j with j + 1/2 in [mn - margin, mx + margin], clamped to [0, n-1].
__device__ __forceinline__ void line_range(double mn, double mx, long long n, long long& lo, long long& hi) {
    double l = ceil(__dsub_rn(__dsub_rn(mn, kLineMargin), 0.5));
    double h = floor(__dsub_rn(__dadd_rn(mx, kLineMargin), 0.5));
    lo = l < 0.0 ? 0 : clamp_line(l, n);
    hi = clamp_line(h, n);
    if (hi > n - 1) hi = n - 1;
}

// Twice the signed area of (P, Q, q) in the (b, c) projection.
__device__ __forceinline__ double orient(double Pb, double Pc, double Qb, double Qc, double qb, double qc) {
    double l = __dmul_rn(__dsub_rn(Qb, Pb), __dsub_rn(qc, Pc));
    double r = __dmul_rn(__dsub_rn(Qc, Pc), __dsub_rn(qb, Pb));
    return __dsub_rn(l, r);
}

// The grid line through (qb, qc) parallel to axis a crosses the triangle iff its barycentric weights
// (w0, w1, w2)/W in the projection are all >= -eps_edge; W = 0 (|W| <= eps_det) is the parallel case
// that Moller-Trumbore's determinant test rejects.
__device__ __forceinline__ bool line_hit(const Tri& T, int a, double qb, double qc, double eps_edge,
                                         double eps_det, double& x_hit) {
    const int b = (a + 1) % 3, c = (a + 2) % 3;
    const double* A = T.v[0];
    const double* B = T.v[1];
    const double* C = T.v[2];
    double w0 = orient(B[b], B[c], C[b], C[c], qb, qc);
    double w1 = orient(C[b], C[c], A[b], A[c], qb, qc);
    double w2 = orient(A[b], A[c], B[b], B[c], qb, qc);
    double W = __dadd_rn(__dadd_rn(w0, w1), w2);
    if (!(fabs(W) > eps_det)) return false;
    double thr = __dmul_rn(eps_edge, fabs(W));
    double s0 = W > 0 ? w0 : -w0, s1 = W > 0 ? w1 : -w1, s2 = W > 0 ? w2 : -w2;
    if (!(s0 >= -thr && s1 >= -thr && s2 >= -thr)) return false;
    double num = __dadd_rn(__dadd_rn(__dmul_rn(w0, A[a]), __dmul_rn(w1, B[a])), __dmul_rn(w2, C[a]));
    x_hit = __ddiv_rn(num, W);
    return true;
}

// One hit of a grid line parallel to axis a: the interior face it belongs to and its position t on it.  The
// triangle's coordinates come in the order a, a + 1, a + 2.
__device__ __forceinline__ bool face_hit(const Tri& T, int a, int jb, int jc, const int n[3], double eps_edge, double eps_det,
                                         long long& fid, unsigned long long& bits) {
    double xh;
    if (!line_hit(T, 0, (double)jb + 0.5, (double)jc + 0.5, eps_edge, eps_det, xh)) return false;
    const double xm = __dsub_rn(xh, 0.5);
    const double f = floor(xm);
    const int na = a == 0 ? n[0] : (a == 1 ? n[1] : n[2]);
    if (!(f >= 0.0 && f <= (double)(na - 2))) return false;
    const double t = __dsub_rn(xm, f);
    const int xa = (int)f;
    const int x = a == 0 ? xa : (a == 1 ? jc : jb), y = a == 0 ? jb : (a == 1 ? xa : jc), z = a == 0 ? jc : (a == 1 ? jb : xa);
    fid = a * ((long long)n[0] * n[1] * n[2]) + x + n[0] * (y + (long long)n[1] * z);
    bits = (unsigned long long)__double_as_longlong(t);
    return true;
}

// FP32 test of the same line that only ever says "certainly outside": two of the barycentric weights differ
// in sign by more than the FP32 error (every difference and product is good to a few 2^-24 of the absolute
// products) and the edge tolerance, so the FP64 predicate rejects the line whatever the sign of their sum.  It needs
// the line's coordinates j + 1/2 exact in FP32: on grids of more than 2^23 cells along an axis every line goes to
// the FP64 predicate (TestArgs::fp32).  eps >= 0: a negative tolerance (a triangle shrunk by it) counts as 0 here,
// which rejects less.
__device__ __forceinline__ bool surely_outside(float Ab, float Ac, float Bb, float Bc, float Cb, float Cc, float qb, float qc,
                                               float eps) {
    const float ab = qb - Ab, ac = qc - Ac, bb = qb - Bb, bc = qc - Bc, cb = qb - Cb, cc = qc - Cc;
    float hi = -1.f, lo = 1.f, sum = 0.f, w[3], e[3];
    const float P[3] = {(Cb - Bb) * bc, (Ab - Cb) * cc, (Bb - Ab) * ac}, Q[3] = {(Cc - Bc) * bb, (Ac - Cc) * cb, (Bc - Ac) * ab};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        w[i] = P[i] - Q[i];
        e[i] = 1e-6f * (fabsf(P[i]) + fabsf(Q[i]));      // 16 * 2^-24
        sum += fabsf(w[i]) + e[i];
    }
    const float thr = eps * sum;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        hi = fmaxf(hi, w[i] > e[i] + thr ? 1.f : -1.f);
        lo = fminf(lo, w[i] < -(e[i] + thr) ? -1.f : 1.f);
    }
    return hi > 0.f && lo < 0.f;
}

// Hits found by the marking pass, kept where the soup's size leaves room (else they are found again).
struct HitList {
    unsigned long long* t;
    unsigned* fid;                 // face ids stay below 2^32 (grids of at most 2^31/3 cells)
    long long cap;
    unsigned long long* count;
};

struct TestArgs {
    const float* tri;
    long long ntri;
    int n[3];
    double eps_edge, eps_det;
    int fp32;                      // surely_outside may be asked
    uint8_t* flags;
    unsigned long long *tmin, *tmax, *tests;
    HitList hits;
};

__device__ __forceinline__ void or_byte(uint8_t* p, unsigned bit) {
    // the aligned word around a byte lies in the same allocation; its other bytes are or-ed with 0
    const uintptr_t q = (uintptr_t)p;
    atomicOr(reinterpret_cast<unsigned*>(q & ~(uintptr_t)3), bit << (8 * (q & 3)));
}

// The marking pass (PASS 1) sets the two link bits of every hit face and gives its min/max slot its start
// values (every writer stores the same); the second forms the min/max of t through 64-bit integer atomics on
// the bit patterns of t >= 0 (their order is the order of the values), so nothing depends on the order of the
// threads, and faces without a hit cost nothing.
template <int PASS>
__device__ __forceinline__ void use_hit(const TestArgs& A, long long fid, unsigned long long bits) {
    if (PASS == 1) {
        const long long N = (long long)A.n[0] * A.n[1] * A.n[2];
        const int a = fid >= 2 * N ? 2 : (fid >= N ? 1 : 0);
        const long long c = fid - a * N, st = a == 0 ? 1 : (a == 1 ? (long long)A.n[0] : (long long)A.n[0] * A.n[1]);
        or_byte(A.flags + c, 2u << (2 * a));
        or_byte(A.flags + c + st, 1u << (2 * a));
        A.tmin[fid] = kEmpty;
        A.tmax[fid] = 0ULL;
    } else {
        atomicMin(&A.tmin[fid], bits);
        atomicMax(&A.tmax[fid], bits);
    }
}

// Every (triangle, axis, grid line) test whose line lies in the triangle's widened projected box.  A warp takes
// 32 triangles, lays the tests of one axis end to end (a warp scan of the line counts) and gives each lane
// one test, the owner found by a search over the scan: a soup of small triangles needs no list of tests in
// memory and no idle lanes.  Tests that FP32 cannot rule out wait in a queue of the warp until 32 lanes can
// take the FP64 predicate together: the pass is bound by its FP64 instructions (about 80 with the
// conversions and the division).  An item of more than kBigItem tests goes to the whole block; gridDim.y
// slices share such items when the soup has few triangles.
// Vehicle assembly (2.03 M triangles, 6.0 M tests): 1.01 ms, 2.4 ms without the FP32 test and the queue.
constexpr int kBigItem = 1024;

template <int PASS>
__global__ void __launch_bounds__(256) k_test_lines(TestArgs A, int tpb) {
    if (PASS == 2 && (long long)*A.hits.count <= A.hits.cap) return;       // the list has them all
    __shared__ int big[3 * 256];
    __shared__ int nbig;
    __shared__ unsigned queue[8][64][2];              // [warp]: owner lane | axis << 5, line within the item
    if (threadIdx.x == 0) nbig = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long n3[3] = {A.n[0], A.n[1], A.n[2]};
    const long long t0 = (long long)blockIdx.x * tpb;
    const int mine = w * 32 + lane;
    float v[3][3] = {};             // vertices stay FP32 until a test needs them (conversions cost an FP64 slot)
    int lo[3] = {0, 0, 0}, len[3] = {0, 0, 0};
    if (mine < tpb && t0 + mine < A.ntri) {
        const float* t = A.tri + 9 * (t0 + mine);
        bool ok = true;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            v[q / 3][q % 3] = t[q];
            ok = ok && isfinite(v[q / 3][q % 3]);
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            long long l, h;
            line_range((double)fminf(fminf(v[0][d], v[1][d]), v[2][d]), (double)fmaxf(fmaxf(v[0][d], v[1][d]), v[2][d]), n3[d], l, h);
            if (ok && h >= l) {
                lo[d] = (int)l;
                len[d] = (int)(h - l + 1);
            }
        }
    }
    unsigned long long ntests = 0;
    auto store = [&](bool hit, long long fid, unsigned long long bits) {
        if (PASS == 1) {
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (!m) return;
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(A.hits.count, (unsigned long long)__popc(m));
            base = __shfl_sync(0xffffffffu, base, 0);
            const long long pos = (long long)base + __popc(m & ((1u << lane) - 1u));
            if (hit && pos < A.hits.cap) {
                A.hits.t[pos] = bits;
                A.hits.fid[pos] = (unsigned)fid;
            }
        }
        if (hit) use_hit<PASS>(A, fid, bits);
    };
    if (w * 32 < tpb) {
        int nq = 0;
        // takes the first min(32, nq) entries of the queue
        auto drain = [&]() {
            const bool on = lane < nq;
            const unsigned e = on ? queue[w][lane][0] : 0u, l = on ? queue[w][lane][1] : 0u;
            const int own = (int)(e & 31u), a = (int)(e >> 5);
            float r[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) r[q] = __shfl_sync(0xffffffffu, v[q / 3][q % 3], own);
            int o3[3], l3[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                o3[d] = __shfl_sync(0xffffffffu, lo[d], own);
                l3[d] = __shfl_sync(0xffffffffu, len[d], own);
            }
            Tri Q;
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                const float x = r[3 * p], y = r[3 * p + 1], z = r[3 * p + 2];
                Q.v[p][0] = (double)(a == 0 ? x : (a == 1 ? y : z));
                Q.v[p][1] = (double)(a == 0 ? y : (a == 1 ? z : x));
                Q.v[p][2] = (double)(a == 0 ? z : (a == 1 ? x : y));
            }
            const unsigned nb = (unsigned)(a == 0 ? l3[1] : (a == 1 ? l3[2] : l3[0])), jc = nb ? l / nb : 0u;
            const int b0 = a == 0 ? o3[1] : (a == 1 ? o3[2] : o3[0]), c0 = a == 0 ? o3[2] : (a == 1 ? o3[0] : o3[1]);
            long long fid = 0;
            unsigned long long bits = 0;
            const bool hit = on && face_hit(Q, a, b0 + (int)(l - jc * nb), c0 + (int)jc, A.n, A.eps_edge, A.eps_det, fid, bits);
            store(hit, fid, bits);
            nq -= nq < 32 ? nq : 32;
        };
        const float epsf = A.eps_edge > 0.0 ? (float)A.eps_edge * 1.0001f : 0.f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int b = (a + 1) % 3, c = (a + 2) % 3;
            const long long all = (long long)len[b] * len[c];
            int cnt = 0;
            if (all > kBigItem) big[atomicAdd(&nbig, 1)] = 3 * mine + a;
            else cnt = (int)all;
            ntests += (unsigned long long)all;
            if (blockIdx.y != 0) continue;
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31), excl = incl - cnt;
            for (int g0 = 0; g0 < total; g0 += 32) {
                const int g = g0 + lane;
                int own = 0;                              // last lane with excl <= g (empty ones before it end there too)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const int e = __shfl_sync(0xffffffffu, excl, own + o);
                    if (e <= g) own += o;
                }
                float q[6];
#pragma unroll
                for (int p = 0; p < 3; ++p) {
                    q[2 * p] = __shfl_sync(0xffffffffu, v[p][b], own);
                    q[2 * p + 1] = __shfl_sync(0xffffffffu, v[p][c], own);
                }
                const int e0 = __shfl_sync(0xffffffffu, excl, own), nb = __shfl_sync(0xffffffffu, len[b], own);
                const int b0 = __shfl_sync(0xffffffffu, lo[b], own), c0 = __shfl_sync(0xffffffffu, lo[c], own);
                bool may = false;
                unsigned l = 0;
                if (g < total) {
                    l = (unsigned)(g - e0);
                    const int jc = (int)(l / (unsigned)nb), jb = (int)l - jc * nb;
                    may = !A.fp32 || !surely_outside(q[0], q[1], q[2], q[3], q[4], q[5], (float)(b0 + jb) + 0.5f,
                                                     (float)(c0 + jc) + 0.5f, epsf);
                }
                const unsigned m = __ballot_sync(0xffffffffu, may);
                if (may) {
                    const int pos = nq + __popc(m & ((1u << lane) - 1u));
                    queue[w][pos][0] = (unsigned)own | ((unsigned)a << 5);
                    queue[w][pos][1] = l;
                }
                nq += __popc(m);
                __syncwarp();
                if (nq >= 32) {
                    const int rest = nq - 32;
                    drain();
                    // the entries beyond the first 32 move to the front
                    unsigned t0 = 0, t1 = 0;
                    if (lane < rest) {
                        t0 = queue[w][32 + lane][0];
                        t1 = queue[w][32 + lane][1];
                    }
                    __syncwarp();
                    if (lane < rest) {
                        queue[w][lane][0] = t0;
                        queue[w][lane][1] = t1;
                    }
                    __syncwarp();
                }
            }
        }
        if (nq > 0) drain();
    }
    if (PASS == 1 && blockIdx.y == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ntests += __shfl_down_sync(0xffffffffu, ntests, o);
        if (lane == 0 && ntests) atomicAdd(A.tests, ntests);
    }
    __syncthreads();
    for (int q = 0; q < nbig; ++q) {
        const int item = big[q], a = item % 3, b = (a + 1) % 3, c = (a + 2) % 3;
        const float* t = A.tri + 9 * (t0 + item / 3);
        Tri Q;
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            Q.v[p][0] = (double)t[3 * p + a];
            Q.v[p][1] = (double)t[3 * p + b];
            Q.v[p][2] = (double)t[3 * p + c];
        }
        long long bl, bh, cl, ch;
        line_range(fmin(fmin(Q.v[0][1], Q.v[1][1]), Q.v[2][1]), fmax(fmax(Q.v[0][1], Q.v[1][1]), Q.v[2][1]), n3[b], bl, bh);
        line_range(fmin(fmin(Q.v[0][2], Q.v[1][2]), Q.v[2][2]), fmax(fmax(Q.v[0][2], Q.v[1][2]), Q.v[2][2]), n3[c], cl, ch);
        const long long nb = bh - bl + 1, total = nb * (ch - cl + 1);
        for (long long g0 = (long long)blockIdx.y * 256; g0 < total; g0 += (long long)gridDim.y * 256) {
            const long long g = g0 + threadIdx.x;
            long long fid = 0;
            unsigned long long bits = 0;
            bool hit = false;
            if (g < total) {
                const unsigned jc = (unsigned)g / (unsigned)nb;           // lines of one axis: fewer than 2^31
                hit = face_hit(Q, a, (int)(bl + (g - jc * nb)), (int)(cl + jc), A.n, A.eps_edge, A.eps_det, fid, bits);
            }
            store(hit, fid, bits);
        }
    }
}

__global__ void __launch_bounds__(256) k_apply_hits(TestArgs A) {
    const long long n = (long long)*A.hits.count;
    if (n > A.hits.cap) return;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        use_hit<2>(A, (long long)A.hits.fid[q], A.hits.t[q]);
}

// ---- lists from the flags -----------------------------------------------------------------------
//
// A block takes a tile of 256 * CPT cells, a thread CPT (16 or 64) consecutive ones as 16-byte loads; almost
// all are zero, so the passes cost the flags' bytes (one per cell) and not the tables behind them.
constexpr int kListThreads = IBM_SCAN_NT;

template <int CPT>
struct FlagChunk {
    uint32_t w[CPT / 4];
    __device__ __forceinline__ FlagChunk(const uint8_t* __restrict__ f, long long c0, long long N) {
#pragma unroll
        for (int q = 0; q < CPT / 16; ++q) {
            const long long c = c0 + 16 * q;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (c + 16 <= N && ((uintptr_t)(f + c) & 15u) == 0) {
                v = *reinterpret_cast<const uint4*>(f + c);
            } else if (c < N) {
                unsigned t[4] = {0u, 0u, 0u, 0u};
                for (int m = 0; m < 16 && c + m < N; ++m) t[m >> 2] |= (unsigned)f[c + m] << (8 * (m & 3));
                v = make_uint4(t[0], t[1], t[2], t[3]);
            }
            w[4 * q] = v.x;
            w[4 * q + 1] = v.y;
            w[4 * q + 2] = v.z;
            w[4 * q + 3] = v.w;
        }
    }
};

// Cut faces of the three axes, 20 bits each (a tile has at most 16384 of each).
template <int CPT>
__device__ __forceinline__ long long face_counts(const FlagChunk<CPT>& F) {
    int n0 = 0, n1 = 0, n2 = 0;
#pragma unroll
    for (int q = 0; q < CPT / 4; ++q) {
        n0 += __popc(F.w[q] & 0x02020202u);
        n1 += __popc(F.w[q] & 0x08080808u);
        n2 += __popc(F.w[q] & 0x20202020u);
    }
    return (long long)n0 | ((long long)n1 << 20) | ((long long)n2 << 40);
}

template <int CPT>
__global__ void __launch_bounds__(kListThreads) k_face_counts(const uint8_t* __restrict__ flags, long long N, long long nt,
                                                              long long* __restrict__ tiles) {
    const FlagChunk<CPT> F(flags, ((long long)blockIdx.x * kListThreads + threadIdx.x) * CPT, N);
    long long tot;
    block_exscan(face_counts(F), tot);
    if (threadIdx.x < 3) tiles[threadIdx.x * nt + blockIdx.x] = (tot >> (20 * threadIdx.x)) & 0xfffff;
}

template <int CPT>
__global__ void __launch_bounds__(kListThreads) k_emit_faces(const uint8_t* __restrict__ flags, long long N, long long nt,
                                                             const long long* __restrict__ tiles,
                                                             const unsigned long long* __restrict__ tmin,
                                                             const unsigned long long* __restrict__ tmax,
                                                             int64_t* __restrict__ face_id, double* __restrict__ t_lo,
                                                             double* __restrict__ t_hi, long long cap) {
    const long long c0 = ((long long)blockIdx.x * kListThreads + threadIdx.x) * CPT;
    const FlagChunk<CPT> F(flags, c0, N);
    const long long cnt = face_counts(F);
    if (!__syncthreads_or(cnt != 0)) return;
    long long tot;
    const long long off = block_exscan(cnt, tot);
    if (!cnt) return;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        long long o = tiles[a * nt + blockIdx.x] + ((off >> (20 * a)) & 0xfffff);
#pragma unroll
        for (int q = 0; q < CPT / 4; ++q) {
            unsigned m = F.w[q] & (0x02020202u << (2 * a));
            while (m) {
                const int bit = __ffs(m) - 1;
                m &= m - 1;
                if (o < cap) {
                    const long long f = a * N + c0 + 4 * q + (bit >> 3);
                    face_id[o] = f;
                    t_lo[o] = __longlong_as_double((long long)tmin[f]);
                    t_hi[o] = __longlong_as_double((long long)tmax[f]);
                }
                ++o;
            }
        }
    }
}

inline bool wide_tiles(long long N) { return N >= (4LL << 20); }      // 64 cells per thread (else 16)
inline long long list_tiles(long long N) {
    const long long t = (long long)kListThreads * (wide_tiles(N) ? 64 : 16);
    return (N + t - 1) / t;
}

struct Workspace {
    unsigned long long* tmin;
    unsigned long long* tmax;
    unsigned char* hits;   // 8 (3 ntri + 1) bytes
    long long* tiles;
    long long* scalars;    // [0] tests, [1] cut faces, [2] hits
    size_t bytes;
};

inline size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

Workspace carve(void* base, long long N, long long ntri) {
    Workspace w;
    char* p = (char*)base;
    size_t o = 0;
    const long long nt = scan_tiles(3 * N > 3 * ntri ? 3 * N : 3 * ntri) + 1;
    w.tmin = (unsigned long long*)(p + o); o += align256(sizeof(unsigned long long) * 3 * N);
    w.tmax = (unsigned long long*)(p + o); o += align256(sizeof(unsigned long long) * 3 * N);
    w.hits = (unsigned char*)(p + o); o += align256(sizeof(long long) * (3 * ntri + 1));
    w.tiles = (long long*)(p + o); o += align256(sizeof(long long) * nt);
    w.scalars = (long long*)(p + o); o += align256(sizeof(long long) * 4);
    w.bytes = o;
    return w;
}

unsigned blocks_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    long long cap = 32LL * IBM_NSM;
    if (b > cap) b = cap;
    return (unsigned)(b < 1 ? 1 : b);
}

}  // namespace

extern "C" size_t ibm_classify_workspace_bytes(const ibm_grid* g, int64_t ntri) {
    if (!g || g->nx <= 0 || g->ny <= 0 || g->nz <= 0 || ntri < 0) return 0;
    return carve(nullptr, (long long)g->nx * g->ny * g->nz, ntri).bytes;
}

int ibm_check_grid(const ibm_grid* g);

extern "C" int ibm_classify(const ibm_grid* g, const float* d_tri, int64_t ntri, const ibm_geom_params* gp,
                            uint8_t* d_flags, int64_t* d_face_id, double* d_t_lo, double* d_t_hi, int64_t cap,
                            int64_t* n_cut, int64_t* n_tests, void* d_ws, size_t ws_bytes, void* stream) {
    int rc = ibm_check_grid(g);
    if (rc) return rc;
    if (!gp || !d_flags || !n_cut || (ntri > 0 && !d_tri) || ntri < 0 || cap < 0 ||
        (cap > 0 && (!d_face_id || !d_t_lo || !d_t_hi)))
        return ibm_fail(IBM_E_INVALID, "ibm_classify: null or negative argument");
    const long long N = (long long)g->nx * g->ny * g->nz;
    Workspace w = carve(d_ws, N, ntri);
    if (!d_ws || ws_bytes < w.bytes)
        return ibm_fail(IBM_E_INVALID, "ibm_classify: workspace of %zu bytes, %zu needed", ws_bytes, w.bytes);
    cudaStream_t s = (cudaStream_t)stream;
    IBM_CUDA(cudaMemsetAsync(d_flags, 0, (size_t)N, s));
    IBM_CUDA(cudaMemsetAsync(w.scalars, 0, 4 * sizeof(long long), s));
    if (ntri > 0) {
        TestArgs A;
        A.tri = d_tri;
        A.ntri = ntri;
        A.n[0] = g->nx; A.n[1] = g->ny; A.n[2] = g->nz;
        A.eps_edge = gp->eps_edge;
        A.eps_det = gp->eps_det;
        A.fp32 = g->nx <= 1 << 23 && g->ny <= 1 << 23 && g->nz <= 1 << 23;
        A.flags = d_flags;
        A.tmin = w.tmin;
        A.tmax = w.tmax;
        A.tests = (unsigned long long*)w.scalars;
        A.hits.cap = 8 * (3 * ntri + 1) / 12;
        A.hits.t = (unsigned long long*)w.hits;
        A.hits.fid = (unsigned*)(A.hits.t + A.hits.cap);
        A.hits.count = (unsigned long long*)w.scalars + 2;
        // triangles per block: all SMs for a small soup, then whole blocks; slices where few triangles may be large
        long long tpb = ntri / (4 * IBM_NSM);
        tpb = tpb < 1 ? 1 : (tpb > 256 ? 256 : tpb);
        const long long nb = (ntri + tpb - 1) / tpb;
        const dim3 grid((unsigned)nb, (unsigned)(nb < IBM_NSM ? 8 : 1));
        k_test_lines<1><<<grid, 256, 0, s>>>(A, (int)tpb);
        k_apply_hits<<<8 * IBM_NSM, 256, 0, s>>>(A);
        k_test_lines<2><<<grid, 256, 0, s>>>(A, (int)tpb);
        IBM_LAUNCHED("ibm_classify: k_test_lines");
    }
    // count first; the list is only written as far as it fits
    const long long nt = list_tiles(N);
    if (wide_tiles(N)) k_face_counts<64><<<(unsigned)nt, kListThreads, 0, s>>>(d_flags, N, nt, w.tiles);
    else k_face_counts<16><<<(unsigned)nt, kListThreads, 0, s>>>(d_flags, N, nt, w.tiles);
    k_scan_tile_totals<<<1, IBM_SCAN_NT, 0, s>>>(w.tiles, 3 * nt, w.scalars + 1);
    if (wide_tiles(N))
        k_emit_faces<64><<<(unsigned)nt, kListThreads, 0, s>>>(d_flags, N, nt, w.tiles, w.tmin, w.tmax, d_face_id, d_t_lo, d_t_hi, cap);
    else
        k_emit_faces<16><<<(unsigned)nt, kListThreads, 0, s>>>(d_flags, N, nt, w.tiles, w.tmin, w.tmax, d_face_id, d_t_lo, d_t_hi, cap);
    IBM_LAUNCHED("ibm_classify: cut faces");
    long long host[2];
    IBM_CUDA(cudaMemcpyAsync(host, w.scalars, sizeof(host), cudaMemcpyDeviceToHost, s));
    IBM_CUDA(cudaStreamSynchronize(s));
    *n_cut = host[1];
    if (n_tests) *n_tests = host[0];
    if (host[1] > cap)
        return ibm_fail(IBM_E_CAPACITY, "ibm_classify: %lld cut faces, capacity %lld", host[1], (long long)cap);
    return IBM_OK;
}

// ------------------------------------------------------------------------------------------------
// Setup

struct ibm_geom {
    int device;
    ibm_grid grid;
    ibm_geom_params gp;
    long long N;
    long long n_cut, n_rec, n_inc;
    int pooled;            // cellrec and rec are from the pool
    uint8_t* flags;        // caller-owned
    int32_t* cellrec;      // [N]
    LinkRec* rec;          // [n_rec]
    int32_t* inc;          // [n_inc] Omega_inc cells in index order (behind rec in its allocation)
};

namespace {

// Omega_inc (bit 6) and Omega_adj (bit 7).  W cells per thread (4 as one word where rows are whole words);
// words that come out as they were (nearly all are 0) are not written.
template <int W>
__global__ void __launch_bounds__(256) k_region_bits(int nx, int ny, int nz, uint8_t* flags) {
    const long long N = (long long)nx * ny * nz, nxy = (long long)nx * ny;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < N / W; q += (long long)gridDim.x * blockDim.x) {
        const unsigned c = (unsigned)(q * W), r = c / (unsigned)nx;       // grids of fewer than 2^31 cells
        const int i = (int)(c - r * (unsigned)nx), j = (int)(r % (unsigned)ny), k = (int)(r / (unsigned)ny);
        auto cut = [&](long long o) -> unsigned {                           // 1 in the byte of every cell with a cut link
            if (W == 4) return ((*reinterpret_cast<const unsigned*>(flags + c + o) & 0x3f3f3f3fu) + 0x3f3f3f3fu) >> 6 & 0x01010101u;
            return (flags[c + o] & 63u) ? 1u : 0u;
        };
        const unsigned own = cut(0);
        unsigned nb = 0;
        if (j > 0) nb |= cut(-nx);
        if (j < ny - 1) nb |= cut(nx);
        if (k > 0) nb |= cut(-nxy);
        if (k < nz - 1) nb |= cut(nxy);
        if (W == 4) nb |= (own << 8) | (own >> 8);
        if (i > 0 && (flags[c - 1] & 63u)) nb |= 1u;
        if (i + W < nx && (flags[c + W] & 63u)) nb |= 1u << (8 * (W - 1));
        const unsigned raw = W == 4 ? *reinterpret_cast<const unsigned*>(flags + c) : flags[c];
        const unsigned out = (raw & 0x3f3f3f3fu) | (own << 6) | ((nb & ~own) << 7);
        if (out == raw) continue;
        if (W == 4) *reinterpret_cast<unsigned*>(flags + c) = out;
        else flags[c] = (uint8_t)out;
    }
}

// Records (low 32 bits) and Omega_inc cells (high bits) of a thread's cells.
template <int CPT>
__device__ __forceinline__ long long rec_counts(const FlagChunk<CPT>& F) {
    int nr = 0, ni = 0;
#pragma unroll
    for (int q = 0; q < CPT / 4; ++q) {
        const unsigned m = F.w[q] & 0x3f3f3f3fu;
        nr += __popc(m);
        ni += __popc((m + 0x3f3f3f3fu) & 0x40404040u);
    }
    return (long long)nr | ((long long)ni << 32);
}

template <int CPT>
__global__ void __launch_bounds__(kListThreads) k_rec_counts(const uint8_t* __restrict__ flags, long long N,
                                                             long long* __restrict__ tiles) {
    const FlagChunk<CPT> F(flags, ((long long)blockIdx.x * kListThreads + threadIdx.x) * CPT, N);
    long long tot;
    block_exscan(rec_counts(F), tot);
    if (threadIdx.x == 0) tiles[blockIdx.x] = tot;
}

// First record of every Omega_inc cell (cellrec holds -1 before) and the list of these cells.
template <int CPT>
__global__ void __launch_bounds__(kListThreads) k_emit_cellrec(const uint8_t* __restrict__ flags, long long N,
                                                               const long long* __restrict__ tiles,
                                                               int32_t* __restrict__ cellrec, int32_t* __restrict__ inc) {
    const long long c0 = ((long long)blockIdx.x * kListThreads + threadIdx.x) * CPT;
    const FlagChunk<CPT> F(flags, c0, N);
    const long long cnt = rec_counts(F);
    if (!__syncthreads_or(cnt != 0)) return;
    long long tot;
    long long o = tiles[blockIdx.x] + block_exscan(cnt, tot);
    if (!cnt) return;
#pragma unroll
    for (int q = 0; q < CPT / 4; ++q) {
        if (!(F.w[q] & 0x3f3f3f3fu)) continue;
        for (int m = 0; m < 4; ++m) {
            const unsigned f = (F.w[q] >> (8 * m)) & 63u;
            if (!f) continue;
            const long long c = c0 + 4 * q + m;
            cellrec[c] = (int32_t)(o & 0xffffffffLL);
            inc[o >> 32] = (int32_t)c;
            o += (1LL << 32) | (long long)__popc(f);
        }
    }
}

// Eq. q_axis: upper branch (Dx/d) q_IB + ((d - Dx)/d) q_P on d/Dx >= 1/2; lower branch
// 2 q_IB + ((2d - Dx)/Dx) q_O - (2d/Dx) q_P on d/Dx < 1/2 when the opposite neighbour O is usable;
// otherwise the upper branch at d = 1/2.  Eq. distribution_function weights with the near distance d.
//
// One thread per cut face writes the records of its two cells: a record's place follows from its cell's first
// record and flags, so nothing is searched.  The flags name 2 n_cut links (checked before); a list whose ids
// rise strictly and whose every face is flagged from both of its cells therefore covers each link once.
// Vehicle assembly: 0.29 ms, 2.3 ms with a binary search of the list per record.
__global__ void __launch_bounds__(128) k_build_records(int nx, int ny, int nz, const uint8_t* __restrict__ flags,
                                                       const int32_t* __restrict__ cellrec, const int64_t* __restrict__ fid,
                                                       const double* __restrict__ t_lo, const double* __restrict__ t_hi,
                                                       long long n_cut, LinkRec* __restrict__ rec, int* __restrict__ err) {
    const long long N = (long long)nx * ny * nz;
    const long long stb[3] = {1, nx, (long long)nx * ny};
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n_cut; q += (long long)gridDim.x * blockDim.x) {
        const long long id = fid[q];
        bool ok = id >= 0 && id < 3 * N && (q == 0 || fid[q - 1] < id);
        int a = 0, xa = 0, na = 1;
        long long c = 0, st = 1;
        if (ok) {
            a = id >= 2 * N ? 2 : (id >= N ? 1 : 0);
            c = id - a * N;
            st = stb[a];
            na = a == 0 ? nx : (a == 1 ? ny : nz);
            const unsigned u = (unsigned)c, r = u / (unsigned)nx;
            xa = a == 0 ? (int)(u - r * (unsigned)nx) : (a == 1 ? (int)(r % (unsigned)ny) : (int)(r / (unsigned)ny));
            ok = xa + 1 < na && ((flags[c] >> (2 * a + 1)) & 1u) && ((flags[c + st] >> (2 * a)) & 1u);
        }
        if (!ok) {
            atomicExch(err, 1);
            continue;
        }
        for (int s = 1; s >= -1; s -= 2) {
            const long long P = s > 0 ? c : c + st;
            const int bit = 2 * a + (s > 0), x = s > 0 ? xa : xa + 1;
            const unsigned f = flags[P] & 63u;
            const double d = s > 0 ? t_lo[q] : __dsub_rn(1.0, t_hi[q]);
            LinkRec r;
            r.cell = (int32_t)P;
            r.far = (int32_t)(P + s * st);
            r.axis = (int8_t)a;
            r.side = (int8_t)s;
            r.pad = 0;
            r.d = d;
            const int yo = x - s;
            const bool o_ok = yo >= 0 && yo < na && !((f >> (2 * a + (s > 0 ? 0 : 1))) & 1u);
            if (d >= 0.5) {
                r.branch = 0;
                r.opp = -1;
                r.c_ib = __ddiv_rn(1.0, d);
                r.c_p = __ddiv_rn(__dsub_rn(d, 1.0), d);
                r.c_o = 0.0;
            } else if (o_ok) {
                r.branch = 1;
                r.opp = (int32_t)(P - s * st);
                r.c_ib = 2.0;
                r.c_o = __dsub_rn(__dmul_rn(2.0, d), 1.0);
                r.c_p = -__dmul_rn(2.0, d);
            } else {
                r.branch = 2;
                r.opp = -1;
                r.c_ib = 2.0;
                r.c_p = -1.0;
                r.c_o = 0.0;
            }
            const double den = __dadd_rn(1.0, d);
            r.w_fluid = __ddiv_rn(d, den);
            r.w_ghost = __ddiv_rn(__dsub_rn(1.0, d), den);
            r.uib[0] = r.uib[1] = r.uib[2] = 0.0;
            rec[cellrec[P] + __popc(f & ((1u << bit) - 1u))] = r;
        }
    }
}

__global__ void k_export(const LinkRec* __restrict__ rec, long long n, int64_t* __restrict__ idx,
                         double* __restrict__ coef) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const LinkRec& r = rec[q];
        if (idx) {
            idx[6 * q + 0] = r.cell;
            idx[6 * q + 1] = r.far;
            idx[6 * q + 2] = r.opp;
            idx[6 * q + 3] = r.axis;
            idx[6 * q + 4] = r.side;
            idx[6 * q + 5] = r.branch;
        }
        if (coef) {
            coef[6 * q + 0] = r.d;
            coef[6 * q + 1] = r.c_ib;
            coef[6 * q + 2] = r.c_p;
            coef[6 * q + 3] = r.c_o;
            coef[6 * q + 4] = r.w_fluid;
            coef[6 * q + 5] = r.w_ghost;
        }
    }
}

__global__ void k_export_cellrec(const int32_t* __restrict__ cr, long long n, int64_t* __restrict__ out) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        out[q] = cr[q];
}

__global__ void k_set_uib(LinkRec* __restrict__ rec, long long n, const double* __restrict__ uib) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        for (int c = 0; c < 3; ++c) rec[q].uib[c] = uib ? uib[3 * q + c] : 0.0;
}

// ---- memory of the geometry handles -----------------------------------------------------------------
//
// A moving body is classified again and again; mapping and unmapping the tables (0.8 GB for 201 M cells) took 1.4
// of the 3.4 ms of a vehicle and 160 of the 420 us of a small sphere.  They come from a pool of the stream-ordered
// allocator that keeps up to kPoolKeep bytes of freed memory per device; what lies beyond goes back at the next
// synchronisation, the rest when any allocation of this library fails (ibm_malloc) or the caller asks for it
// (ibm_geom_trim).  A handle may have been used on any stream, so freeing waits for the device, as cudaFree does.
// A pool lives as long as its context: cudaDeviceReset ends it, so pools are found by the context's id, which no later
// context repeats.
const unsigned long long kPoolKeep = 2ULL << 30;
const int kPools = 64;                    // contexts with a pool; the ones after them take cudaMalloc
struct ContextPool {
    unsigned long long ctx;
    cudaMemPool_t pool;                   // null: the device has none
};
std::mutex g_pool_mutex;
ContextPool g_pool[kPools];
int g_pools;

// Id of the current context (made if the device has none), 0 if it cannot be told.
unsigned long long context_id() {
    typedef int (*GetId)(void*, unsigned long long*);         // cuCtxGetId
    static const GetId get = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult r;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &r);
        if (e != cudaSuccess) cudaGetLastError();
        return e == cudaSuccess && r == cudaDriverEntryPointSuccess ? (GetId)f : (GetId) nullptr;
    }();
    unsigned long long id = 0;
    if (!get) return 0;
    if (get(nullptr, &id) == 0) return id;
    return cudaFree(nullptr) == cudaSuccess && get(nullptr, &id) == 0 ? id : 0;
}

cudaMemPool_t context_pool(bool create) {
    const unsigned long long ctx = context_id();
    if (!ctx) return nullptr;
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    for (int k = 0; k < g_pools; ++k)
        if (g_pool[k].ctx == ctx) return g_pool[k].pool;
    int dev = 0;
    if (!create || g_pools == kPools || cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    cudaMemPoolProps p = {};
    p.allocType = cudaMemAllocationTypePinned;
    p.location.type = cudaMemLocationTypeDevice;
    p.location.id = dev;
    cudaMemPool_t q = nullptr;
    unsigned long long keep = kPoolKeep;
    if (cudaMemPoolCreate(&q, &p) != cudaSuccess || cudaMemPoolSetAttribute(q, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        q = nullptr;
    }
    g_pool[g_pools++] = ContextPool{ctx, q};
    return q;
}

// What freed tables hold goes back to the device.
cudaError_t pool_trim() {
    const cudaMemPool_t q = context_pool(false);
    if (!q) return cudaSuccess;
    const cudaError_t e = cudaDeviceSynchronize();
    return e != cudaSuccess ? e : cudaMemPoolTrimTo(q, 0);
}

// q: the context's pool, or null.
cudaError_t geom_alloc(cudaMemPool_t q, void** p, size_t bytes, cudaStream_t s) {
    if (!q) return cudaMalloc(p, bytes);
    cudaError_t e = cudaMallocFromPoolAsync(p, bytes, q, s);
    if (e == cudaErrorMemoryAllocation) {               // memory the pool holds may be in pieces
        cudaGetLastError();
        pool_trim();
        e = cudaMallocFromPoolAsync(p, bytes, q, s);
        if (e != cudaSuccess) cudaGetLastError();
    }
    return e;
}

void geom_free(ibm_geom* G) {
    cudaDeviceSynchronize();
    for (void* p : {(void*)G->cellrec, (void*)G->rec})
        if (p && G->pooled) cudaFreeAsync(p, 0);
        else if (p) cudaFree(p);
}

}  // namespace

cudaError_t ibm_malloc_bytes(void** p, size_t bytes) {
    const cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    if (pool_trim() != cudaSuccess) return e;
    const cudaError_t again = cudaMalloc(p, bytes);
    if (again != cudaSuccess) cudaGetLastError();
    return again;
}

extern "C" int ibm_geom_trim(void) {
    IBM_CUDA(pool_trim());
    return IBM_OK;
}

extern "C" void ibm_geom_destroy(ibm_geom* G) {
    if (!G) return;
    int dev = -1;
    cudaGetDevice(&dev);
    if (dev != G->device) cudaSetDevice(G->device);
    geom_free(G);
    if (dev != G->device && dev >= 0) cudaSetDevice(dev);
    free(G);
}

extern "C" int ibm_setup(const ibm_grid* g, const ibm_geom_params* gp, uint8_t* d_flags, const int64_t* d_face_id,
                         const double* d_t_lo, const double* d_t_hi, int64_t n_cut, ibm_geom** out, void* stream) {
    int rc = ibm_check_grid(g);
    if (rc) return rc;
    if (!gp || !d_flags || !out || n_cut < 0 || (n_cut > 0 && (!d_face_id || !d_t_lo || !d_t_hi)))
        return ibm_fail(IBM_E_INVALID, "ibm_setup: null or negative argument");
    *out = nullptr;
    cudaStream_t s = (cudaStream_t)stream;
    ibm_geom* G = (ibm_geom*)calloc(1, sizeof(ibm_geom));
    if (!G) return ibm_fail(IBM_E_NOMEM, "ibm_setup: host allocation");
    cudaGetDevice(&G->device);
    G->grid = *g;
    G->gp = *gp;
    G->N = (long long)g->nx * g->ny * g->nz;
    G->n_cut = n_cut;
    G->flags = d_flags;
    long long* tiles = nullptr;                 // tile totals, their sum, the error word
    long long host = 0;
    int herr = 0;
    const long long nt = list_tiles(G->N);
    cudaError_t e;
    const cudaMemPool_t pool = context_pool(true);
    G->pooled = pool != nullptr;
    const bool words = g->nx % 4 == 0 && ((uintptr_t)d_flags & 3u) == 0;
    // one allocation for the cell table with the scan's tile totals behind it, one for the cell list and records
    const size_t cellb = (sizeof(int32_t) * (size_t)G->N + 15) & ~(size_t)15;
    if ((e = geom_alloc(pool, (void**)&G->cellrec, cellb + sizeof(long long) * (nt + 2), s)) != cudaSuccess) goto nomem;
    tiles = (long long*)((char*)G->cellrec + cellb);
    if (words) k_region_bits<4><<<blocks_for(G->N / 4, 256), 256, 0, s>>>(g->nx, g->ny, g->nz, d_flags);
    else k_region_bits<1><<<blocks_for(G->N, 256), 256, 0, s>>>(g->nx, g->ny, g->nz, d_flags);
    if (wide_tiles(G->N)) k_rec_counts<64><<<(unsigned)nt, kListThreads, 0, s>>>(d_flags, G->N, tiles);
    else k_rec_counts<16><<<(unsigned)nt, kListThreads, 0, s>>>(d_flags, G->N, tiles);
    k_scan_tile_totals<<<1, IBM_SCAN_NT, 0, s>>>(tiles, nt, tiles + nt);
    if ((e = cudaGetLastError()) != cudaSuccess) goto cuda_err;
    if ((e = cudaMemcpyAsync(&host, tiles + nt, sizeof(long long), cudaMemcpyDeviceToHost, s)) != cudaSuccess) goto cuda_err;
    if ((e = cudaMemsetAsync(G->cellrec, 0xff, sizeof(int32_t) * G->N, s)) != cudaSuccess) goto cuda_err;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) goto cuda_err;
    G->n_rec = host & 0xffffffffLL;
    G->n_inc = host >> 32;
    if (G->n_rec != 2 * n_cut) {
        ibm_geom_destroy(G);
        return ibm_fail(IBM_E_INVALID, "ibm_setup: flags name %lld cut links but the list has %lld faces",
                        host & 0xffffffffLL, (long long)n_cut);
    }
    if ((e = geom_alloc(pool, (void**)&G->rec, sizeof(LinkRec) * (size_t)G->n_rec + sizeof(int32_t) * (size_t)(G->n_inc + 4), s)) != cudaSuccess)
        goto nomem;
    G->inc = (int32_t*)(G->rec + G->n_rec);
    if (n_cut > 0) {
        int* const d_err = (int*)(tiles + nt + 1);
        if ((e = cudaMemsetAsync(d_err, 0, sizeof(int), s)) != cudaSuccess) goto cuda_err;
        if (wide_tiles(G->N)) k_emit_cellrec<64><<<(unsigned)nt, kListThreads, 0, s>>>(d_flags, G->N, tiles, G->cellrec, G->inc);
        else k_emit_cellrec<16><<<(unsigned)nt, kListThreads, 0, s>>>(d_flags, G->N, tiles, G->cellrec, G->inc);
        k_build_records<<<blocks_for(n_cut, 128), 128, 0, s>>>(g->nx, g->ny, g->nz, d_flags, G->cellrec, d_face_id, d_t_lo,
                                                               d_t_hi, n_cut, G->rec, d_err);
        if ((e = cudaGetLastError()) != cudaSuccess) goto cuda_err;
        if ((e = cudaMemcpyAsync(&herr, d_err, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess) goto cuda_err;
    }
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) goto cuda_err;
    if (herr) {
        ibm_geom_destroy(G);
        return ibm_fail(IBM_E_INVALID, "ibm_setup: a cut link has no entry in the cut-face list");
    }
    *out = G;
    return IBM_OK;
nomem:
    ibm_geom_destroy(G);
    return ibm_fail(IBM_E_NOMEM, "ibm_setup: %s", cudaGetErrorString(e));
cuda_err:
    ibm_geom_destroy(G);
    return ibm_cuda_check(e, "ibm_setup");
}

extern "C" int ibm_geom_info(const ibm_geom* G, int64_t* n_rec, int64_t* n_inc) {
    if (!G) return ibm_fail(IBM_E_INVALID, "ibm_geom_info: null geometry");
    if (n_rec) *n_rec = G->n_rec;
    if (n_inc) *n_inc = G->n_inc;
    return IBM_OK;
}

extern "C" int ibm_geom_export(const ibm_geom* G, int64_t* d_idx, double* d_coef, int64_t* d_cellrec, void* stream) {
    if (!G) return ibm_fail(IBM_E_INVALID, "ibm_geom_export: null geometry");
    cudaStream_t s = (cudaStream_t)stream;
    if ((d_idx || d_coef) && G->n_rec > 0) k_export<<<blocks_for(G->n_rec, 256), 256, 0, s>>>(G->rec, G->n_rec, d_idx, d_coef);
    if (d_cellrec && G->N > 0) k_export_cellrec<<<blocks_for(G->N, 256), 256, 0, s>>>(G->cellrec, G->N, d_cellrec);
    IBM_LAUNCHED("ibm_geom_export");
    return IBM_OK;
}

extern "C" int ibm_set_boundary_velocity(ibm_geom* G, const double* d_uib, void* stream) {
    if (!G) return ibm_fail(IBM_E_INVALID, "ibm_set_boundary_velocity: null geometry");
    if (G->n_rec > 0) k_set_uib<<<blocks_for(G->n_rec, 256), 256, 0, (cudaStream_t)stream>>>(G->rec, G->n_rec, d_uib);
    IBM_LAUNCHED("ibm_set_boundary_velocity");
    return IBM_OK;
}

// Accessors for the solver (api.cu).
void ibm_geom_device(const ibm_geom* G, const uint8_t** flags, const int32_t** cellrec, const LinkRec** rec,
                     const int32_t** inc, long long* n_rec, long long* n_inc) {
    *flags = G->flags;
    *cellrec = G->cellrec;
    *rec = G->rec;
    *inc = G->inc;
    *n_rec = G->n_rec;
    *n_inc = G->n_inc;
}
const ibm_grid* ibm_geom_grid(const ibm_geom* G) { return &G->grid; }
int ibm_geom_deadend(const ibm_geom* G) { return G->gp.deadend_on ? 1 : 0; }

// ------------------------------------------------------------------------------------------------
// Classification without any allocation, for callers that cannot call cudaMalloc.
//
// The scratch lives in a fixed device array of this file.  Its name in host code is only a host-side
// stand-in, so the device address is looked up once per device with cudaGetSymbolAddress (with that
// device current) and cached; kernels receive that address.  The cache holds for the life of the
// device's context: a cudaDeviceReset invalidates it (documented in the header).

#include <mutex>

#define IBM_NOALLOC_SCRATCH_BYTES (32u << 20)   // 32 MiB, held by every GPU that loads the library
#define IBM_NOALLOC_MAX_DEVICES 64

static __device__ __align__(256) unsigned char g_noalloc_scratch[IBM_NOALLOC_SCRATCH_BYTES];

static void* g_noalloc_ptr[IBM_NOALLOC_MAX_DEVICES];
static std::mutex g_noalloc_mutex;

extern "C" int ibm_classify_noalloc(const ibm_grid* g, const float* d_tri, int64_t ntri, const ibm_geom_params* gp,
                                    uint8_t* d_flags, int64_t* d_face_id, double* d_t_lo, double* d_t_hi,
                                    int64_t cap, int64_t* n_cut, int64_t* n_tests, void* stream) {
    int rc = ibm_check_grid(g);
    if (rc) return rc;
    if (ntri < 0) return ibm_fail(IBM_E_INVALID, "ibm_classify_noalloc: negative triangle count");
    const size_t need = ibm_classify_workspace_bytes(g, ntri);
    if (need > IBM_NOALLOC_SCRATCH_BYTES)
        return ibm_fail(IBM_E_INVALID,
                        "ibm_classify_noalloc: this grid and soup need %zu bytes of scratch, more than the "
                        "%u bytes the library reserves; use ibm_classify with a caller workspace",
                        need, (unsigned)IBM_NOALLOC_SCRATCH_BYTES);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return ibm_cuda_check(e, "ibm_classify_noalloc: cudaGetDevice");
    if (dev < 0 || dev >= IBM_NOALLOC_MAX_DEVICES)
        return ibm_fail(IBM_E_INVALID, "ibm_classify_noalloc: device ordinal %d not supported", dev);
    void* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        if (!g_noalloc_ptr[dev]) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess) return ibm_cuda_check(e, "ibm_classify_noalloc: cudaGetSymbolAddress");
            g_noalloc_ptr[dev] = p;
        }
        scratch = g_noalloc_ptr[dev];
    }
    // every part of the scratch that must start from a known value is initialised by ibm_classify
    return ibm_classify(g, d_tri, ntri, gp, d_flags, d_face_id, d_t_lo, d_t_hi, cap, n_cut, n_tests, scratch,
                        IBM_NOALLOC_SCRATCH_BYTES, stream);
}
