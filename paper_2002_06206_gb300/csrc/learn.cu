// learn.cu -- learned initial guess of the pressure Poisson solve: a small 3-D convolutional network
// (three 3x3x3 convolutions, 8 -> 8 -> 8 -> 1 channels, ReLU between) on the solver's grid that
// predicts how far p^{n+1} departs from the linear extrapolation 2 p^n - p^{n-1}, from the right-hand
// side, the last pressure change and the solid mask.  Activations and gradients are stored in BF16,
// channel-last (8 channels = 16 bytes per cell); the convolutions run as implicit GEMMs on the tensor
// cores (ldmatrix + mma.sync m16n8k16, BF16 operands, FP32 accumulation): M = 16 consecutive cells of
// a row, N = 8 channels, K = 27 taps x 8 channels (padded to 224).  The weight gradient is a reduction
// over all cells: the same tensor-core form with the cells as K, FP32 sums, per-block partials added in a fixed order.
#include <cuda_bf16.h>
#include <math.h>

#include "solver.cuh"

#define NN_C 8
#define NN_TAPS 27
#define NN_KSTEPS 14            // 224 / 16
#define NN_NPARAM (2 * NN_C * NN_TAPS * NN_C + NN_TAPS * NN_C + 2 * NN_C + 1)

// Per-layer weights: W[co][tap][ci] (layer 3 has co = 1), bias[co].
struct NetParams {
    float* w[3];
    float* b[3];
};

struct ibm_net {
    float* master;            // NN_NPARAM FP32 parameters (W1, W2, W3, b1, b2, b3)
    float* grad;              // gradients, same layout
    float* m;                 // Adam moments
    float* v;
    uint32_t* frag_fwd[3];    // packed BF16 B fragments: [14 k-steps][32 lanes][2 regs]
    uint32_t* frag_bwd[3];    // fragments of the transposed weights (input-gradient convolution)
    long long step;
    // per-grid buffers (resized on demand by the host calls that receive a grid)
    long long cap_cells;
    __nv_bfloat16* x0;        // features
    __nv_bfloat16* y1;
    __nv_bfloat16* y2;
    __nv_bfloat16* d3;        // 2 (out - target) in channel 0
    __nv_bfloat16* d2;
    __nv_bfloat16* d1;
    float* out;
    float* wpart;             // per-block weight-gradient partials
    double* scal;             // [0] feature scale s, [1] loss sum, [2..] reduction scratch
    double* partials;
    unsigned* counter;
};

namespace {


__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void mma_bf16(float d[4], const uint32_t a[4], const uint32_t b[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Convolution of a channel-last BF16 field with 27 taps on the tensor cores (implicit GEMM, K = 27
// taps x 8 channels padded to 224).  SGN = +1: forward (input at c + off); SGN = -1: input gradient
// (input at c - off, transposed weights).  MODE 0: store BF16 relu(acc + bias); 1: store FP32
// channel 0 of acc + bias; 2: store BF16 acc masked by (mask > 0) at the output cell (ReLU
// derivative).  The input is staged in shared memory.  A block owns a 32 x 4 (x, y) tile
// of output cells and walks kz planes; the input planes over the tile plus a one-cell halo sit in a four-plane
// ring (16 bytes per cell, zero outside the grid): three that are read and the one the plane loaded during the
// previous step goes into, so a step has one barrier and no load is waited for.  Warp w computes the
// 16 cells (w % 2) * 16 .. + 15 of row w / 2: for each k-step (two taps x 8 channels) one
// ldmatrix.x4 gathers the A fragment straight from the ring -- each lane names one 16-byte row, the
// input cell of its (cell, tap), a plane's base and a constant -- and one mma.sync accumulates it.
// Bound by the gathers, 27 shared-memory reads of every row per layer: 128^3 cells 38 us (input gradients 50, with the
// mask); 74 us with three planes, loads waited for and ring slots by remainders per tap.
#define NC_TX 32
#define NC_TY 4
#define NC_SX (NC_TX + 2)
#define NC_SY (NC_TY + 2)
#define NC_PL (NC_SX * NC_SY)
#define NC_RING 4

// The plane of the ring a thread fills: one position of the halo tile (threads beyond it: none), its value of the
// plane in flight.
struct RingFill {
    long long at;        // element offset within a plane of the grid, -1 outside
    uint4 v;
    __device__ __forceinline__ RingFill(int tid, int x0, int y0, int nx, int ny) {
        const int gx = x0 + tid % NC_SX - 1, gy = y0 + tid / NC_SX - 1;
        at = tid < NC_PL && gx >= 0 && gx < nx && gy >= 0 && gy < ny ? (gx + (long long)nx * gy) * NN_C : -1;
    }
    __device__ __forceinline__ void fetch(const __nv_bfloat16* __restrict__ in, int k, int nz, long long plane) {
        v = make_uint4(0u, 0u, 0u, 0u);
        if (at >= 0 && k >= 0 && k < nz) v = *reinterpret_cast<const uint4*>(in + k * plane + at);
    }
    __device__ __forceinline__ void put(uint4* ring, int k, int tid) const {
        if (tid < NC_PL) ring[((k + NC_RING) % NC_RING) * NC_PL + tid] = v;
    }
};

__device__ __forceinline__ void ldsm_x4(uint32_t r[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

template <int SGN, int MODE>
__global__ void __launch_bounds__(256, 4) k_nn_conv_tile(int nx, int ny, int nz, int kz, const __nv_bfloat16* __restrict__ in,
                                                         const uint32_t* __restrict__ frag, const float* __restrict__ bias,
                                                         __nv_bfloat16* __restrict__ outb, float* __restrict__ outf,
                                                         const __nv_bfloat16* __restrict__ mask) {
    __shared__ __align__(16) uint4 ring[NC_RING * NC_PL + 1];    // + one zero row for the padding tap
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int x0 = blockIdx.x * NC_TX, y0 = blockIdx.y * NC_TY, z0 = blockIdx.z * kz;
    const int z1 = z0 + kz < nz ? z0 + kz : nz;
    const long long plane = (long long)nx * ny * NN_C;
    if (tid == 0) ring[NC_RING * NC_PL] = make_uint4(0u, 0u, 0u, 0u);
    const int g = lane >> 2, q = lane & 3;
    uint32_t bf[NN_KSTEPS][2];
#pragma unroll
    for (int s = 0; s < NN_KSTEPS; ++s) {
        bf[s][0] = frag[(s * 32 + lane) * 2 + 0];
        bf[s][1] = frag[(s * 32 + lane) * 2 + 1];
    }
    const float b0 = bias ? bias[2 * q] : 0.f, b1 = bias ? bias[2 * q + 1] : 0.f;
    // this lane's ldmatrix row: matrix mj = lane / 8 (cells +8 for odd mj, tap +1 for mj >= 2), row lane % 8
    const int mj = lane >> 3, mr = lane & 7, hi = mj >> 1;
    const int cx = (w & 1) * 16 + ((mj & 1) ? 8 : 0) + mr;          // tile-local output x of the row
    const int cy = w >> 1;
    const uint32_t ring_base = (uint32_t)__cvta_generic_to_shared(ring);
    const uint32_t cell0 = ring_base + (uint32_t)(((cy + 1) * NC_SX + cx + 1) * 16), zero_row = ring_base + NC_RING * NC_PL * 16;
    RingFill fill(tid, x0, y0, nx, ny);
#pragma unroll
    for (int t = -1; t <= 1; ++t) {
        fill.fetch(in, z0 + t, nz, plane);
        fill.put(ring, z0 + t, tid);
    }
    fill.fetch(in, z0 + 2, nz, plane);
    const int i0 = x0 + (w & 1) * 16 + g, j = y0 + cy;
    const bool on[2] = {i0 < nx && j < ny, i0 + 8 < nx && j < ny};
    long long c = i0 + (long long)nx * (j + (long long)ny * z0);
    for (int k = z0; k < z1; ++k, c += (long long)nx * ny) {
        // every warp is done with plane k - 2, planes up to k + 1 are there
        __syncthreads();
        if (k + 2 <= z1) {
            fill.put(ring, k + 2, tid);
            if (k + 3 <= z1) fill.fetch(in, k + 3, nz, plane);
        }
        uint32_t pb[3];                          // planes k - SGN, k, k + SGN: taps 0 .. 8, 9 .. 17, 18 .. 26
#pragma unroll
        for (int e = 0; e < 3; ++e) pb[e] = cell0 + (uint32_t)((k + SGN * (e - 1) + NC_RING) % NC_RING) * (NC_PL * 16);
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        __nv_bfloat162 mk[2] = {};
        if (MODE == 2) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (on[h]) mk[h] = *reinterpret_cast<const __nv_bfloat162*>(mask + (c + 8 * h) * NN_C + 2 * q);
        }
#pragma unroll
        for (int s = 0; s < NN_KSTEPS; ++s) {
            const int ta = 2 * s, tb = 2 * s + 1;                    // compile-time taps of the two halves
            const uint32_t aa = pb[ta / 9] + (uint32_t)(SGN * (((ta / 3) % 3 - 1) * NC_SX + ta % 3 - 1) * 16);
            const uint32_t ab = tb < NN_TAPS ? pb[tb < NN_TAPS ? tb / 9 : 0] + (uint32_t)(SGN * (((tb / 3) % 3 - 1) * NC_SX + tb % 3 - 1) * 16)
                                             : zero_row;
            uint32_t a[4];
            ldsm_x4(a, hi ? ab : aa);
            // ldmatrix returns the matrices in lane order: 0 cells 0-7 tap 2s, 1 cells 8-15 tap 2s,
            // 2 cells 0-7 tap 2s+1, 3 cells 8-15 tap 2s+1 -- the a0..a3 order of mma's A fragment
            mma_bf16(d, a, bf[s]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (!on[h]) continue;
            const long long ch = c + 8 * h;
            float v0 = d[2 * h] + b0, v1 = d[2 * h + 1] + b1;
            if (MODE == 0) {
                v0 = fmaxf(v0, 0.f);
                v1 = fmaxf(v1, 0.f);
                *reinterpret_cast<uint32_t*>(outb + ch * NN_C + 2 * q) = pack_bf16(v0, v1);
            } else if (MODE == 1) {
                if (q == 0) outf[ch] = v0;
            } else {
                if (!(__bfloat162float(mk[h].x) > 0.f)) v0 = 0.f;
                if (!(__bfloat162float(mk[h].y) > 0.f)) v1 = 0.f;
                *reinterpret_cast<uint32_t*>(outb + ch * NN_C + 2 * q) = pack_bf16(v0, v1);
            }
        }
    }
}

// Planes per block: the fewest plane steps over all rounds of `slots` resident blocks (a block of k planes takes
// about k + 2).
inline int conv_planes(int nx, int ny, int nz, long long slots) {
    const long long xy = (long long)((nx + NC_TX - 1) / NC_TX) * ((ny + NC_TY - 1) / NC_TY);
    long long best = -1;
    int kz = nz;
    for (int k = 4; k <= 128; ++k) {
        const long long n = xy * ((nz + k - 1) / k), cost = ((n + slots - 1) / slots) * (k + 2);
        if (best < 0 || cost < best) {
            best = cost;
            kz = k;
        }
        if (k >= nz) break;
    }
    return kz;
}

// Weight and bias gradients of one layer: dW[co][tap][ci] = sum_c dz[c][co] y[c + off(tap)][ci],
// db[co] = sum_c dz[c][co], as a GEMM on the tensor cores: M = 27 taps x 8 channels (padded to 28 taps;
// the padding tap reads a row of ones in channel 0, so its row is db), N = 8 output channels, K = the
// cells.  The tile, the ring and the warps' cells are those of the convolution above: per
// plane a warp takes 16 cells, one ldmatrix.x2.trans gives their dz as the B fragment, and per pair of taps
// one ldmatrix.x4.trans gathers y as the A fragment.  Each mma starts from zero and is added in FP32, so a
// sum is a chain of one FP32 addition per 16 cells.  Blocks walk tiles of a fixed grid and write one partial
// each.  Both operands are read once (16 + 16 bytes per cell, halo from L2).
// 128^3 cells: 62 us per layer, 98 with loads waited for; one thread per (tap, channel) with serial global loads
// took 2.8 ms.
#define WG_MINB 3
#define WG_BLOCKS (WG_MINB * IBM_NSM)       // resident at once
#define WG_STRIDE (NN_TAPS * NN_C * NN_C + NN_C)

__device__ __forceinline__ void ldsm_x4_t(uint32_t r[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2_t(uint32_t r[2], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}

__global__ void __launch_bounds__(256, WG_MINB) k_nn_wgrad(int nx, int ny, int nz, int kz, int ncout,
                                                  const __nv_bfloat16* __restrict__ dz,
                                                  const __nv_bfloat16* __restrict__ y, float* __restrict__ wpart) {
    __shared__ __align__(16) uint4 ring[NC_RING * NC_PL + 1];    // y planes as in the convolution, then the row of ones
    __shared__ __align__(16) uint4 zt[2][NC_TX * NC_TY];         // dz of the plane, double buffered
    __shared__ float red[NN_KSTEPS * 2 * NN_C * NN_C];           // [tap][ci][co]
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid == 0) ring[NC_RING * NC_PL] = make_uint4(0x3f80u, 0u, 0u, 0u);     // bf16 1 in channel 0
    for (int e = tid; e < NN_KSTEPS * 2 * NN_C * NN_C; e += 256) red[e] = 0.f;
    const int gx = (nx + NC_TX - 1) / NC_TX, gy = (ny + NC_TY - 1) / NC_TY, gz = (nz + kz - 1) / kz;
    const unsigned items = (unsigned)gx * gy * gz;
    const long long plane = (long long)nx * ny * NN_C;
    const int mj = lane >> 3, mr = lane & 7;
    // matrix mj of the x4 gather: tap 2s + (mj & 1), cells 8 (mj >> 1) .. + 7 of the warp's 16
    const int cx = (w & 1) * 16 + (mj >> 1) * 8 + mr, cy = w >> 1;
    const uint32_t ring_base = (uint32_t)__cvta_generic_to_shared(ring), ones = ring_base + NC_RING * NC_PL * 16;
    const uint32_t cell0 = (uint32_t)(((cy + 1) * NC_SX + cx + 1) * 16);
    const uint32_t zaddr = (uint32_t)__cvta_generic_to_shared(&zt[0][0]) +
                           (uint32_t)((cy * NC_TX + (w & 1) * 16 + (lane & 15)) * 16);
    float acc[NN_KSTEPS][4];
#pragma unroll
    for (int s = 0; s < NN_KSTEPS; ++s)
#pragma unroll
        for (int h = 0; h < 4; ++h) acc[s][h] = 0.f;
    for (unsigned it = blockIdx.x; it < items; it += gridDim.x) {
        const unsigned q = it / (unsigned)gx;
        const int x0 = (int)(it - q * gx) * NC_TX, y0 = (int)(q % (unsigned)gy) * NC_TY, z0 = (int)(q / (unsigned)gy) * kz;
        const int z1 = z0 + kz < nz ? z0 + kz : nz;
        RingFill fill(tid, x0, y0, nx, ny);
        const int zx = x0 + (tid & (NC_TX - 1)), zy = y0 + tid / NC_TX;
        const bool zin = tid < NC_TX * NC_TY && zx < nx && zy < ny;
        const __nv_bfloat16* zp = dz + (zx + (long long)nx * zy) * NN_C;
        uint4 zv;
        auto fetch_dz = [&](int k) {
            zv = make_uint4(0u, 0u, 0u, 0u);
            if (zin) zv = *reinterpret_cast<const uint4*>(zp + k * plane);
        };
        auto put_dz = [&](int k) {
            if (tid < NC_TX * NC_TY) zt[k & 1][tid] = zv;
        };
        __syncthreads();                        // the previous tile's reads are done
#pragma unroll
        for (int t = -1; t <= 1; ++t) {
            fill.fetch(y, z0 + t, nz, plane);
            fill.put(ring, z0 + t, tid);
        }
        fetch_dz(z0);
        put_dz(z0);
        fill.fetch(y, z0 + 2, nz, plane);
        if (z0 + 1 < z1) fetch_dz(z0 + 1);
        for (int k = z0; k < z1; ++k) {
            // every warp is done with plane k - 2 of y and k - 1 of dz; y up to k + 1 and dz of k are there
            __syncthreads();
            if (k + 2 <= z1) {
                fill.put(ring, k + 2, tid);
                if (k + 3 <= z1) fill.fetch(y, k + 3, nz, plane);
            }
            if (k + 1 < z1) {
                put_dz(k + 1);
                if (k + 2 < z1) fetch_dz(k + 2);
            }
            uint32_t b[2];
            ldsm_x2_t(b, zaddr + (uint32_t)(k & 1) * (NC_TX * NC_TY * 16));
            uint32_t pb[3];
#pragma unroll
            for (int e = 0; e < 3; ++e) pb[e] = cell0 + ring_base + (uint32_t)((k + e - 1 + NC_RING) % NC_RING) * (NC_PL * 16);
#pragma unroll
            for (int s = 0; s < NN_KSTEPS; ++s) {
                const int ta = 2 * s, tb = 2 * s + 1;                    // compile-time taps of the two halves
                const uint32_t aa = pb[ta / 9] + (uint32_t)((((ta / 3) % 3 - 1) * NC_SX + ta % 3 - 1) * 16);
                const uint32_t ab = tb < NN_TAPS ? pb[tb < NN_TAPS ? tb / 9 : 0] + (uint32_t)((((tb / 3) % 3 - 1) * NC_SX + tb % 3 - 1) * 16) : ones;
                uint32_t a[4];
                ldsm_x4_t(a, (mj & 1) ? ab : aa);
                float d[4] = {0.f, 0.f, 0.f, 0.f};
                mma_bf16(d, a, b);
#pragma unroll
                for (int h = 0; h < 4; ++h) acc[s][h] += d[h];
            }
        }
    }
    // the block's sum over its warps, in warp order
    const int g = lane >> 2, qq = lane & 3;
    for (int ww = 0; ww < 8; ++ww) {
        __syncthreads();
        if (w != ww) continue;
#pragma unroll
        for (int s = 0; s < NN_KSTEPS; ++s)
#pragma unroll
            for (int h = 0; h < 4; ++h)
                red[((2 * s + (h >> 1)) * NN_C + g) * NN_C + 2 * qq + (h & 1)] += acc[s][h];
    }
    __syncthreads();
    float* part = wpart + (long long)blockIdx.x * WG_STRIDE;
    for (int e = tid; e < NN_TAPS * NN_C * NN_C; e += 256) {
        const int co = e / (NN_TAPS * NN_C), tc = e - co * (NN_TAPS * NN_C);
        part[e] = co < ncout ? red[tc * NN_C + co] : 0.f;
    }
    if (tid < NN_C) part[NN_TAPS * NN_C * NN_C + tid] = tid < ncout ? red[NN_TAPS * NN_C * NN_C + tid] : 0.f;
}

// Sums the per-block partials; writes dW / db of the layer into grad (scaled by 1/N).  A block takes 32
// entries and splits the partials over 8 warps (coalesced rows), whose sums are added in warp order.
__global__ void __launch_bounds__(256) k_nn_wgrad_reduce(const float* __restrict__ wpart, int nblk, int ncout,
                                                         float inv_n, float* __restrict__ gw, float* __restrict__ gb) {
    __shared__ double sh[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (e < WG_STRIDE)
        for (int b = w; b < nblk; b += 8) s += wpart[(long long)b * WG_STRIDE + e];
    sh[w][lane] = s;
    __syncthreads();
    if (w != 0 || e >= WG_STRIDE) return;
    for (int q = 1; q < 8; ++q) s += sh[q][lane];
    if (e < NN_TAPS * NN_C * NN_C) {
        const int co = e / (NN_TAPS * NN_C);
        if (co < ncout) gw[e] = (float)(s * inv_n);
    } else {
        const int co = e - NN_TAPS * NN_C * NN_C;
        if (co < ncout) gb[co] = (float)(s * inv_n);
    }
}

// Packs the BF16 B fragments of m16n8k16 for one layer.  Forward: B[kk][n] = W[n][tap][ci] with
// kk = 8 tap + ci.  Input gradient: B[kk][n] = W[co][tap][n] with kk = 8 tap + co.
__global__ void k_nn_pack(const float* __restrict__ w, int ncout, uint32_t* __restrict__ ffwd, uint32_t* __restrict__ fbwd) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;   // (kstep, lane)
    if (idx >= NN_KSTEPS * 32) return;
    const int s = idx / 32, lane = idx % 32, g = lane >> 2, q = lane & 3;
    for (int r = 0; r < 2; ++r) {
        const int kk0 = 16 * s + 8 * r + 2 * q;     // rows kk0, kk0 + 1
        float f[2], bw[2];
        for (int e = 0; e < 2; ++e) {
            const int kk = kk0 + e, t = kk / NN_C, c = kk % NN_C;
            f[e] = (t < NN_TAPS && g < ncout) ? w[(g * NN_TAPS + t) * NN_C + c] : 0.f;
            bw[e] = (t < NN_TAPS && c < ncout) ? w[(c * NN_TAPS + t) * NN_C + g] : 0.f;
        }
        ffwd[idx * 2 + r] = pack_bf16(f[0], f[1]);
        fbwd[idx * 2 + r] = pack_bf16(bw[0], bw[1]);
    }
}

// Features of a snapshot: channel 0 = b dx^2 / s, 1 = (p - p_prev) / s, 2 = 1 on cells with a cut link;
// s = RMS of p - p_prev (or of b dx^2 when the pressure has not moved), read from scal[0].
__global__ void k_nn_features(long long N, const double* __restrict__ b, const double* __restrict__ p,
                              const double* __restrict__ pp, const uint8_t* __restrict__ flags, double dx2,
                              const double* __restrict__ scal, __nv_bfloat16* __restrict__ x) {
    const double inv = scal[0] > 0.0 ? 1.0 / scal[0] : 0.0;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const float f0 = (float)(b[c] * dx2 * inv), f1 = (float)((p[c] - pp[c]) * inv);
        const float f2 = (flags && (flags[c] & 63u)) ? 1.f : 0.f;
        uint4 v;
        v.x = pack_bf16(f0, f1);
        v.y = pack_bf16(f2, 0.f);
        v.z = 0u;
        v.w = 0u;
        *reinterpret_cast<uint4*>(x + c * NN_C) = v;
    }
}

// scal[0] = RMS of (p - p_prev), or of b dx^2 if that is zero.
__global__ void k_nn_scale(long long N, const double* __restrict__ b, const double* __restrict__ p,
                           const double* __restrict__ pp, double dx2, double* partials, unsigned* counter,
                           double* scal) {
    float a0 = 0.f, a1 = 0.f;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const float dp = (float)(p[c] - pp[c]);
        const float bb = (float)(b[c] * dx2);
        a0 += dp * dp;
        a1 += bb * bb;
    }
    double acc[2] = {(double)a0, (double)a1};
    grid_reduce<2>(acc, partials, counter, [&](double* t) {
        const double r0 = sqrt(t[0] / (double)N), r1 = sqrt(t[1] / (double)N);
        scal[0] = r0 > 0.0 ? r0 : (r1 > 0.0 ? r1 : 1.0);
    });
}

// Loss gradient seed: d3 channel 0 = 2 (out - target), others 0; the loss sum goes to scal[1].
__global__ void k_nn_loss(long long N, const float* __restrict__ out, const float* __restrict__ target,
                          __nv_bfloat16* __restrict__ d3, double* partials, unsigned* counter, double* scal) {
    float a = 0.f;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const float e = out[c] - target[c];
        a += e * e;
        uint4 v;
        v.x = pack_bf16(2.f * e, 0.f);
        v.y = v.z = v.w = 0u;
        *reinterpret_cast<uint4*>(d3 + c * NN_C) = v;
    }
    double acc[1] = {(double)a};
    grid_reduce<1>(acc, partials, counter, [&](double* t) { scal[1] = t[0]; });
}

__global__ void k_nn_adam(int n, float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                          float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const float gi = g[e];
        const float mi = b1 * m[e] + (1.f - b1) * gi;
        const float vi = b2 * v[e] + (1.f - b2) * gi * gi;
        m[e] = mi;
        v[e] = vi;
        p[e] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// x_guess = p + s * out
// Guess = linear extrapolation 2 p^n - p^{n-1} plus the network's scaled correction.
__global__ void k_nn_apply(long long N, const double* __restrict__ p, const double* __restrict__ pprev,
                           const float* __restrict__ out, const double* __restrict__ scal, double* __restrict__ xg) {
    const double s = scal[0];
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x)
        xg[c] = (2.0 * p[c] - pprev[c]) + s * (double)out[c];
}

unsigned blocks_n(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    long long cap = 8LL * IBM_NSM;
    if (b > cap) b = cap;
    return (unsigned)(b < 1 ? 1 : b);
}

long long offset_w(int l) { return l == 0 ? 0 : (l == 1 ? NN_C * NN_TAPS * NN_C : 2 * NN_C * NN_TAPS * NN_C); }
long long offset_b(int l) { return 2 * NN_C * NN_TAPS * NN_C + NN_TAPS * NN_C + l * NN_C; }
int cout_of(int l) { return l == 2 ? 1 : NN_C; }

// The training target of a snapshot, (p^{n+1} - 2 p^n + p^{n-1}) / s, formed in FP64 and stored in FP32.
__global__ void k_net_target(long long N, const double* __restrict__ pnext, const double* __restrict__ p,
                             const double* __restrict__ pprev, double s, float* __restrict__ out) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < N; q += (long long)gridDim.x * blockDim.x)
        out[q] = (float)((pnext[q] - 2.0 * p[q] + pprev[q]) / s);
}

}  // namespace

// ---- host side -----------------------------------------------------------------------------------

static int net_reserve(ibm_net* n, long long N) {
    if (N <= n->cap_cells) return IBM_OK;
    cudaFree(n->x0); cudaFree(n->y1); cudaFree(n->y2); cudaFree(n->d3); cudaFree(n->d2); cudaFree(n->d1);
    cudaFree(n->out); cudaFree(n->wpart);
    n->x0 = n->y1 = n->y2 = n->d3 = n->d2 = n->d1 = nullptr;
    n->out = n->wpart = nullptr;
    n->cap_cells = 0;
    const size_t act = (size_t)N * NN_C * sizeof(__nv_bfloat16);
    cudaError_t e;
    if ((e = ibm_malloc(&n->x0, act)) != cudaSuccess || (e = ibm_malloc(&n->y1, act)) != cudaSuccess ||
        (e = ibm_malloc(&n->y2, act)) != cudaSuccess || (e = ibm_malloc(&n->d3, act)) != cudaSuccess ||
        (e = ibm_malloc(&n->d2, act)) != cudaSuccess || (e = ibm_malloc(&n->d1, act)) != cudaSuccess ||
        (e = ibm_malloc(&n->out, (size_t)N * sizeof(float))) != cudaSuccess ||
        (e = ibm_malloc(&n->wpart, (size_t)WG_BLOCKS * WG_STRIDE * sizeof(float))) != cudaSuccess)
        return ibm_fail(IBM_E_NOMEM, "ibm_net: %s", cudaGetErrorString(e));
    n->cap_cells = N;
    return IBM_OK;
}

extern "C" void ibm_net_destroy(ibm_net* n) {
    if (!n) return;
    cudaFree(n->master); cudaFree(n->grad); cudaFree(n->m); cudaFree(n->v);
    for (int l = 0; l < 3; ++l) { cudaFree(n->frag_fwd[l]); cudaFree(n->frag_bwd[l]); }
    cudaFree(n->x0); cudaFree(n->y1); cudaFree(n->y2); cudaFree(n->d3); cudaFree(n->d2); cudaFree(n->d1);
    cudaFree(n->out); cudaFree(n->wpart); cudaFree(n->scal); cudaFree(n->partials); cudaFree(n->counter);
    free(n);
}

static int net_pack(ibm_net* n, cudaStream_t s) {
    for (int l = 0; l < 3; ++l)
        k_nn_pack<<<(NN_KSTEPS * 32 + 127) / 128, 128, 0, s>>>(n->master + offset_w(l), cout_of(l), n->frag_fwd[l],
                                                                n->frag_bwd[l]);
    IBM_LAUNCHED("ibm_net: pack");
    return IBM_OK;
}

extern "C" int ibm_net_create(const float* h_params, ibm_net** out) {
    if (!out) return ibm_fail(IBM_E_INVALID, "ibm_net_create: null output");
    *out = nullptr;
    ibm_net* n = (ibm_net*)calloc(1, sizeof(ibm_net));
    if (!n) return ibm_fail(IBM_E_NOMEM, "ibm_net_create: host allocation");
    cudaError_t e;
    const size_t pb = (NN_NPARAM + 16) * sizeof(float);   // padded: layer 3's bias is read as 8 lanes
    const size_t fb = NN_KSTEPS * 32 * 2 * sizeof(uint32_t);
    if ((e = ibm_malloc(&n->master, pb)) != cudaSuccess || (e = ibm_malloc(&n->grad, pb)) != cudaSuccess ||
        (e = ibm_malloc(&n->m, pb)) != cudaSuccess || (e = ibm_malloc(&n->v, pb)) != cudaSuccess ||
        (e = ibm_malloc(&n->scal, 8 * sizeof(double))) != cudaSuccess ||
        (e = ibm_malloc(&n->partials, 8 * 8 * IBM_NSM * sizeof(double) * 2)) != cudaSuccess ||
        (e = ibm_malloc(&n->counter, 4 * sizeof(unsigned))) != cudaSuccess) {
        ibm_net_destroy(n);
        return ibm_fail(IBM_E_NOMEM, "ibm_net_create: %s", cudaGetErrorString(e));
    }
    for (int l = 0; l < 3; ++l)
        if ((e = ibm_malloc(&n->frag_fwd[l], fb)) != cudaSuccess || (e = ibm_malloc(&n->frag_bwd[l], fb)) != cudaSuccess) {
            ibm_net_destroy(n);
            return ibm_fail(IBM_E_NOMEM, "ibm_net_create: %s", cudaGetErrorString(e));
        }
    if ((e = cudaMemset(n->m, 0, pb)) != cudaSuccess || (e = cudaMemset(n->v, 0, pb)) != cudaSuccess ||
        (e = cudaMemset(n->grad, 0, pb)) != cudaSuccess ||
        (e = cudaMemset(n->counter, 0, 4 * sizeof(unsigned))) != cudaSuccess ||
        (e = cudaMemset(n->scal, 0, 8 * sizeof(double))) != cudaSuccess ||
        (e = cudaMemset(n->master, 0, pb)) != cudaSuccess) {
        ibm_net_destroy(n);
        return ibm_cuda_check(e, "ibm_net_create");
    }
    if (h_params && (e = cudaMemcpy(n->master, h_params, NN_NPARAM * sizeof(float), cudaMemcpyHostToDevice)) != cudaSuccess) {
        ibm_net_destroy(n);
        return ibm_cuda_check(e, "ibm_net_create");
    }
    int rc = net_pack(n, 0);
    if (!rc && (e = cudaDeviceSynchronize()) != cudaSuccess) rc = ibm_cuda_check(e, "ibm_net_create");
    if (rc) {
        ibm_net_destroy(n);
        return rc;
    }
    *out = n;
    return IBM_OK;
}

extern "C" int ibm_net_num_params(void) { return NN_NPARAM; }

extern "C" int ibm_net_get_params(const ibm_net* n, float* h_params) {
    if (!n || !h_params) return ibm_fail(IBM_E_INVALID, "ibm_net_get_params: null argument");
    IBM_CUDA(cudaMemcpy(h_params, n->master, NN_NPARAM * sizeof(float), cudaMemcpyDeviceToHost));
    return IBM_OK;
}

extern "C" int ibm_net_get_grads(const ibm_net* n, float* h_grads) {
    if (!n || !h_grads) return ibm_fail(IBM_E_INVALID, "ibm_net_get_grads: null argument");
    IBM_CUDA(cudaMemcpy(h_grads, n->grad, NN_NPARAM * sizeof(float), cudaMemcpyDeviceToHost));
    return IBM_OK;
}

static void conv(const ibm_net* n, int nx, int ny, int nz, const __nv_bfloat16* in, int l, int sgn, int mode,
                 __nv_bfloat16* outb, float* outf, const __nv_bfloat16* mask, cudaStream_t s) {
    const int kz = conv_planes(nx, ny, nz, 4LL * IBM_NSM);
    const dim3 grid((unsigned)((nx + NC_TX - 1) / NC_TX), (unsigned)((ny + NC_TY - 1) / NC_TY), (unsigned)((nz + kz - 1) / kz));
    const uint32_t* frag = sgn > 0 ? n->frag_fwd[l] : n->frag_bwd[l];
    const float* bias = sgn > 0 ? n->master + offset_b(l) : nullptr;
    if (mode == 0) k_nn_conv_tile<1, 0><<<grid, 256, 0, s>>>(nx, ny, nz, kz, in, frag, bias, outb, outf, mask);
    else if (mode == 1) k_nn_conv_tile<1, 1><<<grid, 256, 0, s>>>(nx, ny, nz, kz, in, frag, bias, outb, outf, mask);
    else k_nn_conv_tile<-1, 2><<<grid, 256, 0, s>>>(nx, ny, nz, kz, in, frag, bias, outb, outf, mask);
}

static int net_forward(ibm_net* n, const ibm_grid* g, cudaStream_t s) {
    conv(n, g->nx, g->ny, g->nz, n->x0, 0, +1, 0, n->y1, nullptr, nullptr, s);
    conv(n, g->nx, g->ny, g->nz, n->y1, 1, +1, 0, n->y2, nullptr, nullptr, s);
    conv(n, g->nx, g->ny, g->nz, n->y2, 2, +1, 1, nullptr, n->out, nullptr, s);
    IBM_LAUNCHED("ibm_net: forward");
    return IBM_OK;
}

static int net_features(ibm_net* n, const ibm_grid* g, const double* b, const double* p, const double* pprev,
                        const uint8_t* flags, cudaStream_t s) {
    const long long N = (long long)g->nx * g->ny * g->nz;
    int rc = net_reserve(n, N);
    if (rc) return rc;
    const double dx2 = g->dx * g->dx;
    k_nn_scale<<<blocks_n(N, 256), 256, 0, s>>>(N, b, p, pprev, dx2, n->partials, n->counter, n->scal);
    k_nn_features<<<blocks_n(N, 256), 256, 0, s>>>(N, b, p, pprev, flags, dx2, n->scal, n->x0);
    IBM_LAUNCHED("ibm_net: features");
    return IBM_OK;
}

// Forward pass on a snapshot: d_out[N] (float) = the network's normalised pressure change; *scale
// (host, may be NULL, synchronises) = the normalisation s.
extern "C" int ibm_net_forward(ibm_net* n, const ibm_grid* g, const double* d_b, const double* d_p,
                               const double* d_pprev, const uint8_t* d_flags, float* d_out, double* scale,
                               void* stream) {
    int rc = ibm_check_grid(g);
    if (rc) return rc;
    if (!n || !d_b || !d_p || !d_pprev) return ibm_fail(IBM_E_INVALID, "ibm_net_forward: null argument");
    cudaStream_t s = (cudaStream_t)stream;
    if ((rc = net_features(n, g, d_b, d_p, d_pprev, d_flags, s))) return rc;
    if ((rc = net_forward(n, g, s))) return rc;
    const long long N = (long long)g->nx * g->ny * g->nz;
    if (d_out) IBM_CUDA(cudaMemcpyAsync(d_out, n->out, N * sizeof(float), cudaMemcpyDeviceToDevice, s));
    if (scale) {
        IBM_CUDA(cudaMemcpyAsync(scale, n->scal, sizeof(double), cudaMemcpyDeviceToHost, s));
        IBM_CUDA(cudaStreamSynchronize(s));
    }
    return IBM_OK;
}

// The training target of a snapshot: d_target[N] = (p_next - 2 p + p_prev) / s in FP32, s the scale that
// ibm_net_forward returned for (b, p, p_prev).
extern "C" int ibm_net_target(const ibm_grid* g, const double* d_pnext, const double* d_p, const double* d_pprev,
                              double s, float* d_target, void* stream) {
    int rc = ibm_check_grid(g);
    if (rc) return rc;
    if (!d_pnext || !d_p || !d_pprev || !d_target) return ibm_fail(IBM_E_INVALID, "ibm_net_target: null argument");
    if (!(s > 0.0) || !isfinite(s)) return ibm_fail(IBM_E_INVALID, "ibm_net_target: the scale must be positive");
    const long long N = (long long)g->nx * g->ny * g->nz;
    k_net_target<<<blocks_n(N, 256), 256, 0, (cudaStream_t)stream>>>(N, d_pnext, d_p, d_pprev, s, d_target);
    IBM_LAUNCHED("ibm_net: target");
    IBM_CUDA(cudaGetLastError());
    return IBM_OK;
}

// One training step on a snapshot: features from (b, p, p_prev, flags) against the target of
// ibm_net_target, forward, mean squared error, backward, Adam (lr; betas 0.9, 0.999).  *loss (host,
// synchronises) = the mean squared error before the update.  lr = 0 computes the gradients only.
extern "C" int ibm_net_train_step(ibm_net* n, const ibm_grid* g, const double* d_b, const double* d_p,
                                  const double* d_pprev, const uint8_t* d_flags, const float* d_target, float lr,
                                  double* loss, void* stream) {
    int rc = ibm_check_grid(g);
    if (rc) return rc;
    if (!n || !d_b || !d_p || !d_pprev || !d_target) return ibm_fail(IBM_E_INVALID, "ibm_net_train_step: null argument");
    cudaStream_t s = (cudaStream_t)stream;
    const long long N = (long long)g->nx * g->ny * g->nz;
    if ((rc = net_features(n, g, d_b, d_p, d_pprev, d_flags, s))) return rc;
    if ((rc = net_forward(n, g, s))) return rc;
    k_nn_loss<<<blocks_n(N, 256), 256, 0, s>>>(N, n->out, d_target, n->d3, n->partials, n->counter, n->scal);
    // input gradients (ReLU derivative of the layer below applied at the output cell)
    conv(n, g->nx, g->ny, g->nz, n->d3, 2, -1, 2, n->d2, nullptr, n->y2, s);
    conv(n, g->nx, g->ny, g->nz, n->d2, 1, -1, 2, n->d1, nullptr, n->y1, s);
    // weight gradients
    const int kz = conv_planes(g->nx, g->ny, g->nz, WG_BLOCKS);
    const long long tiles = (long long)((g->nx + NC_TX - 1) / NC_TX) * ((g->ny + NC_TY - 1) / NC_TY) * ((g->nz + kz - 1) / kz);
    const int nblk = (int)(tiles < WG_BLOCKS ? tiles : WG_BLOCKS);
    const __nv_bfloat16* dz[3] = {n->d1, n->d2, n->d3};
    const __nv_bfloat16* yin[3] = {n->x0, n->y1, n->y2};
    for (int l = 0; l < 3; ++l) {
        k_nn_wgrad<<<nblk, 256, 0, s>>>(g->nx, g->ny, g->nz, kz, cout_of(l), dz[l], yin[l], n->wpart);
        k_nn_wgrad_reduce<<<(WG_STRIDE + 31) / 32, 256, 0, s>>>(n->wpart, nblk, cout_of(l), 1.f / (float)N, n->grad + offset_w(l),
                                            n->grad + offset_b(l));
    }
    IBM_LAUNCHED("ibm_net: backward");
    if (lr > 0.f) {
        n->step += 1;
        const float c1 = 1.f - powf(0.9f, (float)n->step), c2 = 1.f - powf(0.999f, (float)n->step);
        k_nn_adam<<<(NN_NPARAM + 255) / 256, 256, 0, s>>>(NN_NPARAM, n->master, n->grad, n->m, n->v, lr, 0.9f, 0.999f,
                                                          1e-8f, c1, c2);
        if ((rc = net_pack(n, s))) return rc;
    }
    if (loss) {
        double h[2];
        IBM_CUDA(cudaMemcpyAsync(h, n->scal, 2 * sizeof(double), cudaMemcpyDeviceToHost, s));
        IBM_CUDA(cudaStreamSynchronize(s));
        *loss = h[1] / (double)N;
    }
    return IBM_OK;
}

// x_guess = p + s * net(b, p, p_prev, flags) on the state's grid (used by les_step).
int net_guess(ibm_net* n, const ibm_grid* g, const double* b, const double* p, const double* pprev,
              const uint8_t* flags, double* xg, cudaStream_t s) {
    int rc = net_features(n, g, b, p, pprev, flags, s);
    if (rc) return rc;
    if ((rc = net_forward(n, g, s))) return rc;
    const long long N = (long long)g->nx * g->ny * g->nz;
    k_nn_apply<<<blocks_n(N, 256), 256, 0, s>>>(N, p, pprev, n->out, n->scal, xg);
    IBM_LAUNCHED("ibm_net: guess");
    return IBM_OK;
}
