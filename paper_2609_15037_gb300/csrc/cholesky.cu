// Cholesky factorisation of the refresh's l x l Gram matrices together with
// the inverse of the factor's diagonal superblocks, for every module of a
// group, one launch per 64 columns.
//
// Launch `step` = s (s = -1 .. nb - 1, nb = ceil(l / 64)) holds, for each
// module, tiles (64 x 64; bulk and ibulk 128 x 128) that depend on earlier
// launches only:
//
//   crit    L[d, s], then the factor of the diagonal block d = s + 1 and its
//           inverse: the chain that the next launch waits for
//   slab    L[i, s] = (A[i, s] - L[i, s-1] L[s, s-1]^T) Linv[s, s]^T, i > d
//   bulk    A[i, t] -= L[i, s-1] L[t, s-1]^T for i >= t > s: the update by the
//           previous column block, one launch behind (so that it runs beside
//           the chain instead of in it)
//   islab   Linv[s, c] = Linv[s, s] (U[s, c] - L[s, s-1] Linv[s-1, c])
//   ibulk   U[t, c] -= L[t, s-1] Linv[s-1, c], t > s (U grows in Linv's place)
//   zero    the rest of Linv's row block s
//
// islab and ibulk stay within superblocks of kTriSuper blocks (2304 columns,
// the whole of every sketch up to r = 2272); the levels of the inverse past
// that are products of their own.  All sums are fp32 FMAs.
//
// What bounds it is the chain, one CTA per module and step: two 64-deep
// products, then 64 pivots one after the other.  With a factor kernel that
// spent two barriers per pivot (43 us a launch), a panel solve (11 us) and a
// trailing update (14 us) as launches of their own, a 64-column step took
// 68 us, and the inverse's levels up to 256 another 36 us each; here a step
// takes 14 us (seven modules, l = 160 / 288) to 21 us (l = 544 to 2080, mean
// over the steps; up to 33 us where the updates of seven modules fill the GPU
// more than once) and the whole inverse is inside it.  The first form of this
// kernel took a refresh plus alignment of the 1024 / 2816 layer from 10.33 to
// 4.71 ms, of the 4096 / 11008 layer from 68.0 to 39.8 ms.
#include <algorithm>
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "launch.cuh"

namespace moara {

namespace {

constexpr int NB = kTriBase;          // 64
constexpr int LD = NB + 4;            // pitch of a k-major operand tile (16-byte rows, 2-way conflicts on the fill)
constexpr int LDW = 2 * NB + 4;       // pitch of a 128-wide one
constexpr int NT = 256;
constexpr int kCritCtas = 4;          // CTAs of the chain per module (a cluster)
constexpr int kCritModules = 38;      // modules up to which they fit beside each other, one per SM
constexpr int CHOL_SMEM = 5 * NB * LD * sizeof(float);
static_assert(5 * LD >= 2 * LDW, "two 128-wide operand tiles fit the chain's five buffers");
// A launch of at most two CTAs per SM whose chain runs on clusters asks for so
// much shared memory that a CTA has its SM to itself: an update tile beside the
// chain slows every link of it (refresh and alignment of a 1024 / 2816 layer
// 3.04 -> 2.79 ms, of a 4096 / 11008 layer 22.6 -> 21.6).  Larger launches are
// bound by their tiles and lose by it: the refresh of five 4096 / 11008 layers
// 72.1 -> 79.4 ms with every launch so, 71.9 with this line; lines of 228, 400
// and 500 CTAs give the same within 1%.
constexpr int kAloneCtas = 304;
constexpr int CHOL_SMEM_ALONE = 120 * 1024;
constexpr int SP = 8;                 // pivots per sub-panel of the diagonal block

// Tile counts of one module at step s; the same on the host and the device.
struct CholTiles {
    int slab, islab, bulk, ibulk, zero;
    __host__ __device__ int total() const { return slab + islab + bulk + ibulk + zero; }
};

__host__ __device__ inline int imin(int a, int b) { return a < b ? a : b; }
__host__ __device__ inline int imax(int a, int b) { return a > b ? a : b; }

constexpr int ZCOLS = 512;            // columns a zero tile clears

__host__ __device__ inline CholTiles chol_tiles(int l, int s) {
    CholTiles t{0, 0, 0, 0, 0};
    const int nb = (l + NB - 1) / NB;
    if (s < 0 || s >= nb) return t;
    t.slab = imax(0, nb - (s + 2));
    t.islab = s - s / kTriSuper * kTriSuper;
    // nothing to clear in the last row block of a matrix of one superblock
    t.zero = s == nb - 1 && s < kTriSuper ? 0 : (l + ZCOLS - 1) / ZCOLS;
    if (s >= 1) {
        const int q = (nb - (s + 1) + 1) / 2;          // pairs of blocks from s + 1 on
        t.bulk = q > 0 ? q * (q + 1) / 2 : 0;
        const int b1 = (s - 1) / kTriSuper * kTriSuper;
        t.ibulk = (imax(0, imin(b1 + kTriSuper, nb) - (s + 1)) + 1) / 2 * ((s - b1 + 1) / 2);
    }
    return t;
}

// A 64 x 64 block of a row-major matrix of pitch l, rows and columns past
// (nr, nc) zero.  Thread t holds row t / 4, columns 16 kk + 4 (t % 4) .. + 3.
struct Block {
    float4 v[4];
    __device__ __forceinline__ void load(const float* src, long long l, int nr, int nc, bool vec) {
        const int i = threadIdx.x >> 2, k0 = (threadIdx.x & 3) * 4;
        if (vec && nr >= NB && nc >= NB) {            // the same for every thread: four loads, no branches
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) v[kk] = *reinterpret_cast<const float4*>(src + i * l + kk * 16 + k0);
            return;
        }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            const int k = kk * 16 + k0;
            const float* p = src + i * l + k;
            if (vec && i < nr && k + 3 < nc) {
                v[kk] = *reinterpret_cast<const float4*>(p);
            } else {
                v[kk].x = (i < nr && k < nc) ? p[0] : 0.0f;
                v[kk].y = (i < nr && k + 1 < nc) ? p[1] : 0.0f;
                v[kk].z = (i < nr && k + 2 < nc) ? p[2] : 0.0f;
                v[kk].w = (i < nr && k + 3 < nc) ? p[3] : 0.0f;
            }
        }
    }
    // k-major: dst[k][i] = block[i][k]
    __device__ __forceinline__ void store_t(float (*dst)[LD]) const {
        const int i = threadIdx.x >> 2, k0 = (threadIdx.x & 3) * 4;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            const int k = kk * 16 + k0;
            dst[k][i] = v[kk].x;
            dst[k + 1][i] = v[kk].y;
            dst[k + 2][i] = v[kk].z;
            dst[k + 3][i] = v[kk].w;
        }
    }
    // the same into a tile of 128 columns, from column off on
    __device__ __forceinline__ void store_t(float (*dst)[LDW], int off) const {
        const int i = (threadIdx.x >> 2) + off, k0 = (threadIdx.x & 3) * 4;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            const int k = kk * 16 + k0;
            dst[k][i] = v[kk].x;
            dst[k + 1][i] = v[kk].y;
            dst[k + 2][i] = v[kk].z;
            dst[k + 3][i] = v[kk].w;
        }
    }
    __device__ __forceinline__ void store_n(float (*dst)[LDW], int off) const {
        const int i = threadIdx.x >> 2, k0 = (threadIdx.x & 3) * 4 + off;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) *reinterpret_cast<float4*>(&dst[i][kk * 16 + k0]) = v[kk];
    }
    // as stored: dst[i][k]
    __device__ __forceinline__ void store_n(float (*dst)[LD]) const {
        const int i = threadIdx.x >> 2, k0 = (threadIdx.x & 3) * 4;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) *reinterpret_cast<float4*>(&dst[i][kk * 16 + k0]) = v[kk];
    }
};

// Output tile: thread (ty, tx) = (t / 16, t % 16) holds rows 4 ty .. + 3 and
// columns 4 tx .. + 3.
struct Acc {
    float v[4][4];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) v[a][b] = 0.0f;
    }
    // += A B with A[k][i], B[k][j]
    __device__ __forceinline__ void mac(const float (*A)[LD], const float (*B)[LD]) {
        const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll 8
        for (int k = 0; k < NB; ++k) {
            const float4 a = *reinterpret_cast<const float4*>(&A[k][4 * ty]);
            const float4 b = *reinterpret_cast<const float4*>(&B[k][4 * tx]);
            const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) v[p][q] = fmaf(av[p], bv[q], v[p][q]);
        }
    }
    __device__ __forceinline__ void load(const float* src, long long l, int nr, int nc, bool vec) {
        const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = 4 * ty + a, j = 4 * tx;
            const float* p = src + i * l + j;
            if (vec && i < nr && j + 3 < nc) {
                const float4 x = *reinterpret_cast<const float4*>(p);
                v[a][0] = x.x; v[a][1] = x.y; v[a][2] = x.z; v[a][3] = x.w;
            } else {
#pragma unroll
                for (int b = 0; b < 4; ++b) v[a][b] = (i < nr && j + b < nc) ? p[b] : 0.0f;
            }
        }
    }
    __device__ __forceinline__ void store(float* dst, long long l, int nr, int nc, bool vec) const {
        const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = 4 * ty + a, j = 4 * tx;
            float* p = dst + i * l + j;
            if (vec && i < nr && j + 3 < nc) {
                *reinterpret_cast<float4*>(p) = make_float4(v[a][0], v[a][1], v[a][2], v[a][3]);
            } else {
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (i < nr && j + b < nc) p[b] = v[a][b];
            }
        }
    }
    // v = c - v
    __device__ __forceinline__ void sub_from(const Acc& c) {
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) v[a][b] = c.v[a][b] - v[a][b];
    }
    // as a k-major A operand whose k is this tile's column: dst[j][i]
    __device__ __forceinline__ void store_t(float (*dst)[LD]) const {
        const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            *reinterpret_cast<float4*>(&dst[4 * tx + b][4 * ty]) = make_float4(v[0][b], v[1][b], v[2][b], v[3][b]);
    }
    // row-major: dst[i][j] (a k-major B operand whose k is this tile's row)
    __device__ __forceinline__ void store_n(float (*dst)[LD]) const {
        const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
        for (int a = 0; a < 4; ++a)
            *reinterpret_cast<float4*>(&dst[4 * ty + a][4 * tx]) = make_float4(v[a][0], v[a][1], v[a][2], v[a][3]);
    }
};

// 1 / sqrt(d) to about fp32 rounding: CUDA's rsqrtf and one step of Newton's
// iteration on 1 / r^2 = d.
__device__ __forceinline__ float rsqrt_newton(float d) {
    const float r = rsqrtf(d);
    const float e = fmaf(-d * r, r, 1.0f);
    return fmaf(0.5f * r, e, r);
}

// 1 / d for a normal d (rcp.approx and one step of Newton's iteration on
// 1 / r = d).
__device__ __forceinline__ float rcp_newton(float d) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return fmaf(r, fmaf(-d, r, 1.0f), r);
}

__device__ __forceinline__ void bar(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ void get8(float (&x)[8], const float* p) {
    const float4 u = reinterpret_cast<const float4*>(p)[0], v = reinterpret_cast<const float4*>(p)[1];
    x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w; x[4] = v.x; x[5] = v.y; x[6] = v.z; x[7] = v.w;
}

__device__ __forceinline__ void put8(float* p, const float (&x)[8]) {
    reinterpret_cast<float4*>(p)[0] = make_float4(x[0], x[1], x[2], x[3]);
    reinterpret_cast<float4*>(p)[1] = make_float4(x[4], x[5], x[6], x[7]);
}

// Factor F of the 64 x 64 block in tile (lower triangle; rows past nd hold the
// identity) and its inverse, by sub-panels of eight pivots.
//
// Warps 0 and 1, one thread per row, run the chain: a thread keeps its row's
// eight entries of the sub-panel, repeats the 8 x 8 diagonal factor for itself
// (so that eight pivots need no exchange; as L D L^T, one reciprocal, one
// multiplication and one FMA deep per pivot, scaled by 1 / sqrt(D) at the end)
// and brings its entries of the next sub-panel up to date.  Warps 4 - 7 keep
// the block (4 x 8 entries a thread), apply the sub-panel to the columns after
// the next one meanwhile and write it out.  Warps 2 and 3 follow one sub-panel
// behind with the inverse: row r of F^-T = I F^-T, a dot product with the
// finished columns of F per entry.  With 128 rows (the block's and the
// identity's) and the whole update in the chain a block took 16,000 clocks,
// here 13,200: a sub-panel's 1,430 are 520 for its eight pivots, 470 for the
// next sub-panel's columns (shared-memory broadcasts), the rest exchange.
// (Chain and inverse on one warp each, two rows a lane: 14,800.)
//
// The block comes scaled by sigma = 2^(-2h), near unit diagonal, so that the
// reciprocals stay in range; F and its inverse are written times 2^h and 2^-h.
constexpr int PIN = SP * SP;                          // floats of scratch: the sub-panel's diagonal rows,
static_assert(PIN + 2 * NB * SP <= NB * LD, "the factor's scratch fits one tile");   // and two of the next columns

__device__ __forceinline__ void factor64(const float (*tile)[LD], float* scratch, float (*F)[LD], float (*Z)[LD],
                                         float* A, float* X, long long l, int nd, bool vec, float up, float down,
                                         int* fail) {
    float* const pin = scratch;
    float* const nbuf = scratch + PIN;                // [2][row][8]
    const int t = threadIdx.x;
    if (t < NB) {
        float v[SP];
        get8(v, &tile[t][0]);
        bool bad = false;
#pragma unroll 1
        for (int c0 = 0; c0 < NB; c0 += SP) {
            if (t >= c0 && t < c0 + SP) put8(pin + (t - c0) * SP, v);
            bar(1, NB);
            float D[SP][SP], rs[SP];
#pragma unroll
            for (int i = 0; i < SP; ++i) {            // its lower triangle
                const float4 u = *reinterpret_cast<const float4*>(pin + i * SP);
                D[i][0] = u.x; D[i][1] = u.y; D[i][2] = u.z; D[i][3] = u.w;
                if (i >= 4) {
                    const float4 y = *reinterpret_cast<const float4*>(pin + i * SP + 4);
                    D[i][4] = y.x; D[i][5] = y.y; D[i][6] = y.z; D[i][7] = y.w;
                }
            }
#pragma unroll
            for (int j = 0; j < SP; ++j) {
                float d = D[j][j];
                // a pivot that is not a positive normal number marks the
                // failure; the module keeps its projector
                const bool ok = d >= 1.17549435e-38f && d <= 3.402823466e38f;
                bad = bad || !ok;
                d = ok ? d : 1.0f;
                const float rd = rcp_newton(d);
                rs[j] = rsqrt_newton(d);
                const float qv = v[j] * rd;
#pragma unroll
                for (int k = j + 1; k < SP; ++k) {
                    const float q = D[k][j] * rd;
#pragma unroll
                    for (int i = k; i < SP; ++i) D[i][k] = fmaf(-D[i][j], q, D[i][k]);
                    v[k] = fmaf(-qv, D[k][j], v[k]);
                }
            }
#pragma unroll
            for (int j = 0; j < SP; ++j) {
                v[j] = c0 + j <= t ? v[j] * rs[j] : 0.0f;             // zero above the diagonal
                F[c0 + j][t] = v[j];
            }
            if (t == 0) {
#pragma unroll
                for (int j = 0; j < SP; ++j) F[c0 + j][NB] = rs[j];   // 1 / F[j][j], in the pitch's padding
            }
            bar(2, NT);
            if (c0 + SP < NB) {
                float n[SP];
                get8(n, nbuf + ((c0 / SP) & 1) * NB * SP + t * SP);
#pragma unroll
                for (int j = 0; j < SP; ++j) {
                    float f[SP];
                    get8(f, &F[c0 + j][c0 + SP]);
#pragma unroll
                    for (int k = 0; k < SP; ++k) n[k] = fmaf(-v[j], f[k], n[k]);
                }
#pragma unroll
                for (int k = 0; k < SP; ++k) v[k] = n[k];
            }
        }
        if (t == 0 && bad) *fail = 1;
    } else if (t < 2 * NB) {
        // row r of F^-T: z[c] = (e_r[c] - sum_{k < c} z[k] F[c][k]) / F[c][c]
        const int r = t - NB;
#pragma unroll 1
        for (int c0 = 0; c0 < NB; c0 += SP) {
            bar(2, NT);
            float z[SP];
#pragma unroll
            for (int j = 0; j < SP; ++j) z[j] = r == c0 + j ? 1.0f : 0.0f;
            // z of the second warp's rows begins with 32 zeros
#pragma unroll 8
            for (int k = r & 32; k < c0; ++k) {
                const float x = Z[k][r];
                float f[SP];
                get8(f, &F[k][c0]);
#pragma unroll
                for (int j = 0; j < SP; ++j) z[j] = fmaf(-x, f[j], z[j]);
            }
#pragma unroll
            for (int j = 0; j < SP; ++j) {
                float f[SP];
                get8(f, &F[c0 + j][c0]);
                z[j] *= F[c0 + j][NB];
#pragma unroll
                for (int k = j + 1; k < SP; ++k) z[k] = fmaf(-z[j], f[k], z[k]);
                Z[c0 + j][r] = z[j];
            }
            // entry (r, c) of F^-T is entry (c, r) of the inverse, zero for r > c
            if (r < nd) {
#pragma unroll
                for (int j = 0; j < SP; ++j)
                    if (c0 + j < nd) X[(c0 + j) * l + r] = z[j] * down;
            }
        }
    } else {
        const int tx = t & 7, row0 = 4 * ((t - 2 * NB) >> 3);
        float a[4][SP];
#pragma unroll
        for (int i = 0; i < 4; ++i) get8(a[i], &tile[row0 + i][SP * tx]);
        if (tx == 1) {
#pragma unroll
            for (int i = 0; i < 4; ++i) put8(nbuf + (row0 + i) * SP, a[i]);
        }
#pragma unroll 1
        for (int c0 = 0; c0 < NB; c0 += SP) {
            bar(2, NT);
            if (row0 + 3 >= c0 + SP && SP * tx >= c0 + 2 * SP) {
#pragma unroll 4
                for (int j = 0; j < SP; ++j) {
                    const float4 f = *reinterpret_cast<const float4*>(&F[c0 + j][row0]);
                    const float fv[4] = {f.x, f.y, f.z, f.w};
                    float k8[SP];
                    get8(k8, &F[c0 + j][SP * tx]);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int k = 0; k < SP; ++k) a[i][k] = fmaf(-fv[i], k8[k], a[i][k]);
                }
            }
            if (SP * tx == c0 + 2 * SP) {
                float* const nb = nbuf + ((c0 / SP + 1) & 1) * NB * SP;
#pragma unroll
                for (int i = 0; i < 4; ++i) put8(nb + (row0 + i) * SP, a[i]);
            }
            // the sub-panel's columns of the factor: two threads a row
            const int row = (t - 2 * NB) >> 1, h = 4 * (t & 1);
            if (row < nd) {
                float* dst = A + row * l + c0 + h;
                float v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) v[j] = F[c0 + h + j][row] * up;
                if (vec && c0 + h + 3 < nd) {
                    *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (c0 + h + j < nd) dst[j] = v[j];
                }
            }
        }
    }
}

__device__ __forceinline__ float block_sum_256(float v, float* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.0f;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) t += red[w];
    return t;
}

// (row, column) of entry e of a lower triangle stored row by row.
__device__ __forceinline__ void tri_index(int e, int& i, int& j) {
    i = static_cast<int>((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
    while (i * (i + 1) / 2 > e) --i;
    while ((i + 1) * (i + 2) / 2 <= e) ++i;
    j = e - i * (i + 1) / 2;
}

// C (128 x 128 at row i0, column j0 of C, of which nr x nc exist) -= A B from
// k-major tiles, in four 64 x 64 quadrants: thread (ty, tx) holds rows
// 4 ty .. + 3 and columns 4 tx .. + 3 of each.  zero[h]: column half h starts
// from zero instead of C; quadrant (0, 0) is left alone when skip.
__device__ __forceinline__ void wide_update(const float (*As)[LDW], const float (*Bs)[LDW], float* C, long long l,
                                            int nr, int nc, bool vec, bool zero0, bool zero1, bool skip) {
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    // Two columns per packed FMA (each rounded by itself): half the FMA
    // instructions to issue beside the shared-memory loads (refresh and alignment
    // of a 4096 / 11008 layer 21.7 -> 21.3 ms; five layers' refresh 72.1 -> 71.3).
    unsigned long long acc2[8][4];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc2[p][q] = 0ull;
#pragma unroll 4
    for (int k = 0; k < NB; ++k) {
        const float4 a0 = *reinterpret_cast<const float4*>(&As[k][4 * ty]);
        const float4 a1 = *reinterpret_cast<const float4*>(&As[k][NB + 4 * ty]);
        const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&Bs[k][4 * tx]);
        const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&Bs[k][NB + 4 * tx]);
        const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const unsigned long long bv[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            unsigned long long aa;
            asm("mov.b64 %0, {%1, %1};" : "=l"(aa) : "f"(av[p]));
#pragma unroll
            for (int q = 0; q < 4; ++q) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc2[p][q]) : "l"(aa), "l"(bv[q]));
        }
    }
    float acc[8][8];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[p][2 * q]), "=f"(acc[p][2 * q + 1]) : "l"(acc2[p][q]));
    // A column half's entries of C are all fetched before the first is stored:
    // read and written one after the other, sixteen L2 latencies stood in a row
    // and a step with l = 2080 alone took 24 us instead of 16, with the seven
    // modules of a 4096 / 11008 layer up to 43 instead of 32 (its refresh and
    // alignment 24.4 ms instead of 22.4).
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = h * NB + 4 * tx;
        if (j >= nc) continue;
        const bool z = h == 0 ? zero0 : zero1;
        const int i0 = 4 * ty, li = static_cast<int>(l);
        float* const c = C + (i0 * li + j);
        auto at = [&](int p) { return ((p >> 2) * NB + (p & 3)) * li; };
        auto mine = [&](int p) { return i0 + (p >> 2) * NB + (p & 3) < nr && !(skip && h == 0 && p < 4); };
        if (vec && j + 3 < nc) {
            float4 o[8];
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                o[p] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (!z && mine(p)) o[p] = *reinterpret_cast<const float4*>(c + at(p));
            }
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const float* x = &acc[p][4 * h];
                if (mine(p))
                    *reinterpret_cast<float4*>(c + at(p)) =
                        make_float4(o[p].x - x[0], o[p].y - x[1], o[p].z - x[2], o[p].w - x[3]);
            }
        } else {
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                if (!mine(p)) continue;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (j + q < nc) c[at(p) + q] = (z ? 0.0f : c[at(p) + q]) - acc[p][4 * h + q];
            }
        }
    }
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__global__ void __launch_bounds__(NT, 2) k_chol_step(const __grid_constant__ CholBatch b) {
    pdl_begin();
    extern __shared__ __align__(16) float smem[];
    float (*const buf0)[LD] = reinterpret_cast<float (*)[LD]>(smem);
    float (*const buf1)[LD] = reinterpret_cast<float (*)[LD]>(smem + NB * LD);
    float (*const wide0)[LDW] = reinterpret_cast<float (*)[LDW]>(smem);
    float (*const wide1)[LDW] = reinterpret_cast<float (*)[LDW]>(smem + NB * LDW);
    __shared__ float red[NT / 32];
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int s = b.step, C = static_cast<int>(cl.num_blocks());
    if (static_cast<int>(blockIdx.x) < C * b.count) {
        // ------------------------------------------------ crit
        // The cluster's C CTAs (kCritCtas, or one where the group has enough
        // modules to fill the GPU) share the products by rows of the block, 16
        // at a time, the K range split over four groups of 64 threads; the
        // factor is the first one's.  One CTA alone takes 2,700 to 3,700 clocks
        // for each of the four 64-deep products, bound by its shared-memory
        // reads; four CTAs 11,300 clocks from launch to factor instead of
        // 19,500, but 224 modules' refresh 526 ms instead of 509.
        const CholItem& p = b.p[blockIdx.x / C];
        const int l = p.l, d = s + 1, nb = (l + NB - 1) / NB;
        if (d >= nb) return;                          // the whole cluster
        const int rank = static_cast<int>(cl.block_rank());
        if (s < 0 && rank != 0) return;
        const bool vec = (l & 3) == 0;
        const int nd = min(NB, l - d * NB);
        float* const A = p.A;
        float (*const bufF)[LD] = reinterpret_cast<float (*)[LD]>(smem);                  // L[d, s-1]; F
        float (*const bufT)[LD] = reinterpret_cast<float (*)[LD]>(smem + NB * LD);        // L[s, s-1]; the block
        float (*const bufI)[LD] = reinterpret_cast<float (*)[LD]>(smem + 2 * NB * LD);    // Linv[s, s]; scratch
        float (*const part)[LD] = reinterpret_cast<float (*)[LD]>(smem + 3 * NB * LD);    // four 16-row partial tiles; Z
        float (*const bufG)[LD] = reinterpret_cast<float (*)[LD]>(smem + 4 * NB * LD);    // X, then L[d, s]
        const int t = threadIdx.x;
        int half;
        if (s < 0) {
            float tr = 0.0f;
            for (int i = t; i < l; i += NT) tr += A[(long long)i * l + i];
            tr = block_sum_256(tr, red);
            const float shift = b.shift_rel * sqrtf(static_cast<float>(p.rows)) * tr;
            // h: half the exponent of the mean diagonal entry (0 where it has none)
            const float mean = tr / static_cast<float>(l);
            half = (mean > 0.0f && isfinite(mean)) ? max(-60, ilogbf(mean) / 2) : 0;
            if (t == 0) {
                p.shift[0] = shift;
                p.shift[1] = static_cast<float>(half);
            }
            const float sigma = exp2f(static_cast<float>(-2 * half));
            Acc D;
            D.load(A, l, nd, nd, vec);
            const int ty = t >> 4, tx = t & 15;
            if (ty == tx) {
#pragma unroll
                for (int a = 0; a < 4; ++a) D.v[a][a] += shift;
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    D.v[a][c] = 4 * ty + a < nd ? D.v[a][c] * sigma : (4 * ty + a == 4 * tx + c ? 1.0f : 0.0f);
            D.store_n(bufT);
            __syncthreads();
        } else {
            cluster_arrive();                         // waited for before the first access to a peer
            // this thread's four entries of a group of 16 rows from r0 on
            const int lr = t >> 4, j0 = 4 * (t & 15);
            auto entry4 = [&](const float* src, int row, int nc) {
                float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                const float* q = src + (long long)row * l + j0;
                if (row < nd) {
                    if (vec && j0 + 3 < nc) return *reinterpret_cast<const float4*>(q);
                    if (j0 < nc) x.x = q[0];
                    if (j0 + 1 < nc) x.y = q[1];
                    if (j0 + 2 < nc) x.z = q[2];
                    if (j0 + 3 < nc) x.w = q[3];
                }
                return x;
            };
            Block q0, q1, q2;
            if (s >= 1) {
                q0.load(A + (long long)d * NB * l + (s - 1) * NB, l, nd, NB, vec);
                q1.load(A + (long long)s * NB * l + (s - 1) * NB, l, NB, NB, vec);
            }
            q2.load(p.X + (long long)s * NB * l + s * NB, l, NB, NB, vec);
            float* const Ads = A + (long long)d * NB * l + s * NB;
            const float* const Add = A + (long long)d * NB * l + d * NB;
            float4 tA = entry4(Ads, 16 * rank + lr, NB), tD = entry4(Add, 16 * rank + lr, nd);
            const float shift = p.shift[0];
            half = static_cast<int>(p.shift[1]);
            const float sigma = exp2f(static_cast<float>(-2 * half));
            // thread (g, ty, tx): rows 4 ty .. + 3 of the 16, columns tx + 16 j,
            // k in 16 g .. + 15; acc += a b^T from row-major tiles
            const int g = t >> 6, ty = (t >> 4) & 3, tx = t & 15;
            auto mac16 = [&](float (&acc)[4][4], const float (*a)[LD], int ar, const float (*bb)[LD]) {
#pragma unroll
                for (int k = 16 * g; k < 16 * g + 16; k += 4) {
                    float4 x[4], y[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        x[i] = *reinterpret_cast<const float4*>(&a[ar + 4 * ty + i][k]);
                        y[i] = *reinterpret_cast<const float4*>(&bb[tx + 16 * i][k]);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            acc[i][j] = fmaf(x[i].x, y[j].x, acc[i][j]);
                            acc[i][j] = fmaf(x[i].y, y[j].y, acc[i][j]);
                            acc[i][j] = fmaf(x[i].z, y[j].z, acc[i][j]);
                            acc[i][j] = fmaf(x[i].w, y[j].w, acc[i][j]);
                        }
                }
            };
            // sum of the four groups' partial tiles: this thread's four entries
            auto reduce = [&](const float (&acc)[4][4]) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) part[16 * g + 4 * ty + i][tx + 16 * j] = acc[i][j];
                __syncthreads();
                float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 x = *reinterpret_cast<const float4*>(&part[16 * q + (t >> 4)][j0]);
                    v = make_float4(v.x + x.x, v.y + x.y, v.z + x.z, v.w + x.w);
                }
                return v;
            };
            if (s >= 1) {
                q0.store_n(bufF);
                q1.store_n(bufT);
            }
            q2.store_n(bufI);
            __syncthreads();
            for (int r0 = 16 * rank; r0 < NB; r0 += 16 * C) {
                const int row = r0 + lr;
                if (r0 != 16 * rank) tA = entry4(Ads, row, NB);
                float4 x = tA;
                if (s >= 1) {
                    float acc[4][4] = {};
                    mac16(acc, bufF, r0, bufT);
                    const float4 u = reduce(acc);
                    x = make_float4(tA.x - u.x, tA.y - u.y, tA.z - u.z, tA.w - u.w);
                }
                *reinterpret_cast<float4*>(&bufG[row][j0]) = x;       // X
                __syncthreads();
                float acc[4][4] = {};
                mac16(acc, bufG, r0, bufI);
                x = reduce(acc);                      // L[d, s]; its barrier: every thread is done with these rows of X
                if (row < nd) {
                    float* q = Ads + (long long)row * l + j0;
                    if (vec) *reinterpret_cast<float4*>(q) = x;
                    else { q[0] = x.x; q[1] = x.y; q[2] = x.z; q[3] = x.w; }
                }
                if (r0 == 16 * rank) cluster_wait();
                for (int q = 0; q < C; ++q)           // to every CTA
                    *reinterpret_cast<float4*>(cl.map_shared_rank(&bufG[0][0], q) + row * LD + j0) = x;
                __syncthreads();
            }
            cl.sync();
            for (int r0 = 16 * rank; r0 < NB; r0 += 16 * C) {
                const int row = r0 + lr;
                if (r0 != 16 * rank) tD = entry4(Add, row, nd);
                float acc[4][4] = {};
                if (s >= 1) mac16(acc, bufF, r0, bufF);
                mac16(acc, bufG, r0, bufG);
                const float4 u = reduce(acc);
                float e[4] = {tD.x - u.x, tD.y - u.y, tD.z - u.z, tD.w - u.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const bool dia = j0 + k == row;
                    e[k] = row < nd ? (e[k] + (dia ? shift : 0.0f)) * sigma : (dia ? 1.0f : 0.0f);
                }
                // the first CTA is past its products with bufT (the cluster barrier)
                *reinterpret_cast<float4*>(cl.map_shared_rank(&bufT[0][0], 0) + row * LD + j0) =
                    make_float4(e[0], e[1], e[2], e[3]);
                __syncthreads();
            }
            cl.sync();
            if (rank != 0) return;
        }
        factor64(bufT, &bufI[0][0], bufF, part, A + (long long)d * NB * l + d * NB,
                 p.X + (long long)d * NB * l + d * NB, l, nd, vec, exp2f(static_cast<float>(half)),
                 exp2f(static_cast<float>(-half)), p.fail);
        return;
    }
    // locate (module, tile)
    const int tile = blockIdx.x - C * b.count;
    if (tile >= b.tile_start[b.count]) return;        // the last cluster's padding
    int lo = 0, hi = b.count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (b.tile_start[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    const CholItem& p = b.p[lo];
    const int l = p.l, nb = (l + NB - 1) / NB;
    const CholTiles n = chol_tiles(l, s);
    int e = tile - b.tile_start[lo];
    const bool vec = (l & 3) == 0;
    float* const A = p.A;
    float* const X = p.X;
    auto at = [&](float* m, int i, int j) { return m + (long long)i * NB * l + j * NB; };
    auto rows = [&](int i) { return min(NB, l - i * NB); };
    Block r0, r1, r2;
    Acc c, acc;
    acc.zero();
    if (e < n.slab) {
        const int i = s + 2 + e;
        c.load(at(A, i, s), l, rows(i), NB, vec);
        r2.load(at(X, s, s), l, NB, NB, vec);
        if (s >= 1) {
            r0.load(at(A, i, s - 1), l, rows(i), NB, vec);
            r1.load(at(A, s, s - 1), l, NB, NB, vec);
            r0.store_t(buf0);
            r1.store_t(buf1);
            __syncthreads();
            acc.mac(buf0, buf1);
            __syncthreads();
        }
        acc.sub_from(c);
        acc.store_t(buf0);
        r2.store_t(buf1);
        __syncthreads();
        acc.zero();
        acc.mac(buf0, buf1);
        acc.store(at(A, i, s), l, rows(i), NB, vec);
        return;
    }
    e -= n.slab;
    if (e < n.islab) {
        const int cb = s / kTriSuper * kTriSuper + e;
        r0.load(at(A, s, s - 1), l, rows(s), NB, vec);
        r1.load(at(X, s - 1, cb), l, NB, NB, vec);
        r2.load(at(X, s, s), l, rows(s), rows(s), vec);
        if (cb < s - 1) c.load(at(X, s, cb), l, rows(s), NB, vec);
        else c.zero();
        r0.store_t(buf0);
        r1.store_n(buf1);
        __syncthreads();
        acc.mac(buf0, buf1);
        acc.sub_from(c);
        __syncthreads();
        r2.store_t(buf0);
        acc.store_n(buf1);
        __syncthreads();
        acc.zero();
        acc.mac(buf0, buf1);
        acc.store(at(X, s, cb), l, rows(s), NB, vec);
        return;
    }
    e -= n.islab;
    if (e < n.bulk) {
        // pairs of row blocks and of column blocks from s + 1 on; of the first
        // the chain has block (s + 1, s + 1)
        int i, t;
        tri_index(e, i, t);
        i = s + 1 + 2 * i;
        t = s + 1 + 2 * t;
        const int nr = min(2 * NB, l - i * NB), nc = min(2 * NB, l - t * NB);
        Block q0, q1;
        r0.load(at(A, i, s - 1), l, nr, NB, vec);
        r1.load(at(A, i + 1, s - 1), l, nr - NB, NB, vec);
        q0.load(at(A, t, s - 1), l, nc, NB, vec);
        q1.load(at(A, t + 1, s - 1), l, nc - NB, NB, vec);
        r0.store_t(wide0, 0);
        r1.store_t(wide0, NB);
        q0.store_t(wide1, 0);
        q1.store_t(wide1, NB);
        __syncthreads();
        wide_update(wide0, wide1, at(A, i, t), l, nr, nc, vec, false, false, e == 0);
        return;
    }
    e -= n.bulk;
    if (e < n.ibulk) {
        const int b1 = (s - 1) / kTriSuper * kTriSuper, w = (s - b1 + 1) / 2;
        const int t = s + 1 + e / w * 2, cb = b1 + e % w * 2;
        const int tend = min(b1 + kTriSuper, nb);
        const int nr = min(min(2, tend - t) * NB, l - t * NB), nc = min(2, s - cb) * NB;
        Block q0, q1;
        r0.load(at(A, t, s - 1), l, nr, NB, vec);
        r1.load(at(A, t + 1, s - 1), l, nr - NB, NB, vec);
        q0.load(at(X, s - 1, cb), l, NB, NB, vec);
        q1.load(at(X, s - 1, cb + 1), l, nc > NB ? NB : 0, NB, vec);
        r0.store_t(wide0, 0);
        r1.store_t(wide0, NB);
        q0.store_n(wide1, 0);
        q1.store_n(wide1, NB);
        __syncthreads();
        // column block s - 1 is touched for the first time
        wide_update(wide0, wide1, at(X, t, cb), l, nr, nc, vec, cb == s - 1, cb + 1 == s - 1, false);
        return;
    }
    e -= n.ibulk;
    // zero: Linv's row block s outside its superblock's part up to the diagonal
    const int z0 = s / kTriSuper * kTriSuper * NB, z1 = min(l, (s + 1) * NB);
    const int nr = rows(s);
    for (int k = threadIdx.x; k < nr * ZCOLS; k += NT) {
        const int i = k / ZCOLS, j = e * ZCOLS + k % ZCOLS;
        if (j < l && (j < z0 || j >= z1)) X[((long long)s * NB + i) * l + j] = 0.0f;
    }
}

}  // namespace

cudaError_t launch_cholesky(CholBatch& b, cudaStream_t s, int64_t* launches) {
    if (b.count <= 0) return cudaSuccess;
    const cudaError_t ea = cudaFuncSetAttribute(k_chol_step, cudaFuncAttributeMaxDynamicSharedMemorySize, CHOL_SMEM_ALONE);
    if (ea != cudaSuccess) return ea;
    int nbmax = 0;
    for (int i = 0; i < b.count; ++i) nbmax = std::max(nbmax, (b.p[i].l + NB - 1) / NB);
    for (int step = -1; step < nbmax; ++step) {
        int total = 0;
        for (int i = 0; i < b.count; ++i) {
            b.tile_start[i] = total;
            total += chol_tiles(b.p[i].l, step).total();
        }
        b.tile_start[b.count] = total;
        b.step = step;
        if (total == 0 && step == nbmax - 1) break;           // no module has anything left
        const int C = b.count <= kCritModules ? kCritCtas : 1;
        const int ctas = C * b.count + (total + C - 1) / C * C;
        ++*launches;
        const cudaError_t e = launch(k_chol_step, dim3(ctas), NT, C > 1 && ctas <= kAloneCtas ? CHOL_SMEM_ALONE : CHOL_SMEM,
                                     s, C, b);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace moara
