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
// takes 16 us (seven modules, l = 160 / 288) to 21 us (l = 544 to 2080, mean
// over the steps) and the levels up to 256 are inside it.  A refresh plus
// alignment of the 1024 / 2816 layer went from 10.33 to 4.71 ms, of the 4096 /
// 11008 layer from 68.0 to 39.8 ms.
#include <algorithm>
#include <cuda_runtime.h>

#include "internal.h"

namespace moara {

namespace {

constexpr int NB = kTriBase;          // 64
constexpr int LD = NB + 4;            // pitch of a k-major operand tile (16-byte rows, 2-way conflicts on the fill)
constexpr int LDW = 2 * NB + 4;       // pitch of a 128-wide one
constexpr int NT = 256;
constexpr int CHOL_SMEM = 2 * NB * LDW * sizeof(float);
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
    t.zero = (l + ZCOLS - 1) / ZCOLS;
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

// Factor F of the 64 x 64 block in tile (lower triangle; rows past nd hold the
// identity) and its inverse, by right-looking sub-panels of eight pivots.
// The block's 64 rows are followed by 64 identity rows: the same column
// operations turn those into F^-T.  Thread (w, lane) keeps rows
// 16 w + 4 (lane / 8) .. + 3 and columns 8 (lane % 8) .. + 7 of the 128 x 64
// array in registers.  Per sub-panel its eight columns go to shared memory,
// one thread per row forms the row's eight entries of the factor -- every
// thread repeats the 8 x 8 diagonal factor for itself, so that eight pivots
// need no exchange -- and all warps with live rows update the columns to the
// right.  Chain per pivot: one reciprocal square root, one multiplication,
// one FMA.
__device__ __forceinline__ void factor64(float (*tile)[LD], float* pin, float* pout, float* A, float* X, long long l,
                                         int nd, bool vec, int* fail) {
    constexpr int PP = 2 * NB + 4;                    // pitch of pout[c][row]
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const int tx = lane & 7, row0 = 16 * w + 4 * (lane >> 3);
    float a[4][8];
    if (w < 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 x = *reinterpret_cast<const float4*>(&tile[row0 + i][8 * tx]);
            const float4 y = *reinterpret_cast<const float4*>(&tile[row0 + i][8 * tx + 4]);
            a[i][0] = x.x; a[i][1] = x.y; a[i][2] = x.z; a[i][3] = x.w;
            a[i][4] = y.x; a[i][5] = y.y; a[i][6] = y.z; a[i][7] = y.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < 8; ++k) a[i][k] = (row0 - NB + i == 8 * tx + k) ? 1.0f : 0.0f;
    }
    bool bad = false;
#pragma unroll 1
    for (int c0 = 0; c0 < NB; c0 += SP) {
        if (8 * tx == c0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float4* p = reinterpret_cast<float4*>(pin + (row0 + i) * SP);
                p[0] = make_float4(a[i][0], a[i][1], a[i][2], a[i][3]);
                p[1] = make_float4(a[i][4], a[i][5], a[i][6], a[i][7]);
            }
        }
        __syncthreads();
        if (t < 2 * NB) {
            float v[SP];
            {
                const float4* p = reinterpret_cast<const float4*>(pin + t * SP);
                const float4 x = p[0], y = p[1];
                v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
            }
            float D[SP][SP];
#pragma unroll
            for (int i = 0; i < SP; ++i) {
                const float4* p = reinterpret_cast<const float4*>(pin + (c0 + i) * SP);
                const float4 x = p[0], y = p[1];
                D[i][0] = x.x; D[i][1] = x.y; D[i][2] = x.z; D[i][3] = x.w;
                D[i][4] = y.x; D[i][5] = y.y; D[i][6] = y.z; D[i][7] = y.w;
            }
#pragma unroll
            for (int j = 0; j < SP; ++j) {
                float d = D[j][j];
                if (!(d > 0.0f) || !isfinite(d)) {   // marks the failure; the module keeps its projector
                    d = 1.0f;
                    bad = true;
                }
                const float r = rsqrt_newton(d);
                v[j] *= r;
#pragma unroll
                for (int i = j + 1; i < SP; ++i) D[i][j] *= r;
#pragma unroll
                for (int k = j + 1; k < SP; ++k) {
                    v[k] = fmaf(-v[j], D[k][j], v[k]);
#pragma unroll
                    for (int i = k; i < SP; ++i) D[i][k] = fmaf(-D[i][j], D[k][j], D[i][k]);
                }
            }
            const int row = t & (NB - 1);
            if (t < NB) {
                // rows of the factor: zero above the diagonal
#pragma unroll
                for (int j = 0; j < SP; ++j) v[j] = c0 + j <= row ? v[j] : 0.0f;
                if (row < nd) {
                    float* dst = A + row * l + c0;
                    if (vec && c0 + SP <= nd) {
                        reinterpret_cast<float4*>(dst)[0] = make_float4(v[0], v[1], v[2], v[3]);
                        reinterpret_cast<float4*>(dst)[1] = make_float4(v[4], v[5], v[6], v[7]);
                    } else {
#pragma unroll
                        for (int j = 0; j < SP; ++j)
                            if (c0 + j < nd) dst[j] = v[j];
                    }
                }
            } else if (row < nd) {
                // F^-T: entry (row, c) is entry (c, row) of the inverse, zero for row > c
#pragma unroll
                for (int j = 0; j < SP; ++j)
                    if (c0 + j < nd) X[(c0 + j) * l + row] = v[j];
            }
#pragma unroll
            for (int j = 0; j < SP; ++j) pout[j * PP + t] = v[j];
        }
        __syncthreads();
        // rows past the sub-panel of the block, identity rows up to its end
        const bool live = w < 4 ? 16 * w + 15 >= c0 + SP : 16 * (w - 4) < c0 + SP;
        if (live && 8 * tx >= c0 + SP) {
#pragma unroll
            for (int j = 0; j < SP; ++j) {
                const float4 f = *reinterpret_cast<const float4*>(pout + j * PP + row0);
                const float4 x = *reinterpret_cast<const float4*>(pout + j * PP + 8 * tx);
                const float4 y = *reinterpret_cast<const float4*>(pout + j * PP + 8 * tx + 4);
                const float fv[4] = {f.x, f.y, f.z, f.w};
                const float kv[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int k = 0; k < 8; ++k) a[i][k] = fmaf(-fv[i], kv[k], a[i][k]);
            }
        }
    }
    if (t == 0 && bad) *fail = 1;
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
    float acc[8][8];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[p][q] = 0.0f;
#pragma unroll 4
    for (int k = 0; k < NB; ++k) {
        const float4 a0 = *reinterpret_cast<const float4*>(&As[k][4 * ty]);
        const float4 a1 = *reinterpret_cast<const float4*>(&As[k][NB + 4 * ty]);
        const float4 b0 = *reinterpret_cast<const float4*>(&Bs[k][4 * tx]);
        const float4 b1 = *reinterpret_cast<const float4*>(&Bs[k][NB + 4 * tx]);
        const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
            for (int q = 0; q < 8; ++q) acc[p][q] = fmaf(av[p], bv[q], acc[p][q]);
    }
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        const int i = (p >> 2) * NB + 4 * ty + (p & 3);
        if (i >= nr) continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = h * NB + 4 * tx;
            if (j >= nc || (skip && h == 0 && p < 4)) continue;
            const bool z = h == 0 ? zero0 : zero1;
            float* c = C + i * l + j;
            const float* x = &acc[p][4 * h];
            if (vec && j + 3 < nc) {
                const float4 o = z ? make_float4(0.0f, 0.0f, 0.0f, 0.0f) : *reinterpret_cast<const float4*>(c);
                *reinterpret_cast<float4*>(c) = make_float4(o.x - x[0], o.y - x[1], o.z - x[2], o.w - x[3]);
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (j + q < nc) c[q] = (z ? 0.0f : c[q]) - x[q];
            }
        }
    }
}

__global__ void __launch_bounds__(NT, 2) k_chol_step(const __grid_constant__ CholBatch b) {
    extern __shared__ __align__(16) float smem[];
    float (*const buf0)[LD] = reinterpret_cast<float (*)[LD]>(smem);
    float (*const buf1)[LD] = reinterpret_cast<float (*)[LD]>(smem + NB * LD);
    float (*const wide0)[LDW] = reinterpret_cast<float (*)[LDW]>(smem);
    float (*const wide1)[LDW] = reinterpret_cast<float (*)[LDW]>(smem + NB * LDW);
    __shared__ float red[NT / 32];
    const int s = b.step;
    if (static_cast<int>(blockIdx.x) < b.count) {
        // ------------------------------------------------ crit
        const CholItem& p = b.p[blockIdx.x];
        const int l = p.l, d = s + 1, nb = (l + NB - 1) / NB;
        if (d >= nb) return;
        const bool vec = (l & 3) == 0;
        const int nd = min(NB, l - d * NB);
        float* const A = p.A;
        float shift;
        Block r0, r1, r2;
        Acc tA, tD, acc, sq;
        tD.load(A + (long long)d * NB * l + d * NB, l, nd, nd, vec);
        sq.zero();
        if (s < 0) {
            float tr = 0.0f;
            for (int i = threadIdx.x; i < l; i += NT) tr += A[(long long)i * l + i];
            tr = block_sum_256(tr, red);
            shift = b.shift_rel * sqrtf(static_cast<float>(p.rows)) * tr;
            if (threadIdx.x == 0) *p.shift = shift;
        } else {
            shift = *p.shift;
            tA.load(A + (long long)d * NB * l + s * NB, l, nd, NB, vec);
            r2.load(p.X + (long long)s * NB * l + s * NB, l, NB, NB, vec);
            acc.zero();
            if (s >= 1) {
                r0.load(A + (long long)d * NB * l + (s - 1) * NB, l, nd, NB, vec);
                r1.load(A + (long long)s * NB * l + (s - 1) * NB, l, NB, NB, vec);
                r0.store_t(buf0);
                r1.store_t(buf1);
                __syncthreads();
                acc.mac(buf0, buf1);
                sq.mac(buf0, buf0);
                __syncthreads();
            }
            acc.sub_from(tA);
            acc.store_t(buf0);
            r2.store_t(buf1);
            __syncthreads();
            acc.zero();
            acc.mac(buf0, buf1);                      // L[d, s]
            acc.store(A + (long long)d * NB * l + s * NB, l, nd, NB, vec);
            __syncthreads();
            acc.store_t(buf0);
            __syncthreads();
            sq.mac(buf0, buf0);
        }
        sq.sub_from(tD);
        {
            const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
            if (ty == tx) {
#pragma unroll
                for (int a = 0; a < 4; ++a) sq.v[a][a] = 4 * ty + a < nd ? sq.v[a][a] + shift : 1.0f;
            }
        }
        __syncthreads();
        sq.store_n(buf1);
        __syncthreads();
        float* const pin = &buf0[0][0];               // 128 x 8, then 8 x 132
        factor64(buf1, pin, pin + 2 * NB * SP, A + (long long)d * NB * l + d * NB,
                 p.X + (long long)d * NB * l + d * NB, l, nd, vec, p.fail);
        return;
    }
    // locate (module, tile)
    const int tile = blockIdx.x - b.count;
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
    const cudaError_t ea = cudaFuncSetAttribute(k_chol_step, cudaFuncAttributeMaxDynamicSharedMemorySize, CHOL_SMEM);
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
        k_chol_step<<<b.count + total, NT, CHOL_SMEM, s>>>(b);
        ++*launches;
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace moara
