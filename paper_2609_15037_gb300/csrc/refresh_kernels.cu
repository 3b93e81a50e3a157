// Small dense kernels of the projector refresh (TruncatedSVD of Algorithm 1
// computed by randomized subspace iteration): the Gaussian test matrix, plane
// splits and transposes, the ordering of Ritz vectors, and the final sign
// convention.  The problems of a group run side by side in one launch.
#include <algorithm>
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "internal.h"
#include "launch.cuh"
#include "ritz.h"

namespace moara {

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, "Parallel random numbers: as easy
// as 1, 2, 3", SC'11): 10 rounds of the 4x32 S-box with the published
// multipliers and Weyl key increments.  Box-Muller turns pairs of uniforms
// into standard normals.
// ---------------------------------------------------------------------------
struct U4 { uint32_t x, y, z, w; };

__device__ __forceinline__ U4 philox4x32_10(U4 c, uint32_t k0, uint32_t k1) {
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
    const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
        const uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
        U4 n;
        n.x = hi1 ^ c.y ^ k0;
        n.y = lo1;
        n.z = hi0 ^ c.w ^ k1;
        n.w = lo0;
        c = n;
        k0 += W0;
        k1 += W1;
    }
    return c;
}

// uniform in (0, 1]: (x + 1) * 2^-32 with x the top 24 bits scaled
__device__ __forceinline__ float u01(uint32_t x) {
    return (static_cast<float>(x >> 8) + 1.0f) * (1.0f / 16777216.0f);
}

__global__ void k_philox_gaussian(const __grid_constant__ SmallBatch b) {
    pdl_begin();
    const int pi = blockIdx.y;
    float* out = b.a[pi];
    uint16_t* hout = b.h[pi];
    const long long count = (long long)b.rows[pi] * b.l[pi];
    const uint32_t k0 = static_cast<uint32_t>(b.key[pi]);
    const uint32_t k1 = static_cast<uint32_t>(b.key[pi] >> 32);
    const long long groups = (count + 3) / 4;
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < groups;
         g += (long long)gridDim.x * blockDim.x) {
        U4 c{static_cast<uint32_t>(g), static_cast<uint32_t>(g >> 32), 0x4D6F4152u, 0x52616E64u};
        const U4 r = philox4x32_10(c, k0, k1);
        const float u1 = u01(r.x), u2 = u01(r.y), u3 = u01(r.z), u4 = u01(r.w);
        const float ra = sqrtf(-2.0f * logf(u1)), rb = sqrtf(-2.0f * logf(u3));
        float s2, c2, s4, c4;
        sincospif(2.0f * u2, &s2, &c2);
        sincospif(2.0f * u4, &s4, &c4);
        const float z[4] = {ra * c2, ra * s2, rb * c4, rb * s4};
        const long long base = g * 4;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (base + q >= count) continue;
            if (hout != nullptr) {
                const __nv_bfloat16 h = __float2bfloat16_rn(z[q]);
                hout[base + q] = *reinterpret_cast<const uint16_t*>(&h);
            } else {
                out[base + q] = z[q];
            }
        }
    }
}

cudaError_t launch_philox_gaussian(const SmallBatch& b, cudaStream_t s, int64_t* launches) {
    if (b.count <= 0) return cudaSuccess;
    // as many blocks per item as the largest needs at four groups a thread
    long long most = 1;
    for (int q = 0; q < b.count; ++q) most = std::max(most, ((long long)b.rows[q] * b.l[q] + 4095) / 4096);
    dim3 grid(static_cast<unsigned>(std::min(2048LL, most)), b.count);
    ++*launches;
    return launch(k_philox_gaussian, grid, 256, 0, s, 1, b);
}

// c <- a and h <- a rounded to bf16 (rows x l entries each).
__global__ void __launch_bounds__(256) k_copy_bf16(const __grid_constant__ SmallBatch b) {
    pdl_begin();
    const int pi = blockIdx.y;
    const float* src = b.a[pi];
    float* dst = b.c[pi];
    uint16_t* hd = b.h[pi];
    const long long count = (long long)b.rows[pi] * b.l[pi];
    const long long quads = count / 4;               // the buffers are 16-byte aligned
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < quads;
         g += (long long)gridDim.x * blockDim.x) {
        const float4 v = reinterpret_cast<const float4*>(src)[g];
        reinterpret_cast<float4*>(dst)[g] = v;
        const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
        reinterpret_cast<uint2*>(hd)[g] =
            make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    }
    if (blockIdx.x == 0 && threadIdx.x < count - 4 * quads) {
        const long long e = 4 * quads + threadIdx.x;
        dst[e] = src[e];
        const __nv_bfloat16 h = __float2bfloat16_rn(src[e]);
        hd[e] = *reinterpret_cast<const uint16_t*>(&h);
    }
}

cudaError_t launch_copy_bf16(const SmallBatch& b, cudaStream_t s, int64_t* launches) {
    if (b.count <= 0) return cudaSuccess;
    long long most = 1;
    for (int q = 0; q < b.count; ++q) most = std::max(most, ((long long)b.rows[q] * b.l[q] + 4095) / 4096);
    ++*launches;
    return launch(k_copy_bf16, dim3(static_cast<unsigned>(std::min(2048LL, most)), b.count), 256, 0, s, 1, b);
}

constexpr int kSmallThreads = 1024;

__device__ float block_sum(float v, float* red) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    float t = 0.0f;
    if (w == 0) {
        t = (lane < static_cast<int>(blockDim.x >> 5)) ? red[lane] : 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) red[32] = t;
    }
    __syncthreads();
    return red[32];
}

// ---------------------------------------------------------------------------
// h <- a^T rounded to bf16 (l x l): 32 x 32 tiles through shared memory.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_transpose_bf16(const __grid_constant__ SmallBatch b) {
    pdl_begin();
    __shared__ float t[32][33];
    const int pi = blockIdx.z;
    const int l = b.l[pi];
    const float* src = b.a[pi];
    uint16_t* dst = b.h[pi];
    const int tiles = (l + 31) / 32;
    for (int tile = blockIdx.x; tile < tiles * tiles; tile += gridDim.x) {
        const int ti = tile / tiles, tj = tile - ti * tiles;
        const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
        for (int r = ty; r < 32; r += 8) {
            const int i = ti * 32 + r, j = tj * 32 + tx;
            t[r][tx] = (i < l && j < l) ? src[(long long)i * l + j] : 0.0f;
        }
        __syncthreads();
        for (int r = ty; r < 32; r += 8) {
            const int i = tj * 32 + r, j = ti * 32 + tx;   // dst row i = src column
            if (i < l && j < l) {
                __nv_bfloat16 h = __float2bfloat16_rn(t[tx][r]);
                dst[(long long)i * l + j] = *reinterpret_cast<uint16_t*>(&h);
            }
        }
        __syncthreads();
    }
}

cudaError_t launch_transpose_bf16(const SmallBatch& b, cudaStream_t s, int64_t* launches) {
    if (b.count <= 0) return cudaSuccess;
    int lmax = 1;
    for (int q = 0; q < b.count; ++q) lmax = std::max(lmax, b.l[q]);
    const int tiles = (lmax + 31) / 32;
    ++*launches;
    return launch(k_transpose_bf16, dim3(std::min(1024, tiles * tiles), 1, b.count), 256, 0, s, 1, b);
}

// ---------------------------------------------------------------------------
// Three bf16 planes of an fp32 matrix (rows x l, row-major, row pitch ld or
// l): hi = bf16(x), mid = bf16(x - hi), lo = bf16(x - hi - mid), so
// hi + mid + lo carries 24 significant bits.  With `transpose` the planes hold the l x rows transpose.
// Planes are consecutive at h, each rows * l elements.  Bound by HBM / L2
// bytes (4 read, 6 written per entry): 64 x 64 tiles, 16-byte loads and
// stores, through shared memory for the transpose (as 32 x 32 tiles with
// 4-byte stores on a 256-CTA grid per matrix, 45 M entries took 167 us, now
// 63 us = 7.1 TB/s); 32 x 32 tiles where a pitch or an address is not a
// multiple of 16 bytes.
// ---------------------------------------------------------------------------
// the three bf16 parts of eight values, as 16-byte units
__device__ __forceinline__ void split8(const float (&x)[8], uint4 (&p)[3]) {
    uint32_t w[3][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float a = x[2 * k], b = x[2 * k + 1];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
            w[q][k] = *reinterpret_cast<const uint32_t*>(&h);
            a -= __low2float(h);
            b -= __high2float(h);
        }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) p[q] = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
}

// Whether both kernels' 16-byte accesses are aligned for item pi.
__device__ __forceinline__ bool split_wide(const SmallBatch& b, int pi) {
    const int lds = b.ld[pi] > 0 ? b.ld[pi] : b.l[pi];
    return ((b.rows[pi] | b.l[pi]) & 7) == 0 && (lds & 3) == 0 &&
           ((reinterpret_cast<uintptr_t>(b.a[pi]) | reinterpret_cast<uintptr_t>(b.h[pi])) & 15) == 0;
}

__global__ void __launch_bounds__(256) k_split3_wide(const __grid_constant__ SmallBatch b, int transpose) {
    pdl_begin();
    __shared__ float t[64][65];
    const int pi = blockIdx.z;
    if (!split_wide(b, pi)) return;
    const int rows = b.rows[pi], cols = b.l[pi];
    const long long lds = b.ld[pi] > 0 ? b.ld[pi] : cols;
    const float* src = b.a[pi];
    uint16_t* dst = b.h[pi];
    const long long plane = (long long)rows * cols;
    const int tr = (rows + 63) / 64, tc = (cols + 63) / 64;
    const int tid = threadIdx.x;
    for (int tile = blockIdx.x; tile < tr * tc; tile += gridDim.x) {
        const int i0 = tile / tc * 64, j0 = (tile - tile / tc * tc) * 64;
        if (!transpose) {
            // thread: rows tid / 8 and 32 further, eight columns
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int i = i0 + (tid >> 3) + 32 * u, j = j0 + 8 * (tid & 7);
                if (i >= rows || j >= cols) continue;
                const float4* s4 = reinterpret_cast<const float4*>(src + i * lds + j);
                const float4 v = s4[0], w = s4[1];
                const float x[8] = {v.x, v.y, v.z, v.w, w.x, w.y, w.z, w.w};
                uint4 p[3];
                split8(x, p);
#pragma unroll
                for (int q = 0; q < 3; ++q) *reinterpret_cast<uint4*>(dst + q * plane + (long long)i * cols + j) = p[q];
            }
            continue;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = (tid >> 4) + 16 * u, c = 4 * (tid & 15);
            float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (i0 + r < rows && j0 + c < cols) v = *reinterpret_cast<const float4*>(src + (i0 + r) * lds + j0 + c);
            t[r][c] = v.x; t[r][c + 1] = v.y; t[r][c + 2] = v.z; t[r][c + 3] = v.w;
        }
        __syncthreads();
        // output row j0 + (tid / 8) and 32 further, eight columns of it
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int c = (tid >> 3) + 32 * u, r = 8 * (tid & 7);
            if (j0 + c < cols && i0 + r < rows) {
                float x[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) x[k] = t[r + k][c];
                uint4 p[3];
                split8(x, p);
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    *reinterpret_cast<uint4*>(dst + q * plane + (long long)(j0 + c) * rows + i0 + r) = p[q];
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(256) k_split3(const __grid_constant__ SmallBatch b, int transpose) {
    pdl_begin();
    __shared__ float t[32][33];
    const int pi = blockIdx.z;
    if (split_wide(b, pi)) return;
    const int rows = b.rows[pi], cols = b.l[pi];
    const long long lds = b.ld[pi] > 0 ? b.ld[pi] : cols;
    const float* src = b.a[pi];
    uint16_t* dst = b.h[pi];
    const long long plane = (long long)rows * cols;
    const int tr = (rows + 31) / 32, tc = (cols + 31) / 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    // stores: thread (ty2, tx2) writes output rows ty2 and ty2 + 16 of the
    // tile, columns 2 tx2 and 2 tx2 + 1, as 4-byte pairs where aligned
    const int tx2 = threadIdx.x & 15, ty2 = threadIdx.x >> 4;
    const int orows = transpose ? cols : rows, ocols = transpose ? rows : cols;
    for (int tile = blockIdx.x; tile < tr * tc; tile += gridDim.x) {
        const int ti = tile / tc, tj = tile - ti * tc;
        for (int r = ty; r < 32; r += 8) {
            const int i = ti * 32 + r, j = tj * 32 + tx;
            t[r][tx] = (i < rows && j < cols) ? src[(long long)i * lds + j] : 0.0f;
        }
        __syncthreads();
        for (int rr = ty2; rr < 32; rr += 16) {
            const int i = (transpose ? tj : ti) * 32 + rr;          // output row
            const int j = (transpose ? ti : tj) * 32 + 2 * tx2;     // output column of the pair
            if (i < orows && j < ocols) {
                const float x0 = transpose ? t[2 * tx2][rr] : t[rr][2 * tx2];
                const float x1 = transpose ? t[2 * tx2 + 1][rr] : t[rr][2 * tx2 + 1];
                uint16_t h[3], g[3];
                {
                    const __nv_bfloat16 a0 = __float2bfloat16_rn(x0);
                    const float r0 = x0 - __bfloat162float(a0);
                    const __nv_bfloat16 a1 = __float2bfloat16_rn(r0);
                    const __nv_bfloat16 a2 = __float2bfloat16_rn(r0 - __bfloat162float(a1));
                    h[0] = *reinterpret_cast<const uint16_t*>(&a0);
                    h[1] = *reinterpret_cast<const uint16_t*>(&a1);
                    h[2] = *reinterpret_cast<const uint16_t*>(&a2);
                }
                {
                    const __nv_bfloat16 a0 = __float2bfloat16_rn(x1);
                    const float r0 = x1 - __bfloat162float(a0);
                    const __nv_bfloat16 a1 = __float2bfloat16_rn(r0);
                    const __nv_bfloat16 a2 = __float2bfloat16_rn(r0 - __bfloat162float(a1));
                    g[0] = *reinterpret_cast<const uint16_t*>(&a0);
                    g[1] = *reinterpret_cast<const uint16_t*>(&a1);
                    g[2] = *reinterpret_cast<const uint16_t*>(&a2);
                }
                const long long o = (long long)i * ocols + j;
                if (j + 1 < ocols && ((o | plane) & 1) == 0 && (reinterpret_cast<uintptr_t>(dst) & 3) == 0) {
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        *reinterpret_cast<uint32_t*>(dst + q * plane + o) =
                            static_cast<uint32_t>(h[q]) | (static_cast<uint32_t>(g[q]) << 16);
                } else {
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        dst[q * plane + o] = h[q];
                        if (j + 1 < ocols) dst[q * plane + o + 1] = g[q];
                    }
                }
            }
        }
        __syncthreads();
    }
}

cudaError_t launch_split3(const SmallBatch& b, int transpose, cudaStream_t s, int64_t* launches) {
    if (b.count <= 0) return cudaSuccess;
    // as many blocks per item as the largest item has tiles
    long long wide = 0, narrow = 0;
    for (int q = 0; q < b.count; ++q) {
        const int lds = b.ld[q] > 0 ? b.ld[q] : b.l[q];
        if (((b.rows[q] | b.l[q]) & 7) == 0 && (lds & 3) == 0 &&
            ((reinterpret_cast<uintptr_t>(b.a[q]) | reinterpret_cast<uintptr_t>(b.h[q])) & 15) == 0)
            wide = std::max(wide, (long long)((b.rows[q] + 63) / 64) * ((b.l[q] + 63) / 64));
        else
            narrow = std::max(narrow, (long long)((b.rows[q] + 31) / 32) * ((b.l[q] + 31) / 32));
    }
    cudaError_t e = cudaSuccess;
    if (wide > 0) {
        e = launch(k_split3_wide, dim3(static_cast<unsigned>(std::min(2048LL, wide)), 1, b.count), 256, 0, s, 1, b, transpose);
        ++*launches;
    }
    if (narrow > 0 && e == cudaSuccess) {
        e = launch(k_split3, dim3(static_cast<unsigned>(std::min(256LL, narrow)), 1, b.count), 256, 0, s, 1, b, transpose);
        ++*launches;
    }
    return e;
}

// ---------------------------------------------------------------------------
// a <- I (l x l)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_set_identity(const __grid_constant__ SmallBatch b) {
    pdl_begin();
    const int pi = blockIdx.y;
    const int l = b.l[pi];
    for (int i = blockIdx.x; i < l; i += gridDim.x) {
        float* row = b.a[pi] + (long long)i * l;
        for (int c = threadIdx.x; c < l; c += blockDim.x) row[c] = (i == c) ? 1.0f : 0.0f;
    }
}

cudaError_t launch_set_identity(const SmallBatch& b, cudaStream_t s, int64_t* launches) {
    if (b.count <= 0) return cudaSuccess;
    int lmax = 1;
    for (int q = 0; q < b.count; ++q) lmax = std::max(lmax, b.l[q]);
    ++*launches;
    return launch(k_set_identity, dim3(std::min(1024, lmax), b.count), 256, 0, s, 1, b);
}

// ---------------------------------------------------------------------------
// Ritz values d_j = x_j^T (C x_j) / x_j^T x_j from X (a) and W = C X (b) into
// c: a CTA per 32 columns, lane = column, its 32 warps split the rows.  (With
// one CTA per module for values and order, l = 2080 took 2.9 ms; now the two
// launches together take 0.05 ms.)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kSmallThreads) k_ritz_values(const __grid_constant__ SmallBatch b) {
    pdl_begin();
    __shared__ float s_acc[32][33], s_nrm[32][33];
    const int pi = blockIdx.y;
    const int l = b.l[pi];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j0 = blockIdx.x * 32, j = j0 + lane;
    if (j0 >= l) return;
    const float* X = b.a[pi];
    const float* W = b.b[pi];
    float acc = 0.0f, nrm = 0.0f;
    if (j < l) {
#pragma unroll 4
        for (int i = warp; i < l; i += 32) {
            const float x = X[(long long)i * l + j];
            acc = fmaf(x, W[(long long)i * l + j], acc);
            nrm = fmaf(x, x, nrm);
        }
    }
    s_acc[warp][lane] = acc;
    s_nrm[warp][lane] = nrm;
    __syncthreads();
    // warp w reduces column j0 + w
    acc = s_acc[lane][warp];
    nrm = s_nrm[lane][warp];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
        nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
    }
    if (lane == 0 && j0 + warp < l) b.c[pi][j0 + warp] = ritz_value(acc, nrm);
}

// The descending order of the Ritz values (c): iaux[rank] = j,
// rank_j = #{i : d_i before d_j}.
__global__ void __launch_bounds__(256) k_ritz_order(const __grid_constant__ SmallBatch b) {
    pdl_begin();
    __shared__ float d[1024];
    const int pi = blockIdx.y;
    const int l = b.l[pi];
    if (static_cast<int>(blockIdx.x) * 256 >= l) return;
    const int j = blockIdx.x * 256 + threadIdx.x;
    const float dj = j < l ? b.c[pi][j] : 0.0f;
    int rank = 0;
    for (int i0 = 0; i0 < l; i0 += 1024) {
        const int cnt = min(1024, l - i0);
        __syncthreads();
        for (int i = threadIdx.x; i < cnt; i += 256) d[i] = b.c[pi][i0 + i];
        __syncthreads();
        for (int i = 0; i < cnt; ++i) rank += ritz_before(d[i], i0 + i, dj, j) ? 1 : 0;
    }
    if (j < l) b.iaux[pi][rank] = j;
}

// ---------------------------------------------------------------------------
// Exact Rayleigh-Ritz on the leading w = min(64, l) columns of an orthonormal
// X (a, l x l) with W = C X (b): H = X_w^T W_w (w x w, symmetric), its
// eigen-decomposition H = J diag(h) J^T by the cyclic Jacobi method (Golub
// and Van Loan, Matrix Computations, 4th ed., §8.5: one rotation per index
// pair zeroes H_pq; the pairs of a sweep are scheduled as a round-robin
// tournament so that the w / 2 rotations of a round touch disjoint rows and
// columns and run in parallel), then X_w <- X_w J and W_w <- W_w J.  The
// orthogonal iteration before it leaves span(X_w) close to the leading
// invariant subspace of C; within it the individual eigenvectors of
// separated eigenvalues are then exact up to rounding.
//
// Three launches: partial Gram blocks over slabs of rows, one CTA per module
// for the Jacobi sweeps, and the rotation over slabs of rows.  As one CTA per
// module the whole took 0.32 / 0.63 / 1.20 ms at l = 64 / 288 / 2080, now
// 0.22 / 0.36 / 0.37 ms; what is left is the chain of the sweeps.  h: scratch of
// l x l floats, the partial Gram blocks and then J.
// ---------------------------------------------------------------------------
constexpr int kLeadW = 64;

// Slabs of at least 64 rows, so that the partial blocks fit l x l floats.
__host__ __device__ inline int lead_slabs(int l) { return l < 2 * kLeadW ? 1 : l / kLeadW; }

__global__ void __launch_bounds__(256) k_lead_gram(const __grid_constant__ SmallBatch b) {
    pdl_begin();
    __shared__ __align__(16) float xs[32][kLeadW], ws[32][kLeadW];
    const int pi = blockIdx.y;
    const int l = b.l[pi];
    const int w = min(l, kLeadW), ns = lead_slabs(l);
    if (static_cast<int>(blockIdx.x) >= ns) return;
    const int r0 = blockIdx.x * kLeadW, r1 = static_cast<int>(blockIdx.x) + 1 == ns ? l : r0 + kLeadW;
    const float* X = b.a[pi];
    const float* W = b.b[pi];
    const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
    float acc[4][4] = {};
    for (int r = r0; r < r1; r += 32) {
        for (int e = t; e < 32 * kLeadW; e += 256) {
            const int i = e / kLeadW, j = e % kLeadW;
            const bool in = r + i < r1 && j < w;
            xs[i][j] = in ? X[(long long)(r + i) * l + j] : 0.0f;
            ws[i][j] = in ? W[(long long)(r + i) * l + j] : 0.0f;
        }
        __syncthreads();
#pragma unroll 8
        for (int i = 0; i < 32; ++i) {
            const float4 x = *reinterpret_cast<const float4*>(&xs[i][4 * ty]);
            const float4 y = *reinterpret_cast<const float4*>(&ws[i][4 * tx]);
            const float xv[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(xv[p], yv[q], acc[p][q]);
        }
        __syncthreads();
    }
    float* out = reinterpret_cast<float*>(b.h[pi]) + (long long)blockIdx.x * w * w;
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (4 * ty + p < w && 4 * tx + q < w) out[(4 * ty + p) * w + 4 * tx + q] = acc[p][q];
}

constexpr int kJacThreads = 512;
constexpr int kJacPairs = kLeadW / 2;

__global__ void __launch_bounds__(kJacThreads) k_lead_jacobi(const __grid_constant__ SmallBatch b) {
    pdl_begin();
    __shared__ float H[kLeadW][kLeadW + 1];
    __shared__ float J[kLeadW][kLeadW + 1];
    __shared__ float rc[2][kJacPairs], rs_[2][kJacPairs];     // rotations of this round and the last one
    __shared__ int rp[2][kJacPairs], rq[2][kJacPairs];
    __shared__ float red[33];
    const int pi = blockIdx.x;
    const int l = b.l[pi];
    const int w = min(l, kLeadW), ns = lead_slabs(l);
    const int wp = w + (w & 1);                    // even player count (a dummy index when w is odd)
    float* const part = reinterpret_cast<float*>(b.h[pi]);
    const int t = threadIdx.x;
    for (int e = t; e < kLeadW * kLeadW; e += kJacThreads) {
        const int p = e / kLeadW, q = e % kLeadW;
        float v = 0.0f;
        if (p < w && q < w)
            for (int k = 0; k < ns; ++k) v += part[(long long)k * w * w + p * w + q];
        H[p][q] = v;
        J[p][q] = (p == q) ? 1.0f : 0.0f;
    }
    __syncthreads();
    // symmetrise (the two triangles differ by rounding)
    for (int e = t; e < w * w; e += kJacThreads) {
        const int p = e / w, q = e % w;
        if (p < q) {
            const float v = 0.5f * (H[p][q] + H[q][p]);
            H[p][q] = v;
            H[q][p] = v;
        }
    }
    __syncthreads();
    const int npairs = wp / 2;
    const int lane = t & 31, warp = t >> 5;
    constexpr int WARPS = kJacThreads / 32;
    // J <- J G for the rotations in buffer k, rows dealt to warps first, first + 1, ..
    auto turn_j = [&](int k, int first) {
        if (lane >= npairs || rq[k][lane] >= w) return;
        const int p2 = rp[k][lane], q2 = rq[k][lane];
        const float c2 = rc[k][lane], s2 = rs_[k][lane];
#pragma unroll 4
        for (int row = warp - first; row < w; row += WARPS - first) {
            const float jp = J[row][p2], jq = J[row][q2];
            J[row][p2] = c2 * jp - s2 * jq;
            J[row][q2] = s2 * jp + c2 * jq;
        }
    };
    int done = 0;                                  // rounds so far; J is one behind
    for (int sweep = 0; sweep < 20; ++sweep) {
        // stop once the off-diagonal mass is below fp32 resolution of the diagonal
        float off = 0.0f, dia = 0.0f;
        for (int e = t; e < w * w; e += kJacThreads) {
            const int p = e / w, q = e % w;
            const float v = H[p][q];
            if (p == q) dia = fmaf(v, v, dia); else off = fmaf(v, v, off);
        }
        off = block_sum(off, red);
        dia = block_sum(dia, red);
        if (!(off > 1e-14f * dia)) break;          // also ends on a non-finite H
        for (int round = 0; round < wp - 1; ++round, ++done) {
            const int k = done & 1;
            if (warp == 0) {
                if (t < npairs) {
                    // tournament: player 0 fixed, the others rotate by one each round
                    auto player = [&](int pos) {
                        int x = pos - 1 + round;
                        if (x >= wp - 1) x -= wp - 1;
                        return pos == 0 ? 0 : 1 + x;
                    };
                    int p = player(t), q = player(wp - 1 - t);
                    if (p > q) { const int x = p; p = q; q = x; }
                    float c = 1.0f, sn = 0.0f;
                    if (q < w) {
                        const float hpq = H[p][q];
                        if (fabsf(hpq) > 1e-30f) {
                            // the angle to a few ulp (approximate division),
                            // the rotation orthonormal to rounding: c from the
                            // tangent that sn uses, by rsqrtf and one step of
                            // Newton's iteration
                            const float tau = __fdividef(H[q][q] - H[p][p], 2.0f * hpq);
                            const float at = fabsf(tau);
                            // |tau| past 1e15: tan = 1 / (2 tau), below it (tau^2 does not overflow)
                            const float tt = copysignf(at < 1e15f ? __fdividef(1.0f, at + __fsqrt_rn(fmaf(tau, tau, 1.0f)))
                                                                  : __fdividef(0.5f, at), tau);
                            const float d = fmaf(tt, tt, 1.0f);
                            const float r = rsqrtf(d);
                            c = fmaf(0.5f * r, fmaf(-d * r, r, 1.0f), r);
                            sn = tt * c;
                        }
                    }
                    rp[k][t] = p; rq[k][t] = q; rc[k][t] = c; rs_[k][t] = sn;
                }
            } else if (done > 0) {
                turn_j(k ^ 1, 1);
            }
            __syncthreads();
            // H <- G^T H G by 2 x 2 blocks: the block of pairs (k1, k2) is read
            // and written by one thread (lane = k2, a warp takes two k1)
            if (lane < npairs) {
                const int p2 = rp[k][lane], q2 = rq[k][lane];
                const float c2 = rc[k][lane], s2 = rs_[k][lane];
                const bool two = q2 < w;
#pragma unroll
                for (int u = 0; u < kJacPairs / WARPS; ++u) {
                    const int k1 = warp + u * WARPS;
                    if (k1 >= npairs) break;
                    const int p1 = rp[k][k1], q1 = rq[k][k1];
                    const float c1 = rc[k][k1], s1 = rs_[k][k1];
                    const float a = H[p1][p2], d = q1 < w && two ? H[q1][q2] : 0.0f;
                    const float h = two ? H[p1][q2] : 0.0f, v = q1 < w ? H[q1][p2] : 0.0f;
                    // columns, then rows
                    const float a1 = c2 * a - s2 * h, u1 = s2 * a + c2 * h;
                    const float v1 = c2 * v - s2 * d, d1 = s2 * v + c2 * d;
                    H[p1][p2] = c1 * a1 - s1 * v1;
                    if (two) H[p1][q2] = c1 * u1 - s1 * d1;
                    if (q1 < w) H[q1][p2] = s1 * a1 + c1 * v1;
                    if (two && q1 < w) H[q1][q2] = s1 * u1 + c1 * d1;
                }
            }
            __syncthreads();
        }
    }
    if (done > 0) turn_j((done - 1) & 1, 0);
    __syncthreads();
    for (int e = t; e < w * w; e += kJacThreads) part[e] = J[e / w][e % w];
}

// X_w <- X_w J, W_w <- W_w J: 32 rows of one of the two per CTA.
__global__ void __launch_bounds__(256) k_lead_rotate(const __grid_constant__ SmallBatch b) {
    pdl_begin();
    __shared__ float js[kLeadW][kLeadW], xs[32][kLeadW];
    const int pi = blockIdx.y;
    const int l = b.l[pi];
    const int w = min(l, kLeadW);
    const int r0 = static_cast<int>(blockIdx.x) * 32;
    if (r0 >= l) return;
    float* const X = blockIdx.z == 0 ? b.a[pi] : b.b[pi];
    const float* J = reinterpret_cast<const float*>(b.h[pi]);
    for (int e = threadIdx.x; e < w * w; e += 256) js[e / w][e % w] = J[e];
    for (int e = threadIdx.x; e < 32 * kLeadW; e += 256) {
        const int i = e / kLeadW, j = e % kLeadW;
        xs[i][j] = (r0 + i < l && j < w) ? X[(long long)(r0 + i) * l + j] : 0.0f;
    }
    __syncthreads();
    const int j = threadIdx.x & 63;
    if (j >= w) return;
    for (int i = threadIdx.x >> 6; i < 32 && r0 + i < l; i += 4) {
        float o = 0.0f;
        for (int k = 0; k < w; ++k) o = fmaf(xs[i][k], js[k][j], o);
        X[(long long)(r0 + i) * l + j] = o;
    }
}

cudaError_t launch_lead_ritz(const SmallBatch& b, cudaStream_t s, int64_t* launches) {
    if (b.count <= 0) return cudaSuccess;
    int lmax = 1;
    for (int q = 0; q < b.count; ++q) lmax = std::max(lmax, b.l[q]);
    *launches += 3;
    cudaError_t e = launch(k_lead_gram, dim3(lead_slabs(lmax), b.count), 256, 0, s, 1, b);
    if (e == cudaSuccess) e = launch(k_lead_jacobi, b.count, kJacThreads, 0, s, 1, b);
    if (e == cudaSuccess) e = launch(k_lead_rotate, dim3((lmax + 31) / 32, b.count, 2), 256, 0, s, 1, b);
    return e;
}

cudaError_t launch_ritz_sort(const SmallBatch& b, cudaStream_t s, int64_t* launches) {
    if (b.count <= 0) return cudaSuccess;
    int lmax = 1;
    for (int q = 0; q < b.count; ++q) lmax = std::max(lmax, b.l[q]);
    *launches += 2;
    cudaError_t e = launch(k_ritz_values, dim3((lmax + 31) / 32, b.count), kSmallThreads, 0, s, 1, b);
    if (e == cudaSuccess) e = launch(k_ritz_order, dim3((lmax + 255) / 256, b.count), 256, 0, s, 1, b);
    return e;
}

// ---------------------------------------------------------------------------
// c[:, q] = a[:, iaux[q]] for q < rows (a is l x l, c is l x rows).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_gather_cols(const __grid_constant__ SmallBatch b) {
    pdl_begin();
    const int pi = blockIdx.y;
    const int l = b.l[pi], r = b.rows[pi];
    const int* perm = b.iaux[pi];
    for (int i = blockIdx.x; i < l; i += gridDim.x) {
        const float* src = b.a[pi] + (long long)i * l;
        float* dst = b.c[pi] + (long long)i * r;
        for (int q = threadIdx.x; q < r; q += blockDim.x) dst[q] = src[perm[q]];
    }
}

cudaError_t launch_gather_cols(const SmallBatch& b, cudaStream_t s, int64_t* launches) {
    if (b.count <= 0) return cudaSuccess;
    int lmax = 1;
    for (int q = 0; q < b.count; ++q) lmax = std::max(lmax, b.l[q]);
    ++*launches;
    return launch(k_gather_cols, dim3(std::min(1024, lmax), b.count), 256, 0, s, 1, b);
}

// ---------------------------------------------------------------------------
// Final projector: each column of a (rows x l, here l = r columns) is scaled
// to unit length and signed so that its largest-magnitude entry is positive
// (lowest row wins ties), then stored to c (fp32) and h (bf16).  Skipped when
// the problem's fail flag is set, which leaves the previous projector in place.
// ---------------------------------------------------------------------------
// A cluster of kSignCtas CTAs owns 32 columns: lane = column, the CTAs' 8 warps
// each split the rows (every row segment one coalesced 128-byte access), and
// the column's maximum and norm are combined through distributed shared
// memory.  Two passes over a, the second out of L2: bound by the loads in
// flight, so the rows are spread over eight SMs (one CTA per 32 columns took
// 1.0 ms on the seven weights of a 4096 / 11008 layer, a cluster 0.2 ms).
constexpr int kSignCtas = 8;

__global__ void __launch_bounds__(256) k_sign_fix_store(const __grid_constant__ SmallBatch b) {
    pdl_begin();
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ float s_best[8][32];
    __shared__ int s_bi[8][32];
    __shared__ float s_ss[8][32];
    __shared__ float c_best[32], c_ss[32];
    __shared__ int c_bi[32];
    const int pi = blockIdx.y;
    const int rows = b.rows[pi], r = b.l[pi];
    const int q0 = static_cast<int>(blockIdx.x) / kSignCtas * 32;
    // the whole cluster leaves together
    if (q0 >= r || (b.fail[pi] != nullptr && *b.fail[pi] != 0)) return;
    const int rank = static_cast<int>(cl.block_rank());
    const float* Pt = b.a[pi];
    float* P = b.c[pi];
    uint16_t* Pb = b.h[pi];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i0 = static_cast<int>((long long)rows * rank / kSignCtas);
    const int i1 = static_cast<int>((long long)rows * (rank + 1) / kSignCtas);
    const int q = q0 + lane;
    const bool col = q < r;
    // largest |entry| of the column over this warp's rows (ascending, so
    // the lowest row wins ties)
    float best = -1.0f, ss = 0.0f;
    int bi = 0x7fffffff;
    if (col) {
#pragma unroll 4
        for (int i = i0 + warp; i < i1; i += 8) {
            const float v = Pt[(long long)i * r + q];
            const float a = fabsf(v);
            ss = fmaf(v, v, ss);
            if (a > best) { best = a; bi = i; }
        }
    }
    s_best[warp][lane] = best;
    s_bi[warp][lane] = bi;
    s_ss[warp][lane] = ss;
    __syncthreads();
    if (warp == 0) {
        for (int w = 1; w < 8; ++w) {
            const float ob = s_best[w][lane];
            const int oi = s_bi[w][lane];
            ss += s_ss[w][lane];
            if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        c_best[lane] = best;
        c_bi[lane] = bi;
        c_ss[lane] = ss;
    }
    cl.sync();
    best = -1.0f;
    bi = 0x7fffffff;
    ss = 0.0f;
#pragma unroll
    for (int k = 0; k < kSignCtas; ++k) {
        const float ob = cl.map_shared_rank(c_best, k)[lane];
        const int oi = cl.map_shared_rank(c_bi, k)[lane];
        ss += cl.map_shared_rank(c_ss, k)[lane];
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    const float sg = (col && bi < rows && Pt[(long long)bi * r + q] < 0.0f) ? -1.0f : 1.0f;
    // unit length (a zero or non-finite column is left unscaled)
    const float nrm = sqrtf(ss);
    const float sgnv = (nrm > 0.0f && isfinite(nrm)) ? sg / nrm : sg;
    cl.sync();          // no CTA leaves while a peer may still read its sums
    if (col) {
#pragma unroll 4
        for (int i = i0 + warp; i < i1; i += 8) {
            const float v = Pt[(long long)i * r + q] * sgnv;
            P[(long long)i * r + q] = v;
            if (Pb != nullptr) {
                __nv_bfloat16 h = __float2bfloat16_rn(v);
                Pb[(long long)i * r + q] = *reinterpret_cast<uint16_t*>(&h);
            }
        }
    }
}

cudaError_t launch_sign_fix_store(const SmallBatch& b, cudaStream_t s, int64_t* launches) {
    if (b.count <= 0) return cudaSuccess;
    int rmax = 1;
    for (int q = 0; q < b.count; ++q) rmax = std::max(rmax, b.l[q]);
    ++*launches;
    return launch(k_sign_fix_store, dim3((rmax + 31) / 32 * kSignCtas, b.count), 256, 0, s, kSignCtas, b);
}

}  // namespace moara
