// fp32 SIMT kernels of the step: block decomposition with the magnitude
// branch's Adam, and grouped tiled GEMMs (128 x 128 tiles, or 64 x 64 tiles
// with a split K range) whose operand loaders apply the block scales of the
// decomposition and whose epilogues run the direction branch's Adam or the
// weight update.  Every product is an fp32 FMA, so this
// path meets the all-fp32 tolerance; it also serves the refresh.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "internal.h"
#include "launch.cuh"

namespace moara {

__device__ __forceinline__ float bf16_bits_to_f32(uint16_t h) {
    return __uint_as_float(static_cast<uint32_t>(h) << 16);
}

template <bool BF16>
__device__ __forceinline__ float load_elem(const void* base, long long idx) {
    if (BF16) {
        return bf16_bits_to_f32(__ldg(reinterpret_cast<const unsigned short*>(base) + idx));
    } else {
        return __ldg(reinterpret_cast<const float*>(base) + idx);
    }
}

// ---------------------------------------------------------------------------
// Decompose(G, B) of §3.1 / Appendix B.1 for every (row, block) item, plus
// Optimizer_M (Adam on the block magnitudes, Algorithm 1).  Writes the inverse
// scales 1 / (m_{i,b} + eps) used by the projection's operand loader.
// Columns past n (the right zero padding) contribute nothing to the norm.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int find_item(const long long* start, int count, long long item) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (start[mid] <= item) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ void finish_item(const DecompBatch& b, const DecompItem& it,
                                            long long local, float ss) {
    float mag = sqrtf(ss);
    it.inv[local] = 1.0f / (mag + b.decomp_eps);
    if (b.do_mag) {
        // a clipped gradient c G has block norms c M and the same direction V
        if (b.clip != nullptr) mag *= *b.clip;
        float ma = b.beta1 * it.mag_avg[local] + (1.0f - b.beta1) * mag;
        float mas = b.beta2 * it.mag_avg_sq[local] + (1.0f - b.beta2) * mag * mag;
        it.mag_avg[local] = ma;
        it.mag_avg_sq[local] = mas;
        it.dM[local] = (ma / b.bc1) / (sqrtf(mas / b.bc2) + b.adam_eps);
    }
}

// One thread per (row, block): used for B <= 32.
__global__ void __launch_bounds__(256) k_decompose_thread(const __grid_constant__ DecompBatch b) {
    pdl_begin();
    const long long total = b.item_start[b.count];
    for (long long item = blockIdx.x * (long long)blockDim.x + threadIdx.x; item < total;
         item += (long long)gridDim.x * blockDim.x) {
        const int pi = find_item(b.item_start, b.count, item);
        const DecompItem& it = b.p[pi];
        const long long local = item - b.item_start[pi];
        const int row = static_cast<int>(local / it.kb);
        const int blk = static_cast<int>(local - (long long)row * it.kb);
        const int c0 = blk * b.B;
        const int c1 = min(c0 + b.B, it.n);
        const long long base = (long long)row * it.n;
        float ss = 0.0f;
        if (it.dtype == MOARA_DTYPE_BF16) {
            for (int c = c0; c < c1; ++c) { float x = load_elem<true>(it.G, base + c); ss = fmaf(x, x, ss); }
        } else {
            for (int c = c0; c < c1; ++c) { float x = load_elem<false>(it.G, base + c); ss = fmaf(x, x, ss); }
        }
        finish_item(b, it, local, ss);
    }
}

// One warp per (row, block): used for B > 32.
__global__ void __launch_bounds__(256) k_decompose_warp(const __grid_constant__ DecompBatch b) {
    pdl_begin();
    const long long total = b.item_start[b.count];
    const int lane = threadIdx.x & 31;
    const long long warp0 = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long item = warp0; item < total; item += nwarps) {
        const int pi = find_item(b.item_start, b.count, item);
        const DecompItem& it = b.p[pi];
        const long long local = item - b.item_start[pi];
        const int row = static_cast<int>(local / it.kb);
        const int blk = static_cast<int>(local - (long long)row * it.kb);
        const int c0 = blk * b.B;
        const int c1 = min(c0 + b.B, it.n);
        const long long base = (long long)row * it.n;
        float ss = 0.0f;
        if (it.dtype == MOARA_DTYPE_BF16) {
            for (int c = c0 + lane; c < c1; c += 32) { float x = load_elem<true>(it.G, base + c); ss = fmaf(x, x, ss); }
        } else {
            for (int c = c0 + lane; c < c1; c += 32) { float x = load_elem<false>(it.G, base + c); ss = fmaf(x, x, ss); }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        if (lane == 0) finish_item(b, it, local, ss);
    }
}

cudaError_t launch_decompose(const DecompBatch& b, cudaStream_t s, int64_t* launches) {
    const long long total = b.item_start[b.count];
    if (total <= 0) return cudaSuccess;
    const int threads = 256;
    if (b.B > 32) {
        long long blocks = (total * 32 + threads - 1) / threads;
        if (blocks > 152LL * 64) blocks = 152LL * 64;
        ++*launches;
        return launch(k_decompose_warp, static_cast<unsigned>(blocks), threads, 0, s, 1, b);
    } else {
        long long blocks = (total + threads - 1) / threads;
        if (blocks > 152LL * 64) blocks = 152LL * 64;
        ++*launches;
        return launch(k_decompose_thread, static_cast<unsigned>(blocks), threads, 0, s, 1, b);
    }
}

// ---------------------------------------------------------------------------
// Grouped SIMT GEMM: 128 x 128 tile, BK = 8, 256 threads, 8 x 8 per thread,
// register-staged double buffering.  blockIdx.x enumerates the tiles of all
// problems of the batch (problems are ordered longest-K first by the host).
// ---------------------------------------------------------------------------
constexpr int TM = 128, TN = 128, TK = 16, TPAD = 4;
constexpr int NQ = TK * 128 / 256;   // elements of A (and of B) each thread stages per k-tile

// Index of the block holding column c: a shift when B is a power of two.
__device__ __forceinline__ int block_of(int c, int B, int log2B) { return log2B >= 0 ? (c >> log2B) : c / B; }

template <int ALAY, bool ASC, bool ABF, int BLAY, bool BSC, bool BBF>
struct TileLoader {
    float ra[NQ], rb[NQ];

    __device__ __forceinline__ void load(const GemmProb& p, int m0, int n0, int k0, int B, int log2B) {
        const int t = threadIdx.x;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            int i, k;
            if (ALAY == A_KCONTIG) { k = t & (TK - 1); i = (t / TK) + (256 / TK) * q; }
            else                   { i = t & 127; k = (t >> 7) + 2 * q; }
            const int gi = m0 + i, gk = k0 + k;
            float v = 0.0f;
            if (gi < p.M && gk < p.K) {
                long long idx;
                int vrow, vcol;
                if (ALAY == A_KCONTIG) { idx = (long long)gi * p.lda + gk; vrow = gi; vcol = gk; }
                else                   { idx = (long long)gk * p.lda + gi; vrow = gk; vcol = gi; }
                v = load_elem<ABF>(p.A, idx);
                if (ASC) v *= __ldg(p.a_inv + (long long)vrow * p.kb + block_of(vcol, B, log2B));
            }
            ra[q] = v;
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            int j, k;
            if (BLAY == B_NCONTIG) { j = t & 127; k = (t >> 7) + 2 * q; }
            else                   { k = t & (TK - 1); j = (t / TK) + (256 / TK) * q; }
            const int gj = n0 + j, gk = k0 + k;
            float v = 0.0f;
            if (gj < p.N && gk < p.K) {
                long long idx;
                int vrow, vcol;
                if (BLAY == B_NCONTIG) { idx = (long long)gk * p.ldb + gj; vrow = gk; vcol = gj; }
                else                   { idx = (long long)gj * p.ldb + gk; vrow = gj; vcol = gk; }
                v = load_elem<BBF>(p.Bm, idx);
                if (BSC) v *= __ldg(p.b_inv + (long long)vrow * p.kb + block_of(vcol, B, log2B));
            }
            rb[q] = v;
        }
    }

    __device__ __forceinline__ void store(float (*As)[TM + TPAD], float (*Bs)[TN + TPAD]) {
        const int t = threadIdx.x;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            int i, k;
            if (ALAY == A_KCONTIG) { k = t & (TK - 1); i = (t / TK) + (256 / TK) * q; }
            else                   { i = t & 127; k = (t >> 7) + 2 * q; }
            As[k][i] = ra[q];
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            int j, k;
            if (BLAY == B_NCONTIG) { j = t & 127; k = (t >> 7) + 2 * q; }
            else                   { k = t & (TK - 1); j = (t / TK) + (256 / TK) * q; }
            Bs[k][j] = rb[q];
        }
    }
};

// What the epilogue of entry (i, j) reads: the moments (EPI_ADAM), or W and dM
// (EPI_UPDATE).
struct Old {
    float x, y;
};

template <int EPI, int CAP>
__device__ __forceinline__ Old epilogue_old(const GemmBatchT<CAP>& b, const GemmProb& p, int i, int j) {
    const long long o = (long long)i * p.ldc + j;
    if (EPI == EPI_ADAM) return Old{p.aux0[o], p.aux1[o]};
    if (EPI == EPI_UPDATE)
        return Old{p.aux0[o], p.aux2 != nullptr ? p.aux2[(long long)i * p.kb + block_of(j, b.B, b.log2B)] : 1.0f};
    return Old{0.0f, 0.0f};
}

template <int EPI, int CAP>
__device__ __forceinline__ void epilogue(const GemmBatchT<CAP>& b, const GemmProb& p, int i, int j, float acc,
                                         const Old& old) {
    const long long o = (long long)i * p.ldc + j;
    if (EPI == EPI_STORE) {
        p.C[o] = acc;
        if (p.c_bf16 != nullptr) {
            __nv_bfloat16 h = __float2bfloat16_rn(acc);
            p.c_bf16[o] = *reinterpret_cast<uint16_t*>(&h);
        }
    } else if (EPI == EPI_STORE_NEG) {
        p.C[o] = -acc;
    } else if (EPI == EPI_ADAM) {
        // Optimizer_V (Algorithm 1): Adam on the projected direction R = acc
        // (of the clipped gradient when a clipping coefficient is given).
        if (b.clip != nullptr) acc *= *b.clip;
        float ea = b.beta1 * old.x + (1.0f - b.beta1) * acc;
        float eas = b.beta2 * old.y + (1.0f - b.beta2) * acc * acc;
        p.aux0[o] = ea;
        p.aux1[o] = eas;
        p.C[o] = (ea / b.bc1) / (sqrtf(eas / b.bc2) + b.adam_eps);
    } else {
        // W <- W - lr*alpha*(Rep_B(dM) (.) dV)  (Algorithm 1; Rep_B of §3.1).
        float u = acc;
        if (p.aux2 != nullptr) u *= old.y;
        p.aux0[o] = old.x - b.step_scale * u;
    }
}

template <int ALAY, bool ASC, bool ABF, int BLAY, bool BSC, bool BBF, int EPI>
__global__ void __launch_bounds__(256, 2) k_gemm(const __grid_constant__ GemmBatch b) {
    pdl_begin();
    __shared__ __align__(16) float As[2][TK][TM + TPAD];
    __shared__ __align__(16) float Bs[2][TK][TN + TPAD];

    // locate (problem, tile)
    const int tile = blockIdx.x;
    int lo = 0, hi = b.count - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (b.tile_start[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    const GemmProb& p = b.p[lo];
    const int local = tile - b.tile_start[lo];
    const int tn = b.tiles_n[lo];
    const int m0 = (local / tn) * TM;
    const int n0 = (local % tn) * TN;
    if (p.lower_only && n0 >= m0 + TM) return;

    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float acc[8][8];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[a][c] = 0.0f;

    TileLoader<ALAY, ASC, ABF, BLAY, BSC, BBF> ld;
    int kbeg = 0, kend = p.K;
    if (p.k_tri == KTRI_B_UPPER) kend = min(p.K, n0 + TN);
    else if (p.k_tri == KTRI_B_LOWER) kbeg = min(p.K, n0) & ~(TK - 1);
    else if (p.k_tri == KTRI_A_LOWER) kend = min(p.K, m0 + TM);
    const int ktiles = kend > kbeg ? (kend - kbeg + TK - 1) / TK : 0;
    if (ktiles > 0) {
        ld.load(p, m0, n0, kbeg, b.B, b.log2B);
        ld.store(As[0], Bs[0]);
    }
    __syncthreads();
    for (int kt = 0; kt < ktiles; ++kt) {
        const int cur = kt & 1;
        if (kt + 1 < ktiles) ld.load(p, m0, n0, kbeg + (kt + 1) * TK, b.B, b.log2B);
#pragma unroll
        for (int k = 0; k < TK; ++k) {
            float av[8], bv[8];
            const float4 a0 = *reinterpret_cast<const float4*>(&As[cur][k][ty * 4]);
            const float4 a1 = *reinterpret_cast<const float4*>(&As[cur][k][64 + ty * 4]);
            const float4 b0 = *reinterpret_cast<const float4*>(&Bs[cur][k][tx * 4]);
            const float4 b1 = *reinterpret_cast<const float4*>(&Bs[cur][k][64 + tx * 4]);
            av[0] = a0.x; av[1] = a0.y; av[2] = a0.z; av[3] = a0.w;
            av[4] = a1.x; av[5] = a1.y; av[6] = a1.z; av[7] = a1.w;
            bv[0] = b0.x; bv[1] = b0.y; bv[2] = b0.z; bv[3] = b0.w;
            bv[4] = b1.x; bv[5] = b1.y; bv[6] = b1.z; bv[7] = b1.w;
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[a][c] = fmaf(av[a], bv[c], acc[a][c]);
        }
        if (kt + 1 < ktiles) {
            ld.store(As[cur ^ 1], Bs[cur ^ 1]);
        }
        __syncthreads();
    }

    // Plain stores move four consecutive columns per thread as one 16-byte
    // access when the layout allows it.
    if (EPI == EPI_STORE || EPI == EPI_STORE_NEG) {
        const bool vec = (p.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(p.C) & 15) == 0 &&
                         (EPI != EPI_STORE || p.c_bf16 == nullptr ||
                          (reinterpret_cast<uintptr_t>(p.c_bf16) & 7) == 0);
        if (vec) {
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                const int i = m0 + (a < 4 ? ty * 4 + a : 64 + ty * 4 + (a - 4));
                if (i >= p.M) continue;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int j = n0 + h * 64 + tx * 4;
                    if (j + 3 < p.N) {
                        const long long o = (long long)i * p.ldc + j;
                        float4 v = make_float4(acc[a][4 * h], acc[a][4 * h + 1], acc[a][4 * h + 2],
                                               acc[a][4 * h + 3]);
                        float4* dst = reinterpret_cast<float4*>(p.C + o);
                        if (EPI == EPI_STORE_NEG) v = make_float4(-v.x, -v.y, -v.z, -v.w);
                        *dst = v;
                        if (EPI == EPI_STORE && p.c_bf16 != nullptr) {
                            const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y);
                            const __nv_bfloat162 hi = __floats2bfloat162_rn(v.z, v.w);
                            uint2 pk;
                            pk.x = *reinterpret_cast<const uint32_t*>(&lo);
                            pk.y = *reinterpret_cast<const uint32_t*>(&hi);
                            *reinterpret_cast<uint2*>(p.c_bf16 + o) = pk;
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (j + c < p.N) epilogue<EPI>(b, p, i, j + c, acc[a][4 * h + c], epilogue_old<EPI>(b, p, i, j + c));
                    }
                }
            }
            return;
        }
    }
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        const int i = m0 + (a < 4 ? ty * 4 + a : 64 + ty * 4 + (a - 4));
        if (i >= p.M) continue;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int j = n0 + (c < 4 ? tx * 4 + c : 64 + tx * 4 + (c - 4));
            if (j < p.N) epilogue<EPI>(b, p, i, j, acc[a][c], epilogue_old<EPI>(b, p, i, j));
        }
    }
}

// ---------------------------------------------------------------------------
// Small variant for problems whose 128 x 128 tiles leave SMs idle: 64 x 64
// tiles, and the K range of a tile split over the CTAs of a cluster (up to
// eight), whose partial tiles are summed through distributed shared memory in
// rank order; CTA q of the cluster then runs the epilogue on its 64 / S rows.
// A 128-tile at K = 1024 is a serial chain of 64 k-tiles, each with a global
// load latency: the projection of a 1024 x 1024 weight at r = 128 (8 tiles)
// took 413 us, here 31 us (32 tiles x 8 CTAs, cold); of 256 x 256 at r = 32
// (2 tiles) 122 us, here 12 us.
// ---------------------------------------------------------------------------
constexpr int SM_T = 64, SM_K = 32, SM_LD = SM_T + 4;

// This thread's eight elements of a 32-deep, 64-wide operand slice.
template <int LAY_K, bool SC, bool BF>
struct SliceLoader {
    float r[8];
    // LAY_K: element (x, k) at x * ld + k (k contiguous): a warp takes 4 x 8
    // (x, k) pieces, 32 bytes per row; else at k * ld + x: 32 consecutive x
    static __device__ __forceinline__ void place(int q, int& x, int& k) {
        const int t = threadIdx.x;
        if (LAY_K) { k = (t & 7) + 8 * (q & 3); x = (t >> 3) + 32 * (q >> 2); }
        else       { x = t & 63; k = (t >> 6) + 4 * q; }
    }
    __device__ __forceinline__ void load(const void* base, const float* inv, int ld, int kb, int x0, int X, int k0, int K,
                                         int B, int log2B) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            int x, k;
            place(q, x, k);
            const int gx = x0 + x, gk = k0 + k;
            float v = 0.0f;
            if (gx < X && gk < K) {
                const long long row = LAY_K ? gx : gk;
                const int col = LAY_K ? gk : gx;
                v = load_elem<BF>(base, row * ld + col);
                if (SC) v *= __ldg(inv + row * kb + block_of(col, B, log2B));
            }
            r[q] = v;
        }
    }
    __device__ __forceinline__ void store(float (*dst)[SM_LD]) const {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            int x, k;
            place(q, x, k);
            dst[k][x] = r[q];
        }
    }
};

template <int CAP, int ALAY, bool ASC, bool ABF, int BLAY, bool BSC, bool BBF, int EPI>
__global__ void __launch_bounds__(256, 4) k_gemm_small(const __grid_constant__ GemmBatchT<CAP> b) {
    pdl_begin();
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ __align__(16) float As[2][SM_K][SM_LD];
    __shared__ __align__(16) float Bs[2][SM_K][SM_LD];
    const int S = static_cast<int>(cl.num_blocks()), rank = static_cast<int>(cl.block_rank());
    const int tile = blockIdx.x / S;
    int lo = 0, hi = b.count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (b.tile_start[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    const GemmProb& p = b.p[lo];
    const int local = tile - b.tile_start[lo];
    const int tn = b.tiles_n[lo];
    const int m0 = (local / tn) * SM_T;
    const int n0 = (local % tn) * SM_T;
    if (p.lower_only && n0 >= m0 + SM_T) return;      // the whole cluster

    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    float acc[4][4] = {};
    int kbeg = 0, kend = p.K;
    if (p.k_tri == KTRI_B_UPPER) kend = min(p.K, n0 + SM_T);
    else if (p.k_tri == KTRI_B_LOWER) kbeg = min(p.K, n0);
    else if (p.k_tri == KTRI_A_LOWER) kend = min(p.K, m0 + SM_T);
    const int chunks = kend > kbeg ? (kend - kbeg + SM_K - 1) / SM_K : 0;
    const int split = p.split;                        // <= S; the other ranks only help to store
    const int c0 = rank < split ? chunks * rank / split : 0, c1 = rank < split ? chunks * (rank + 1) / split : 0;
    SliceLoader<ALAY == A_KCONTIG, ASC, ABF> la;
    SliceLoader<BLAY == B_KCONTIG, BSC, BBF> lb;
    auto load = [&](int c) {
        const int k0 = kbeg + c * SM_K;
        la.load(p.A, p.a_inv, p.lda, p.kb, m0, p.M, k0, kend, b.B, b.log2B);
        lb.load(p.Bm, p.b_inv, p.ldb, p.kb, n0, p.N, k0, kend, b.B, b.log2B);
    };
    if (c0 < c1) load(c0);
    for (int c = c0; c < c1; ++c) {
        const int cur = (c - c0) & 1;
        la.store(As[cur]);
        lb.store(Bs[cur]);
        __syncthreads();
        if (c + 1 < c1) load(c + 1);
#pragma unroll 8
        for (int k = 0; k < SM_K; ++k) {
            const float4 x = *reinterpret_cast<const float4*>(&As[cur][k][4 * ty]);
            const float4 y = *reinterpret_cast<const float4*>(&Bs[cur][k][4 * tx]);
            const float xv[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xv[i], yv[j], acc[i][j]);
        }
    }
    // partial tiles in A's buffers, then S row slabs
    __syncthreads();
    float (*part)[SM_LD] = As[0];
    static_assert(2 * SM_K == SM_T, "the partial tile fills both A slices");
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4*>(&part[4 * ty + i][4 * tx]) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    // entries of the CTA's rows, two a thread at a time: what the epilogue reads
    // is fetched first, for the first two before the barrier
    const int R = SM_T / S;
    Old old[2];
    auto fetch = [&](int e0) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = e0 + threadIdx.x + 256 * u, i = m0 + rank * R + e / SM_T, j = n0 + e % SM_T;
            if (e < R * SM_T && i < p.M && j < p.N) old[u] = epilogue_old<EPI>(b, p, i, j);
        }
    };
    fetch(0);
    if (S > 1) cl.sync();
    else __syncthreads();
    auto total = [&](int i, int j) {
        if (S == 1) return part[i][j];
        float x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = q < split ? *cl.map_shared_rank(&part[i][j], q) : 0.0f;
        float v = x[0];
#pragma unroll
        for (int q = 1; q < 8; ++q)
            if (q < split) v += x[q];
        return v;
    };
    for (int e0 = 0; e0 < R * SM_T; e0 += 512) {
        if (e0 > 0) fetch(e0);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = e0 + threadIdx.x + 256 * u, i = rank * R + e / SM_T, j = e % SM_T;
            if (e < R * SM_T && m0 + i < p.M && n0 + j < p.N) epilogue<EPI>(b, p, m0 + i, n0 + j, total(i, j), old[u]);
        }
    }
    if (S > 1) cl.sync();       // no CTA leaves while a peer may still read its partial tile
}

constexpr int kWideTiles = 304;       // two 128 x 128 tiles per SM
constexpr int kSmallCtas = 608;       // four 64 x 64 CTAs per SM

// Parts of a problem's K range: up to eight while the problem's own tiles leave
// SMs idle and a part has a slice of its own.  From the problem alone, so that
// its sums do not depend on what it is grouped with (both kernels add the
// terms of a part in the order of k).
static int k_split(const GemmProb& p) {
    const int tiles = (p.M + SM_T - 1) / SM_T * ((p.N + SM_T - 1) / SM_T);
    int split = 1;
    while (split < 8 && 2 * split * tiles <= kSmallCtas && p.K >= 2 * split * SM_K) split *= 2;
    return split;
}

template <int CAP, int ALAY, bool ASC, bool ABF, int BLAY, bool BSC, bool BBF, int EPI>
static cudaError_t launch_small(const GemmBatch& b, int total, int split, cudaStream_t s) {
    auto fn = k_gemm_small<CAP, ALAY, ASC, ABF, BLAY, BSC, BBF, EPI>;
    if constexpr (CAP == kMaxGroup) {
        return launch(fn, total * split, 256, 0, s, split, b);
    } else {
        GemmBatchT<CAP> f;
        f.count = b.count; f.B = b.B; f.log2B = b.log2B;
        f.beta1 = b.beta1; f.beta2 = b.beta2; f.adam_eps = b.adam_eps; f.bc1 = b.bc1; f.bc2 = b.bc2;
        f.step_scale = b.step_scale;
        f.clip = b.clip;
        for (int i = 0; i < b.count; ++i) {
            f.tiles_n[i] = b.tiles_n[i];
            f.tile_start[i] = b.tile_start[i];
            f.p[i] = b.p[i];
        }
        f.tile_start[b.count] = b.tile_start[b.count];
        return launch(fn, total * split, 256, 0, s, split, f);
    }
}

template <int ALAY, bool ASC, bool ABF, int BLAY, bool BSC, bool BBF, int EPI>
static cudaError_t launch_part(GemmBatch& b, cudaStream_t s, int64_t* launches) {
    auto enumerate = [&](int tm_, int tn_) {
        int total = 0;
        for (int i = 0; i < b.count; ++i) {
            const GemmProb& p = b.p[i];
            const int tm = (p.M + tm_ - 1) / tm_;
            const int tn = (p.N + tn_ - 1) / tn_;
            b.tiles_n[i] = tn;
            b.tile_start[i] = total;
            total += tm * tn;
        }
        b.tile_start[b.count] = total;
        return total;
    };
    int split = 1;
    for (int i = 0; i < b.count; ++i) split = b.p[i].split > split ? b.p[i].split : split;
    int total = enumerate(TM, TN);
    if (total == 0) return cudaSuccess;
    ++*launches;
    if (split == 1 && total >= kWideTiles) {
        // enough 128 x 128 tiles for every SM: half the shared-memory reads
        // per FMA of the small kernel
        return launch(k_gemm<ALAY, ASC, ABF, BLAY, BSC, BBF, EPI>, total, 256, 0, s, 1, b);
    }
    total = enumerate(SM_T, SM_T);
    if (b.count <= kFewGroup)
        return launch_small<kFewGroup, ALAY, ASC, ABF, BLAY, BSC, BBF, EPI>(b, total, split, s);
    return launch_small<kMaxGroup, ALAY, ASC, ABF, BLAY, BSC, BBF, EPI>(b, total, split, s);
}

template <int ALAY, bool ASC, bool ABF, int BLAY, bool BSC, bool BBF, int EPI>
static cudaError_t launch_one(GemmBatch& b, cudaStream_t s, int64_t* launches) {
    b.log2B = -1;
    if (b.B > 0 && (b.B & (b.B - 1)) == 0) {
        int lg = 0;
        while ((1 << lg) < b.B) ++lg;
        b.log2B = lg;
    }
    int whole = 0, tiles = 0, split = 1;
    for (int i = 0; i < b.count; ++i) {
        const GemmProb& p = b.p[i];
        b.p[i].split = k_split(p);
        whole += p.split == 1;
        split = p.split > split ? p.split : split;
        tiles += (p.M + SM_T - 1) / SM_T * ((p.N + SM_T - 1) / SM_T);
    }
    if (whole == 0 || whole == b.count || tiles * split <= kSmallCtas)
        return launch_part<ALAY, ASC, ABF, BLAY, BSC, BBF, EPI>(b, s, launches);
    // split problems and whole ones in launches of their own, where the whole
    // ones' idle CTAs would not fit beside the others
    for (int part = 0; part < 2; ++part) {
        GemmBatch c = b;
        c.count = 0;
        for (int i = 0; i < b.count; ++i)
            if ((b.p[i].split == 1) == (part == 1)) c.p[c.count++] = b.p[i];
        const cudaError_t e = launch_part<ALAY, ASC, ABF, BLAY, BSC, BBF, EPI>(c, s, launches);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Dispatch over the operand/epilogue combinations the library uses.
cudaError_t launch_gemm(const GemmKind& k, GemmBatch& b, cudaStream_t s, int64_t* launches) {
    if (b.count <= 0) return cudaSuccess;
#define MOARA_GEMM_CASE(AL, AS, AB, BL, BS, BB, EP)                                         \
    if (k.a_layout == AL && !!k.a_scale == AS && !!k.a_bf16 == AB && k.b_layout == BL &&   \
        !!k.b_scale == BS && !!k.b_bf16 == BB && k.epi == EP)                               \
        return launch_one<AL, AS, AB, BL, BS, BB, EP>(b, s, launches);
    // step: R = P^T V (+ Adam), V = G scaled (bf16 or f32) or G itself
    MOARA_GEMM_CASE(A_MCONTIG, false, false, B_NCONTIG, true, true, EPI_ADAM)
    MOARA_GEMM_CASE(A_MCONTIG, false, false, B_NCONTIG, true, false, EPI_ADAM)
    MOARA_GEMM_CASE(A_MCONTIG, false, false, B_NCONTIG, false, true, EPI_ADAM)
    MOARA_GEMM_CASE(A_MCONTIG, false, false, B_NCONTIG, false, false, EPI_ADAM)
    // step: dV = P N (+ weight update)
    MOARA_GEMM_CASE(A_KCONTIG, false, false, B_NCONTIG, false, false, EPI_UPDATE)
    // refresh: Y = V Omega, V scaled or raw, bf16 or f32
    MOARA_GEMM_CASE(A_KCONTIG, true, true, B_NCONTIG, false, false, EPI_STORE)
    MOARA_GEMM_CASE(A_KCONTIG, true, false, B_NCONTIG, false, false, EPI_STORE)
    MOARA_GEMM_CASE(A_KCONTIG, false, true, B_NCONTIG, false, false, EPI_STORE)
    // refresh: Z = V^T Q
    MOARA_GEMM_CASE(A_MCONTIG, true, true, B_NCONTIG, false, false, EPI_STORE)
    MOARA_GEMM_CASE(A_MCONTIG, true, false, B_NCONTIG, false, false, EPI_STORE)
    MOARA_GEMM_CASE(A_MCONTIG, false, true, B_NCONTIG, false, false, EPI_STORE)
    // plain fp32: Gram X^T X (MCONTIG), products X Y (KCONTIG), X L^-T (B KCONTIG)
    MOARA_GEMM_CASE(A_MCONTIG, false, false, B_NCONTIG, false, false, EPI_STORE)
    MOARA_GEMM_CASE(A_KCONTIG, false, false, B_NCONTIG, false, false, EPI_STORE)
    MOARA_GEMM_CASE(A_KCONTIG, false, false, B_KCONTIG, false, false, EPI_STORE)
    MOARA_GEMM_CASE(A_KCONTIG, false, false, B_NCONTIG, false, false, EPI_STORE_NEG)
#undef MOARA_GEMM_CASE
    return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// Global gradient norm for clipping: sum of squares per chunk in fp32 (at
// most kNormChunk / 256 terms per thread), chunk sums added in fp64; fixed
// chunk-to-CTA assignment and reduction order.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double block_sum_d(double v, double* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i];
    return t;
}

__global__ void __launch_bounds__(256) k_grad_sq(const __grid_constant__ GradNormBatch b, double* partials) {
    __shared__ double red[8];
    // a chunk is kNormChunk elements: 8 x 16 bytes per thread for bf16, 16 for
    // fp32; all of a thread's loads of a chunk are issued before the sums
    constexpr int VB = kNormChunk / (8 * 256);          // uint4 per thread, bf16
    constexpr int VF = kNormChunk / (4 * 256);          // float4 per thread, fp32
    static_assert(VB * 8 * 256 == kNormChunk && VF * 4 * 256 == kNormChunk, "chunk = whole vectors per thread");
    const long long total = b.chunk_start[b.count];
    double acc = 0.0;
    for (long long c = blockIdx.x; c < total; c += gridDim.x) {
        int lo = 0, hi = b.count - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (b.chunk_start[mid] <= c) lo = mid; else hi = mid - 1;
        }
        const long long e0 = (c - b.chunk_start[lo]) * kNormChunk;
        const long long e1 = min(e0 + (long long)kNormChunk, b.elems[lo]);
        float ss = 0.0f;
        if (b.dtype[lo] == MOARA_DTYPE_BF16) {
            const uint16_t* g = static_cast<const uint16_t*>(b.G[lo]);
            if (e1 - e0 == kNormChunk) {
                uint4 w[VB];
#pragma unroll
                for (int k = 0; k < VB; ++k)
                    w[k] = __ldcs(reinterpret_cast<const uint4*>(g + e0 + 8LL * (threadIdx.x + 256 * k)));
#pragma unroll
                for (int k = 0; k < VB; ++k) {
                    const uint32_t ww[4] = {w[k].x, w[k].y, w[k].z, w[k].w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float x = __uint_as_float(ww[q] << 16), y = __uint_as_float(ww[q] & 0xFFFF0000u);
                        ss = fmaf(x, x, ss);
                        ss = fmaf(y, y, ss);
                    }
                }
            } else {
                for (long long k = e0 + threadIdx.x; k < e1; k += blockDim.x) {
                    const float x = bf16_bits_to_f32(g[k]);
                    ss = fmaf(x, x, ss);
                }
            }
        } else {
            const float* g = static_cast<const float*>(b.G[lo]);
            if (e1 - e0 == kNormChunk) {
                float4 w[VF];
#pragma unroll
                for (int k = 0; k < VF; ++k)
                    w[k] = __ldcs(reinterpret_cast<const float4*>(g + e0 + 4LL * (threadIdx.x + 256 * k)));
#pragma unroll
                for (int k = 0; k < VF; ++k) {
                    ss = fmaf(w[k].x, w[k].x, ss);
                    ss = fmaf(w[k].y, w[k].y, ss);
                    ss = fmaf(w[k].z, w[k].z, ss);
                    ss = fmaf(w[k].w, w[k].w, ss);
                }
            } else {
                for (long long k = e0 + threadIdx.x; k < e1; k += blockDim.x) ss = fmaf(g[k], g[k], ss);
            }
        }
        acc += static_cast<double>(ss);
    }
    const double t = block_sum_d(acc, red);
    if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

cudaError_t launch_grad_sq(const GradNormBatch& b, double* partials, cudaStream_t s, int64_t* launches) {
    k_grad_sq<<<kNormParts, 256, 0, s>>>(b, partials);
    ++*launches;
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_clip_finish(const double* partials, int n, const float* extra,
                                                     float max_norm, float* state) {
    __shared__ double red[8];
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) acc += partials[i];
    double t = block_sum_d(acc, red);
    if (threadIdx.x == 0) {
        if (extra != nullptr) t += static_cast<double>(*extra);
        const double norm = sqrt(t);
        const double coef = static_cast<double>(max_norm) / (norm + 1e-6);
        state[0] = static_cast<float>(norm);
        state[1] = static_cast<float>(coef < 1.0 ? coef : 1.0);
    }
}

cudaError_t launch_clip_finish(const double* partials, int n, const float* extra, float max_norm, float* state,
                               cudaStream_t s, int64_t* launches) {
    k_clip_finish<<<1, 256, 0, s>>>(partials, n, extra, max_norm, state);
    ++*launches;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// fp32 -> (fp32 copy, bf16 round-to-nearest-even copy)
// ---------------------------------------------------------------------------
__global__ void k_f32_to_bf16(const float* __restrict__ src, float* dst_f32, uint16_t* dst_bf16,
                              long long count) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
        const float v = src[i];
        if (dst_f32 != nullptr && dst_f32 != src) dst_f32[i] = v;
        if (dst_bf16 != nullptr) {
            __nv_bfloat16 h = __float2bfloat16_rn(v);
            dst_bf16[i] = *reinterpret_cast<uint16_t*>(&h);
        }
    }
}

cudaError_t launch_f32_to_bf16(const float* src, float* dst_f32, uint16_t* dst_bf16,
                               long long count, cudaStream_t s, int64_t* launches) {
    if (count <= 0) return cudaSuccess;
    long long blocks = (count + 255) / 256;
    if (blocks > 152LL * 32) blocks = 152LL * 32;
    k_f32_to_bf16<<<static_cast<unsigned>(blocks), 256, 0, s>>>(src, dst_f32, dst_bf16, count);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace moara
