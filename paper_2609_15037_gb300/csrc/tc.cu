// Tensor-core path of the optimizer step for bf16 gradients (sm_103a):
//
//  K0  Decompose(G, B) of §3.1 / Appendix B.1 as a memory-bound prepass: block
//      norms in fp32 and the direction matrix V written in bf16 (at the first
//      Adam step also the residual V - V_hi, so that the projection carries
//      ~16 bits there), and Optimizer_M (Adam on the block magnitudes) with it;
//      as a pass of its own for blocks below 32 columns and where the clipping
//      coefficient needs every norm first.
//  K1  R = P^T V on tcgen05 (2-SM pairs: 256 ranks x 256 columns per CTA pair,
//      P exact in bf16), then Optimizer_V (Adam) on R in the epilogue; writes
//      the Adam update N as bf16.  (Algorithm 1.)
//  K2  dV = P N (2-SM pairs: 256 rows x 256 columns per CTA pair), then
//      W <- W - lr*alpha*(Rep_B(dM) (.) dV) in the epilogue, reading and
//      writing W once through TMA.  (Algorithm 1.)
//
// K1 and K2 are persistent and warp specialised: one warp issues TMA tile
// loads into a shared-memory ring, one thread of the even CTA of each pair
// issues tcgen05.mma (cta_group::2) into double-buffered TMEM accumulators,
// and epilogue warps drain TMEM while the next tile's MMAs run.  Every
// mbarrier wait is bounded; on expiry the kernel records
// MOARA_ERR_DEVICE_TIMEOUT in the context's status word, drains its own TMA
// copies and MMAs, frees TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <string>
#include <type_traits>
#include <vector>

#include "launch.cuh"
#include "tc.h"
#include "tc_ptx.cuh"

namespace moara {

namespace {

constexpr int kTcGroup = 224;                 // modules per launch (G maps in params)
constexpr long long kWaitLimit = 1LL << 32;   // ~2 s of SM clocks
constexpr int kMaps = 10;                     // tensor maps per module

struct TcMod {
    int m, n, r, kb;
    int right;        // right projector Q (n x r): K1 computes R = V Q (m x r)
    int w3d;          // fp32 W with n % 64 == 0: K2 adds its update in 64 x 64 chunks (map 8)
    uint16_t* Qt;     // r x n bf16 transpose of a right projector (K2's B operand)
    uint16_t* Vhi;    // m x n bf16 direction matrix (written by K0)
    uint16_t* Vlo;    // m x n bf16 residual (first Adam step)
    float* W;
    float* exp_avg;
    float* exp_avg_sq;
    float* mag;       // m x kb block norms (K0 -> magnitude Adam)
    float* mag_avg;
    float* mag_avg_sq;
    uint16_t* Nb;     // r x n bf16 Adam update of the direction branch
    float* dM;        // m x kb Adam update of the magnitude branch
    uint16_t* Pb;     // m x r bf16 projector
};

struct TcTile {
    int mod, slot, t0, t1;
};

// ------------------------------------------------------------------- K0
struct K0Item {
    const uint16_t* G;
    uint16_t* Vhi;
    uint16_t* Vlo;
    float* mag;                        // m x kb block norms M (written when do_mag, unless Optimizer_M runs in K0)
    float* mag_avg;
    float* mag_avg_sq;
    float* dM;
    int m, n, kb, segs;                // segs = ceil(n / 1024) row segments
};

struct K0Params {
    int count;
    int hilo;                          // also write V_lo = V - V_hi
    int do_mag;                        // K0 without Optimizer_M: store the block norms (off when only V is wanted)
    float decomp_eps, beta1, beta2, adam_eps, bc1, bc2;
    const float* clip;                 // gradient clipping coefficient (device) for M, or null
    long long start[kTcGroup + 1];     // warp items (row, 1024-column segment) per module
    long long mstart[kTcGroup + 1];    // magnitude entries (m x kb) per module, prefix sums
    K0Item p[kTcGroup];
};

// ------------------------------------------------------------------- K1
constexpr int K1_BM = 128, K1_BN = 256, K1_BK = 64;
// Columns of a pair tile where the launch's tiles of 256 would leave half of
// the pairs idle: half the MMAs and half the epilogue per tile.  Above that a
// tile of 128 columns is the slower one: it fetches the projector's rows twice
// as often.  A 1024 / 2816 layer (35 tiles of 256, 76 pairs): 27 us instead of
// 31, its step 66.4 instead of 70.7.
constexpr int K1_BN_NARROW = 128;
constexpr int K1_A_BYTES = K1_BM * K1_BK * 2;           // 16 KB: two 64-rank chunks of P^T (MN-major)
constexpr int K1_B_BYTES = K1_BK * (K1_BN / 2) * 2;     // 16 KB: this CTA's two 64-column chunks of V
// The Adam moments stream through a ring of slots, each one 32-column chunk
// of exp_avg and of exp_avg_sq (128 rank rows x 32 fp32, 16 KB each), loaded
// and stored by TMA.
constexpr int K1_MCOLS = 32;                            // fp32 moments: columns per chunk
constexpr int K1_MCHUNK = K1_BM * K1_MCOLS * 4;          // 16 KB (64 columns of bf16 moments)
// Chunk width in columns for fp32 (SB false) or bf16 (SB true) states: one
// 128-byte row of a 128-row chunk either way.
template <bool SB> struct StateCols { static constexpr int N = SB ? 64 : 32; };
template <bool HILO> struct K1Cfg {
    static constexpr int STAGES = HILO ? 3 : 5;
    static constexpr int STAGE_BYTES = K1_A_BYTES + (HILO ? 2 : 1) * K1_B_BYTES;
    static constexpr int MSLOTS = HILO ? 1 : 2;
    static constexpr int RING = STAGES * STAGE_BYTES;     // offset of the moment slots
    static constexpr int CTL = RING + MSLOTS * 2 * K1_MCHUNK;
};
constexpr int K1_WARPS = 12;                            // 0 TMA, 1 MMA, 2 moment loader, 3 moment storer, 4-11 epilogue
constexpr int K1_THREADS = K1_WARPS * 32;
constexpr int kCtlBytes = 512;                         // barrier block of K1 / K2
constexpr int K1_SMEM = 1024 + (K1Cfg<false>::CTL > K1Cfg<true>::CTL ? K1Cfg<false>::CTL : K1Cfg<true>::CTL) + kCtlBytes;

struct K1Params {
    CUtensorMap gmap[kTcGroup];        // G of each launch slot (decomposition off): {n, m}, box {64, 64}
    const int* cta_start;              // tiles of CTA c: tiles[cta_start[c] .. cta_start[c+1])
    const TcTile* tiles;
    const TcMod* mods;
    const CUtensorMap* maps;           // per module: P (K1), P (K2), N, W, V_hi, V_lo, exp_avg, exp_avg_sq, W (3-D), N_lo
    int* status;
    float beta1, beta2, adam_eps, bc1, bc2;
    float inv_bc1, inv_bc2;            // 1 / bias corrections
    int decompose;
    const float* clip;                 // decomposition off: clipping coefficient (device) for R, or null
};

// ------------------------------------------------------------------- K2
constexpr int K2_BM = 128, K2_BN = 256, K2_BK = 64;
constexpr int K2_A_BYTES = K2_BM * K2_BK * 2;           // 16 KB: P rows, K-major
constexpr int K2_B_BYTES = K2_BK * (K2_BN / 2) * 2;     // 16 KB: this CTA's two 64-column chunks of N
constexpr int K2_STAGE_BYTES = K2_A_BYTES + K2_B_BYTES;
// W moves in 16 KB chunks: 128 rows x one 128-byte row (32 fp32 / 64 bf16
// columns), or for an fp32 W whose n is a multiple of 64, 64 rows x 64
// columns through a 3-D view of W (256 contiguous bytes per row).
// fp32 W (SB false): the epilogue writes the update dW = -lr*alpha*(Rep_B(dM)
// (.) dV) into a staging chunk and a TMA reduce-add applies it to W in L2, so
// W never enters the SM: two staging chunks, six operand stages.  bf16 W (SB
// true; the fp32 update is rounded once, which an L2 add of a bf16 dW would
// not reproduce): a four-chunk ring, TMA in and out, five operand stages.
constexpr int K2_WCOLS = 32;
constexpr int K2_WBYTES = K2_BM * K2_WCOLS * 4;         // 16 KB
// ALIGN (the alignment diagnostic): the product is reduced against G instead of
// applied; N (a right projector: V Q) comes as two planes, the residual in a
// third 16 KB slot of each stage.
template <bool SB, bool ALIGN = false> struct K2Cfg {
    static constexpr int STAGES = ALIGN ? 4 : SB ? 5 : 6;
    static constexpr int STAGE_BYTES = K2_STAGE_BYTES + (ALIGN ? K2_B_BYTES : 0);
    static constexpr int WBUF = ALIGN ? 0 : SB ? 4 : 2;
    static constexpr int BYTES = STAGES * STAGE_BYTES + WBUF * K2_WBYTES;
};
static_assert(K2Cfg<false, true>::BYTES <= K2Cfg<true>::BYTES, "the alignment stages fit K2's shared memory");
constexpr int K2_WARPS = 12;                            // 0 TMA, 1 MMA, 2 W loader, 3 W storer, 4-11 epilogue
constexpr int K2_THREADS = K2_WARPS * 32;
constexpr int K2_SMEM = 1024 + (K2Cfg<true>::BYTES > K2Cfg<false>::BYTES ? K2Cfg<true>::BYTES : K2Cfg<false>::BYTES) +
                        kCtlBytes;

struct K2Params {
    const int* cta_start;
    const TcTile* tiles;
    const TcMod* mods;
    const CUtensorMap* maps;
    int* status;
    float step_scale;                  // lr * alpha
    int decompose;
};

// The diagnostic takes the step's work list of its modules where there is one or
// one can be made.  Otherwise (count > 0: a graph is being recorded, which allows
// no allocation, or the context keeps kAlignLists of them already)
// the tiles are numbered through the modules, in descending K, and dealt to the
// clusters in turn, back and forth.  Without lists at all, four weights of 288 to
// 7264 columns (312 tiles) took 129 us instead of 126: a few tiles per cluster
// need the longest-first assignment, and the first touch of each line of the
// parameter block is a miss.  (The lists in the parameter block, 30 KB of it: one
// 500 x 1744 weight 35.6 us instead of 33.5.)
constexpr int kAlignLists = 64;
struct K2AlignParams : K2Params {
    const uint16_t* G[kTcGroup];       // gradient of each launch slot (m x n)
    double* acc;                       // three sums per module of the call: <G, a>, <a, a>, <G, G>
    int count;                         // 0: tiles and slots (places in the call) from the list
    int mod[kTcGroup];                 // module of the slot
    int call_idx[kTcGroup];            // its place in the call
    int col_tiles[kTcGroup];
    int start[kTcGroup + 1];           // first tile of the slot
    long long wait_limit;              // clock cycles of a bounded wait before it gives up
};
static_assert(sizeof(K2AlignParams) <= 32764, "the diagnostic's parameter block fits the kernel parameter space");

struct SmemCtl {
    uint64_t full[8];
    uint64_t empty[8];   // sized for up to eight stages
    uint64_t accf[2];
    uint64_t acce[2];
    uint64_t drain;
    uint64_t wfull[8];
    uint64_t wdone[8];
    uint64_t wempty[8];
    uint32_t tmem_base;
    int abort;
    uint32_t steps;      // stages that this CTA's producer filled (kernels that settle a pair)
};
static_assert(sizeof(SmemCtl) <= kCtlBytes, "the barrier block fits the space K1 and K2 reserve for it");
// K1 and K2 leave room beside them for one K0 CTA (no shared memory of its
// own, 1 KB reserved by the hardware per CTA) out of the SM's 228 KB.
static_assert(K1_SMEM + 1024 + 1024 <= 228 * 1024 && K2_SMEM + 1024 + 1024 <= 228 * 1024,
              "a decomposition CTA fits beside a K1 or K2 CTA");

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
    return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

__device__ __forceinline__ bool wait_drain(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!ptx::mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > kWaitLimit) return false;
    }
    return true;
}

// A pair whose waits may run out while copies are in flight (a wait limit below
// a copy's latency).  A copy of either CTA completes on the even CTA's barrier,
// and a stage's phase ends when both CTAs' copies have landed; the two producers
// may have given up a different number of stages in.
//
// pair_abort, by every warp before the last cluster barrier: if its CTA gave up,
// the peer knows behind that barrier.  pair_settle, by one thread of each CTA
// behind it: the CTA that filled fewer stages fills the missing ones (the MMAs
// are done, what lands there is not used), and the even CTA waits for every
// stage's last phase.  Another cluster barrier, and no copy is left in flight.
__device__ __forceinline__ void pair_abort(SmemCtl* ctl, int crank) {
    if ((threadIdx.x & 31) == 0 && *const_cast<volatile int*>(&ctl->abort) != 0)
        ptx::st_cluster_u32(ptx::mapa(ptx::smem_u32(&ctl->abort), crank ^ 1), 1);
}

template <int STAGES, class Fill>
__device__ __forceinline__ void pair_settle(SmemCtl* ctl, int crank, Fill fill) {
    const uint32_t own = ctl->steps, peer = ptx::ld_cluster_u32(ptx::mapa(ptx::smem_u32(&ctl->steps), crank ^ 1));
    const uint32_t all = own > peer ? own : peer;
    for (uint32_t k = own; k < all; ++k) fill(static_cast<int>(k), static_cast<int>(k % STAGES));
    if (crank == 0)
        for (uint32_t q = 0; q < STAGES && q < all; ++q)
            wait_drain(ptx::smem_u32(&ctl->full[q]), ((all - 1 - q) / STAGES) & 1);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// ===========================================================================
// K0: Decompose(G, B) (§3.1 / App. B.1) and Optimizer_M.  One warp per (row,
// 1024-column segment), taken as four 256-column sub-segments whose loads are
// all issued first; in a sub-segment lane l holds columns 8l..8l+7, so a block
// of B columns spans B/8 lanes, reduced with xor shuffles.  Columns past n (the
// right zero padding of the last block) contribute nothing; V is written for
// c < n only.
// ===========================================================================
constexpr int K0_SEG = 1024;

// One entry of Optimizer_M: the new moments to *ma and *mas, the update returned.
__device__ __forceinline__ float mag_adam(const K0Params& p, float mag, float old_ma, float old_mas, float* ma,
                                          float* mas) {
    const float a = p.beta1 * old_ma + (1.0f - p.beta1) * mag;
    const float s = p.beta2 * old_mas + (1.0f - p.beta2) * mag * mag;
    *ma = a;
    *mas = s;
    return (a / p.bc1) / (sqrtf(s / p.bc2) + p.adam_eps);
}

//
// ADAM (blocks of 32 columns and more): Optimizer_M in the same pass.  The
// item's 32, 16 or 8 block norms go to as many lanes, so that the update is
// one evaluation per item and its moments, loaded with the next item's G, are
// contiguous; the norms themselves are not stored.  As a pass of its own it
// cost a launch and 8 more bytes per norm: the step of a 1024 / 2816 layer went
// from 81.5 to 75.8 us.
template <int BLK, bool ADAM>
__global__ void __launch_bounds__(256, 3) k0_decompose(const __grid_constant__ K0Params p) {
    pdl_begin();
    constexpr int LPB = BLK / 8;                       // lanes per block (1..16)
    constexpr int SUBB = 256 / BLK;                    // blocks of a sub-segment
    static_assert(!ADAM || 4 * SUBB <= 32, "a lane per block of the item");
    const int lane = threadIdx.x & 31;
    const long long total = p.start[p.count];
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    long long item = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    int mod = 0;                                       // module of `item` (items only increase)
    // G of the next item is loaded before the current one is processed, so
    // each warp keeps a 1024-column row segment in flight
    auto locate = [&](long long x, int& row, int& seg) {
        while (mod + 1 < p.count && p.start[mod + 1] <= x) ++mod;
        const int local = static_cast<int>(x - p.start[mod]);
        row = local / p.p[mod].segs;
        seg = local - row * p.p[mod].segs;
    };
    auto load = [&](int md, int row, int seg, uint4 (&g)[4]) {
        const K0Item& it = p.p[md];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c0 = seg * K0_SEG + u * 256 + lane * 8;
            g[u] = make_uint4(0u, 0u, 0u, 0u);
            if (c0 < it.n) g[u] = __ldcs(reinterpret_cast<const uint4*>(it.G + (long long)row * it.n + c0));
        }
    };
    // moments of the item's block `lane`
    auto load_mag = [&](int md, int row, int seg, float& ma, float& mas) {
        const K0Item& it = p.p[md];
        const int b = seg * (4 * SUBB) + lane;
        ma = mas = 0.0f;
        if (lane < 4 * SUBB && b < it.kb) {
            ma = it.mag_avg[(long long)row * it.kb + b];
            mas = it.mag_avg_sq[(long long)row * it.kb + b];
        }
    };
    const float cf = ADAM && p.clip != nullptr ? *p.clip : 1.0f;
    if (item >= total) return;
    int row, seg;
    locate(item, row, seg);
    uint4 g[4];
    float ma = 0.0f, mas = 0.0f;
    load(mod, row, seg, g);
    if (ADAM) load_mag(mod, row, seg, ma, mas);
    while (true) {
        const int cmod = mod, crow = row, cseg = seg;
        const float cma = ma, cmas = mas;
        uint4 cg[4] = {g[0], g[1], g[2], g[3]};
        item += nwarps;
        const bool more = item < total;
        if (more) {
            locate(item, row, seg);
            load(mod, row, seg, g);
            if (ADAM) load_mag(mod, row, seg, ma, mas);
        }
        const K0Item& it = p.p[cmod];
        const int n = it.n;
        float norm = 0.0f;                              // ADAM: of the item's block `lane`
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int cs = cseg * K0_SEG + u * 256;     // first column of the sub-segment
            if (cs >= n) break;                         // warp-uniform
            const int c0 = cs + lane * 8;
            const uint32_t w[4] = {cg[u].x, cg[u].y, cg[u].z, cg[u].w};
            float ss = 0.0f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float a = bf_lo(w[e]), b = bf_hi(w[e]);
                ss = fmaf(a, a, ss);
                ss = fmaf(b, b, ss);
            }
#pragma unroll
            for (int o = 1; o < LPB; o <<= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            const float mag = sqrtf(ss);
            const float sc = 1.0f / (mag + p.decomp_eps);
            if (ADAM) {
                const float x = __shfl_sync(0xffffffffu, mag, (lane % SUBB) * LPB);
                norm = lane / SUBB == u ? x : norm;
            } else if (p.do_mag && (lane & (LPB - 1)) == 0 && c0 < n) {   // first lane of a block that starts before n
                it.mag[(long long)crow * it.kb + c0 / BLK] = mag;
            }
            if (c0 < n) {
                const long long off = (long long)crow * n + c0;
                uint32_t vh[4], vl[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float v0 = bf_lo(w[e]) * sc, v1 = bf_hi(w[e]) * sc;
                    vh[e] = pack_bf16x2(v0, v1);
                    vl[e] = pack_bf16x2(v0 - bf_lo(vh[e]), v1 - bf_hi(vh[e]));
                }
                *reinterpret_cast<uint4*>(it.Vhi + off) = make_uint4(vh[0], vh[1], vh[2], vh[3]);
                if (p.hilo) *reinterpret_cast<uint4*>(it.Vlo + off) = make_uint4(vl[0], vl[1], vl[2], vl[3]);
            }
        }
        if (ADAM) {
            const int b = cseg * (4 * SUBB) + lane;
            if (lane < 4 * SUBB && b < it.kb) {
                const long long o = (long long)crow * it.kb + b;
                it.dM[o] = mag_adam(p, norm * cf, cma, cmas, it.mag_avg + o, it.mag_avg_sq + o);
            }
        }
        if (!more) break;
    }
}

// Optimizer_M (Algorithm 1) on block norms that K0 wrote, as a pass of its own:
// for blocks below 32 columns, and where the clipping coefficient needs every
// norm first.
__global__ void __launch_bounds__(256) k0_mag_adam(const __grid_constant__ K0Params p) {
    pdl_begin();
    const long long total = p.mstart[p.count];
    // a clipped gradient c G has block norms c M and the same direction V
    const float cf = p.clip != nullptr ? *p.clip : 1.0f;
    int mod = 0;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        while (mod + 1 < p.count && p.mstart[mod + 1] <= e) ++mod;
        const K0Item& it = p.p[mod];
        const long long o = e - p.mstart[mod];
        it.dM[o] = mag_adam(p, it.mag[o] * cf, it.mag_avg[o], it.mag_avg_sq[o], it.mag_avg + o, it.mag_avg_sq + o);
    }
}

// Sum of the squared block norms K0 wrote (= ||G||_F^2 of the group, up to
// their rounding) for global-norm clipping: chunks of kNormChunk entries,
// chunk c on CTA c mod gridDim, fp32 per chunk and fp64 across chunks in a
// fixed order, one partial sum per CTA.
__global__ void __launch_bounds__(256) k0_mag_sq(const __grid_constant__ K0Params p, double* partials) {
    __shared__ double red[8];
    const long long total = p.mstart[p.count];
    const long long nchunks = (total + kNormChunk - 1) / kNormChunk;
    double acc = 0.0;
    int mod = 0;
    for (long long c = blockIdx.x; c < nchunks; c += gridDim.x) {
        const long long e0 = c * kNormChunk, e1 = min(e0 + (long long)kNormChunk, total);
        float ss = 0.0f;
        for (long long e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
            while (mod + 1 < p.count && p.mstart[mod + 1] <= e) ++mod;
            while (mod > 0 && p.mstart[mod] > e) --mod;
            const float x = p.p[mod].mag[e - p.mstart[mod]];
            ss = fmaf(x, x, ss);
        }
        acc += static_cast<double>(ss);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        partials[blockIdx.x] = t;
    }
}

// ===========================================================================
// K1: projection R = P^T V (tile 128 ranks x 256 columns x 64 rows, MN-major
// operands), Optimizer_V (Adam) in the epilogue, N written in bf16.  HILO
// adds the MMA with V_lo (first Adam step).
// ===========================================================================
// RT: the launch may hold modules with a right projector (per-tile operand
// roles); without it those branches are compiled out.
template <bool HILO, bool SB, bool RT, int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(K1_THREADS, 1)
k1_project(const __grid_constant__ K1Params p) {
    constexpr int MC = StateCols<SB>::N;              // moment columns per chunk
    constexpr int HC = MC / 2;                        // columns per epilogue thread and chunk
    constexpr int BCH = BN / 128;                     // 64-column chunks of V per CTA
    constexpr int LOADED = K1_A_BYTES + (HILO ? 2 : 1) * BCH * 8192;   // bytes of a stage that are filled (left projector)
    constexpr int STAGES = K1Cfg<HILO>::STAGES;
    constexpr int STAGE_BYTES = K1Cfg<HILO>::STAGE_BYTES;
    constexpr int MSLOTS = K1Cfg<HILO>::MSLOTS;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    uint8_t* mring = smem + K1Cfg<HILO>::RING;
    SmemCtl* ctl = reinterpret_cast<SmemCtl*>(smem + K1Cfg<HILO>::CTL);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int crank = static_cast<int>(ptx::cluster_ctarank());   // rank tile 2 t0 + crank of each pair tile
    const int cluster = blockIdx.x >> 1;
    volatile int* abort_flag = &ctl->abort;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(ptx::smem_u32(&ctl->full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctl->empty[s]), 1);    // the pair MMA consumed the stage
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(ptx::smem_u32(&ctl->accf[b]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctl->acce[b]), 16);    // both CTAs' epilogue warps
        }
        for (int b = 0; b < MSLOTS; ++b) {
            ptx::mbar_init(ptx::smem_u32(&ctl->wfull[b]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctl->wdone[b]), 8);
            ptx::mbar_init(ptx::smem_u32(&ctl->wempty[b]), 1);
        }
        ptx::mbar_init(ptx::smem_u32(&ctl->drain), 1);
        ctl->abort = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 1) {                // collective: one warp of each CTA of the pair
        ptx::tmem_alloc2(ptx::smem_u32(&ctl->tmem_base), 512);
        ptx::tmem_relinquish2();
    }
    ptx::tc_fence_before();
    __syncwarp();
    ptx::cluster_sync();            // barriers of both CTAs initialised before any remote signal
    ptx::tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    const int t_begin = p.cta_start[cluster], t_end = p.cta_start[cluster + 1];
    pdl_begin();

    if (warp == 0) {
        // ------------------------------------------------------ TMA producer
        // P^T rows of this CTA's rank tile and this CTA's half (128 columns)
        // of the V tile: the pair MMA reads A rows and B columns from both.
        // Both CTAs' copies complete on the even CTA's full barrier, which
        // the even CTA arms with the bytes of both.
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t issued = 0, last_par = 0;
            bool ok = true;
            for (int t = t_begin; t < t_end && ok; ++t) {
                const TcTile tl = p.tiles[t];
                const TcMod& md = p.mods[tl.mod];
                const CUtensorMap* pmap = &p.maps[tl.mod * kMaps + 0];
                const CUtensorMap* vmap = p.decompose ? &p.maps[tl.mod * kMaps + 4] : &p.gmap[tl.slot];
                const CUtensorMap* lmap = &p.maps[tl.mod * kMaps + 5];
                const int r0 = (2 * tl.t0 + crank) * K1_BM, n0 = tl.t1 * BN;
                const bool right = RT && md.right != 0;
                const int nk = ((right ? md.n : md.m) + K1_BK - 1) / K1_BK;
                for (int kb = 0; kb < nk; ++kb) {
                    if (!ptx::mbar_wait(ptx::smem_u32(&ctl->empty[stage]), phase ^ 1, abort_flag, p.status,
                                        MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit)) { ok = false; break; }
                    const uint32_t own = ptx::smem_u32(&ctl->full[stage]);
                    const uint32_t fb = ptx::mapa(own, 0);
                    // a right projector's V_lo is as long as its V (128 rows)
                    if (crank == 0)
                        ptx::mbar_arrive_expect_tx(own, 2 * (right ? K1_A_BYTES * (HILO ? 2 : 1) + BCH * 8192 : LOADED));
                    const uint32_t a = ptx::smem_u32(smem + stage * STAGE_BYTES);
                    const uint32_t b = a + K1_A_BYTES;
                    if (!right) {
#pragma unroll
                        for (int c = 0; c < 2; ++c) ptx::tma_load_2d_pair(a + c * 8192, pmap, fb, r0 + 64 * c, kb * K1_BK);
#pragma unroll
                        for (int h = 0; h < BCH; ++h) {
                            const int c = BCH * crank + h;
                            ptx::tma_load_2d_pair(b + h * 8192, vmap, fb, n0 + 64 * c, kb * K1_BK);
                            if (HILO) ptx::tma_load_2d_pair(b + K1_B_BYTES + h * 8192, lmap, fb, n0 + 64 * c, kb * K1_BK);
                        }
                    } else {
                        // A: this CTA's 128 rows of V (64 columns, K-major; V_lo
                        // in the third slot at the first step); B: this CTA's
                        // 128 ranks of Q, two 64-rank chunks (MN-major)
                        ptx::tma_load_2d_pair(a, vmap, fb, kb * K1_BK, r0);
                        if (HILO) ptx::tma_load_2d_pair(b + K1_B_BYTES, lmap, fb, kb * K1_BK, r0);
#pragma unroll
                        for (int h = 0; h < BCH; ++h)
                            ptx::tma_load_2d_pair(b + h * 8192, pmap, fb, n0 + 64 * (BCH * crank + h), kb * K1_BK);
                    }
                    issued |= 1u << stage;
                    last_par = (last_par & ~(1u << stage)) | (phase << stage);
                    if (++stage == STAGES) { stage = 0; phase ^= 1; }
                }
            }
            if (!ok && crank == 0) {   // let the copies already in flight land before the CTA exits
                for (int s = 0; s < STAGES; ++s)
                    if (issued & (1u << s)) wait_drain(ptx::smem_u32(&ctl->full[s]), (last_par >> s) & 1);
            }
        }
    } else if (warp == 1) {
        if (crank == 0) {
            // -------------------------------------------- MMA issuer (even CTA)
            // M = 256 (both CTAs' rank tiles), N = 256, K = 16 per MMA; the
            // full barrier of a stage counts both CTAs' copies
            if (lane == 0) {
                constexpr uint32_t idesc_l = ptx::idesc_bf16(256, BN, 1, 1);   // A MN-major (P^T)
                constexpr uint32_t idesc_r = ptx::idesc_bf16(256, BN, 0, 1);   // A K-major (V rows)
                int stage = 0;
                uint32_t phase = 0;
                int buf = 0;
                uint32_t acc_phase = 0;
                bool ok = true;
                for (int t = t_begin; t < t_end && ok; ++t) {
                    const TcTile tl = p.tiles[t];
                    const TcMod& md = p.mods[tl.mod];
                    const bool right = RT && md.right != 0;
                    const uint32_t idesc = right ? idesc_r : idesc_l;
                    const int nk = ((right ? md.n : md.m) + K1_BK - 1) / K1_BK;
                    if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->acce[buf]), acc_phase ^ 1, abort_flag, p.status,
                                                MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit)) { ok = false; break; }
                    ptx::tc_fence_after();
                    const uint32_t d0 = tmem + buf * 256;
                    for (int kb = 0; kb < nk; ++kb) {
                        if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->full[stage]), phase, abort_flag, p.status,
                                                    MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit)) { ok = false; break; }
                        ptx::tc_fence_after();
                        const uint32_t a = ptx::smem_u32(smem + stage * STAGE_BYTES);
                        const uint32_t b = a + K1_A_BYTES;
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            const uint64_t bdesc = ptx::smem_desc_sw128(b + kk * 2048, 8192, 1024);
                            if (!right) {
                                const uint64_t adesc = ptx::smem_desc_sw128(a + kk * 2048, 8192, 1024);
                                ptx::mma2_f16(d0, adesc, bdesc, idesc, (kb | kk) != 0);
                                if (HILO) {   // P^T V_lo: the bf16 rounding residual of V
                                    const uint64_t ldesc = ptx::smem_desc_sw128(b + K1_B_BYTES + kk * 2048, 8192, 1024);
                                    ptx::mma2_f16(d0, adesc, ldesc, idesc, 1);
                                }
                            } else {
                                const uint64_t adesc = ptx::smem_desc_sw128(a + kk * 32, 16, 1024);
                                ptx::mma2_f16(d0, adesc, bdesc, idesc, (kb | kk) != 0);
                                if (HILO) {   // V_lo Q
                                    const uint64_t ldesc = ptx::smem_desc_sw128(b + K1_B_BYTES + kk * 32, 16, 1024);
                                    ptx::mma2_f16(d0, ldesc, bdesc, idesc, 1);
                                }
                            }
                        }
                        ptx::mma2_commit_mc(ptx::smem_u32(&ctl->empty[stage]), 0x3);
                        if (++stage == STAGES) { stage = 0; phase ^= 1; }
                    }
                    if (!ok) break;
                    ptx::mma2_commit_mc(ptx::smem_u32(&ctl->accf[buf]), 0x3);
                    if (++buf == 2) { buf = 0; acc_phase ^= 1; }
                }
                // wait for every MMA this thread issued before TMEM is released
                ptx::mma2_commit_mc(ptx::smem_u32(&ctl->drain), 0x1);
                wait_drain(ptx::smem_u32(&ctl->drain), 0);
            }
        }
    } else if (warp == 2) {
        // ------------------------------------- moment chunk loader (TMA in)
        if (lane == 0) {
            uint32_t g = 0;
            uint32_t issued = 0, last_par = 0;
            bool ok = true;
            for (int t = t_begin; t < t_end && ok; ++t) {
                const TcTile tl = p.tiles[t];
                const TcMod& md = p.mods[tl.mod];
                const CUtensorMap* amap = &p.maps[tl.mod * kMaps + 6];
                const CUtensorMap* smap = &p.maps[tl.mod * kMaps + 7];
                const int r0 = (2 * tl.t0 + crank) * K1_BM, n0 = tl.t1 * BN;
                const int cols = (RT && md.right) ? md.r : md.n;    // R is r x n, or m x r (right projector)
                const int nc = min(BN / MC, (cols - n0 + MC - 1) / MC);
                for (int c = 0; c < nc; ++c, ++g) {
                    const int b = g % MSLOTS;
                    const uint32_t ph = (g / MSLOTS) & 1;
                    if (!ptx::mbar_wait(ptx::smem_u32(&ctl->wempty[b]), ph ^ 1, abort_flag, p.status,
                                        MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit)) { ok = false; break; }
                    const uint32_t fb = ptx::smem_u32(&ctl->wfull[b]);
                    ptx::mbar_arrive_expect_tx(fb, 2 * K1_MCHUNK);
                    const uint32_t dst = ptx::smem_u32(mring + b * 2 * K1_MCHUNK);
                    ptx::tma_load_2d(dst, amap, fb, n0 + c * MC, r0);
                    ptx::tma_load_2d(dst + K1_MCHUNK, smap, fb, n0 + c * MC, r0);
                    issued |= 1u << b;
                    last_par = (last_par & ~(1u << b)) | (ph << b);
                }
            }
            if (!ok) {
                for (int b = 0; b < MSLOTS; ++b)
                    if (issued & (1u << b)) wait_drain(ptx::smem_u32(&ctl->wfull[b]), (last_par >> b) & 1);
            }
        }
    } else if (warp == 3) {
        // ------------------------------------ moment chunk storer (TMA out)
        if (lane == 0) {
            uint32_t g = 0;
            bool ok = true;
            for (int t = t_begin; t < t_end && ok; ++t) {
                const TcTile tl = p.tiles[t];
                const TcMod& md = p.mods[tl.mod];
                const CUtensorMap* amap = &p.maps[tl.mod * kMaps + 6];
                const CUtensorMap* smap = &p.maps[tl.mod * kMaps + 7];
                const int r0 = (2 * tl.t0 + crank) * K1_BM, n0 = tl.t1 * BN;
                const int cols = (RT && md.right) ? md.r : md.n;    // R is r x n, or m x r (right projector)
                const int nc = min(BN / MC, (cols - n0 + MC - 1) / MC);
                for (int c = 0; c < nc; ++c, ++g) {
                    const int b = g % MSLOTS;
                    const uint32_t ph = (g / MSLOTS) & 1;
                    if (!ptx::mbar_wait(ptx::smem_u32(&ctl->wdone[b]), ph, abort_flag, p.status,
                                        MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit)) { ok = false; break; }
                    const uint32_t src = ptx::smem_u32(mring + b * 2 * K1_MCHUNK);
                    ptx::tma_store_2d(amap, src, n0 + c * MC, r0);
                    ptx::tma_store_2d(smap, src + K1_MCHUNK, n0 + c * MC, r0);
                    ptx::bulk_commit_group();
                    ptx::bulk_wait_read_all();            // the slot may be refilled once read
                    ptx::mbar_arrive(ptx::smem_u32(&ctl->wempty[b]));
                }
            }
            ptx::bulk_wait_all();
        }
    } else {
        // ------------------------------------------------- epilogue warps
        // 8 warps: TMEM lane quarter q = warp % 4 (rank row), column half ch
        // of each 32-column chunk.  Optimizer_V (Adam) on R: each thread
        // updates 16 entries of both moments of its rank row in the swizzled
        // ring slot and writes the update N in bf16 to global memory.
        const int ew = warp - 4;                       // 0..7
        const int q = warp & 3;
        const int ch = ew >> 2;
        const int il = q * 32 + lane;                  // rank row within the tile
        // R of a clipped gradient (decomposition off; with it V is unchanged)
        const float cf = p.clip != nullptr ? *p.clip : 1.0f;
        int buf = 0;
        uint32_t acc_phase = 0;
        uint32_t g = 0;
        bool ok = true;
        for (int t = t_begin; t < t_end && ok; ++t) {
            const TcTile tl = p.tiles[t];
            const TcMod& md = p.mods[tl.mod];
            // R (and the moments, N) is r x n, or m x r with a right projector
            const int rr = (RT && md.right) ? md.m : md.r, nn = (RT && md.right) ? md.r : md.n;
            uint16_t* const nb_p = md.Nb;
            const int r0 = (2 * tl.t0 + crank) * K1_BM, n0 = tl.t1 * BN;
            const int a = r0 + il;
            const bool row_ok = a < rr;
            const int nc = min(BN / MC, (nn - n0 + MC - 1) / MC);
            const bool got = ptx::mbar_wait(ptx::smem_u32(&ctl->accf[buf]), acc_phase, abort_flag, p.status,
                                            MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit);
            if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
            ptx::tc_fence_after();
            for (int c = 0; c < nc; ++c, ++g) {
                const int b = g % MSLOTS;
                const uint32_t ph = (g / MSLOTS) & 1;
                const int j0 = n0 + c * MC + ch * HC;
                // the thread's HC columns in passes of 16: four 16-byte units
                // of its row per chunk, 4 fp32 or 8 bf16 moments each
                constexpr int PU = HC / 4;                  // moments per unit
                constexpr int UPH = 16 / PU;                // units per pass
                const uint32_t tcol = tmem + (static_cast<uint32_t>(q * 32) << 16) + buf * 256 + c * MC + ch * HC;
                float v[16];
                __syncwarp();
                ptx::tmem_ld16(tcol, v);
                const bool gotm = ptx::mbar_wait(ptx::smem_u32(&ctl->wfull[b]), ph, abort_flag, p.status,
                                                 MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit);
                if (!__all_sync(0xffffffffu, gotm)) { ok = false; break; }
                uint8_t* arow = mring + b * 2 * K1_MCHUNK + il * 128;
                uint8_t* srow = arow + K1_MCHUNK;
                const uint32_t x = static_cast<uint32_t>(il & 7);
#pragma unroll
                for (int h = 0; h < HC / 16; ++h) {
                    if (h > 0) ptx::tmem_ld16(tcol + 16 * h, v);
                    float nv[16];
#pragma unroll
                    for (int uu = 0; uu < UPH; ++uu) {
                        const int u = h * UPH + uu;
                        const uint32_t off = ((ch * 4 + u) ^ x) << 4;
                        uint4* a4 = reinterpret_cast<uint4*>(arow + off);
                        uint4* s4 = reinterpret_cast<uint4*>(srow + off);
                        const uint4 av = *a4, sv = *s4;
                        const uint32_t aw[4] = {av.x, av.y, av.z, av.w}, sw[4] = {sv.x, sv.y, sv.z, sv.w};
                        float ea[PU], es[PU];
                        if constexpr (SB) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                ea[2 * k] = bf_lo(aw[k]); ea[2 * k + 1] = bf_hi(aw[k]);
                                es[2 * k] = bf_lo(sw[k]); es[2 * k + 1] = bf_hi(sw[k]);
                            }
                        } else {
#pragma unroll
                            for (int k = 0; k < PU; ++k) { ea[k] = __uint_as_float(aw[k]); es[k] = __uint_as_float(sw[k]); }
                        }
#pragma unroll
                        for (int e = 0; e < PU; ++e) {
                            const float rv = v[PU * uu + e] * cf;
                            ea[e] = p.beta1 * ea[e] + (1.0f - p.beta1) * rv;
                            es[e] = p.beta2 * es[e] + (1.0f - p.beta2) * rv * rv;
                            // N goes to K2 in bf16: approximate sqrt / reciprocal
                            // (relative error ~2^-22) are far below its rounding
                            nv[PU * uu + e] = ea[e] * p.inv_bc1 *
                                              ptx::rcp_approx(ptx::sqrt_approx(es[e] * p.inv_bc2) + p.adam_eps);
                        }
                        if constexpr (SB) {   // the moments are stored rounded to bf16
                            *a4 = make_uint4(pack_bf16x2(ea[0], ea[1]), pack_bf16x2(ea[2], ea[3]),
                                             pack_bf16x2(ea[4], ea[5]), pack_bf16x2(ea[6], ea[7]));
                            *s4 = make_uint4(pack_bf16x2(es[0], es[1]), pack_bf16x2(es[2], es[3]),
                                             pack_bf16x2(es[4], es[5]), pack_bf16x2(es[6], es[7]));
                        } else {
                            *a4 = make_uint4(__float_as_uint(ea[0]), __float_as_uint(ea[1]),
                                             __float_as_uint(ea[2]), __float_as_uint(ea[3]));
                            *s4 = make_uint4(__float_as_uint(es[0]), __float_as_uint(es[1]),
                                             __float_as_uint(es[2]), __float_as_uint(es[3]));
                        }
                    }
                    const int jh = j0 + 16 * h;
                    if (row_ok && jh < nn) {
                        const long long o = (long long)a * nn + jh;
                        if (jh + 16 <= nn) {
                            uint4* n4 = reinterpret_cast<uint4*>(nb_p + o);
                            n4[0] = make_uint4(pack_bf16x2(nv[0], nv[1]), pack_bf16x2(nv[2], nv[3]),
                                               pack_bf16x2(nv[4], nv[5]), pack_bf16x2(nv[6], nv[7]));
                            n4[1] = make_uint4(pack_bf16x2(nv[8], nv[9]), pack_bf16x2(nv[10], nv[11]),
                                               pack_bf16x2(nv[12], nv[13]), pack_bf16x2(nv[14], nv[15]));
                        } else {
#pragma unroll
                            for (int e = 0; e < 16; ++e) {
                                if (jh + e >= nn) continue;
                                __nv_bfloat16 hb = __float2bfloat16_rn(nv[e]);
                                nb_p[o + e] = *reinterpret_cast<uint16_t*>(&hb);
                            }
                        }
                    }
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&ctl->wdone[b]));
            }
            if (!ok) break;
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) {   // the even CTA's issuer waits for both CTAs' epilogues
                if (crank == 0) ptx::mbar_arrive(ptx::smem_u32(&ctl->acce[buf]));
                else ptx::mbar_arrive_remote(ptx::mapa(ptx::smem_u32(&ctl->acce[buf]), 0));
            }
            if (++buf == 2) { buf = 0; acc_phase ^= 1; }
        }
    }

    ptx::tc_fence_before();
    __syncwarp();
    ptx::cluster_sync();            // no CTA leaves while its peer may still signal or fill it
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc2(tmem, 512);
    }
}

// ===========================================================================
// K2: back-projection dV = P N and the weight update in the epilogue.
// ===========================================================================
// ALIGN: S(W, t) of §3.2 instead of the update: each entry of P N (or N Q^T,
// with N = R in two planes) times its block norm M is dotted with G.  The
// reduction of a tile runs beside the next tile's MMAs, and a thread reads its
// row of G 16 entries at a time, the next ones before it needs them.  (As a
// transposed product with one tile per CTA, whose reduction read G down its
// columns after the MMAs, two layers' 4096 / 11008 diagnostic took 4.72 ms;
// now 2.84 ms.)
template <int BLK, bool SB, bool ALIGN = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(K2_THREADS, 1)
k2_backproject(const __grid_constant__ typename std::conditional<ALIGN, K2AlignParams, K2Params>::type p) {
    constexpr int WC = StateCols<SB>::N;              // W columns per ring chunk
    constexpr int HC = WC / 2;                        // columns per epilogue thread and chunk
    // fp32 W, blocks of >= 32 columns: 64 x 64 update chunks through the 3-D
    // map where the module allows it (TcMod::w3d)
    constexpr bool W3D = !ALIGN && !SB && BLK >= 32 && K2_BN % BLK == 0;
    static_assert(!SB || BLK >= 32, "bf16 states: a thread's 32 columns lie in one block");
    constexpr int K2_STAGES = K2Cfg<SB, ALIGN>::STAGES, K2_WBUF = ALIGN ? 1 : K2Cfg<SB>::WBUF;
    constexpr int STAGE_BYTES = K2Cfg<SB, ALIGN>::STAGE_BYTES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    uint8_t* wring = smem + K2_STAGES * STAGE_BYTES;
    SmemCtl* ctl = reinterpret_cast<SmemCtl*>(smem + K2Cfg<SB, ALIGN>::BYTES);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int crank = static_cast<int>(ptx::cluster_ctarank());   // row tile 2 t0 + crank of each pair tile
    const int cluster = blockIdx.x >> 1;
    volatile int* abort_flag = &ctl->abort;

    if (threadIdx.x == 0) {
        for (int s = 0; s < K2_STAGES; ++s) {
            ptx::mbar_init(ptx::smem_u32(&ctl->full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctl->empty[s]), 1);    // the pair MMA consumed the stage
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(ptx::smem_u32(&ctl->accf[b]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctl->acce[b]), 16);    // both CTAs' epilogue warps
        }
        for (int b = 0; b < K2_WBUF; ++b) {
            ptx::mbar_init(ptx::smem_u32(&ctl->wfull[b]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctl->wdone[b]), 8);
            ptx::mbar_init(ptx::smem_u32(&ctl->wempty[b]), 1);
        }
        ptx::mbar_init(ptx::smem_u32(&ctl->drain), 1);
        ctl->abort = 0;
        ctl->steps = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 1) {                // collective: one warp of each CTA of the pair
        ptx::tmem_alloc2(ptx::smem_u32(&ctl->tmem_base), 512);
        ptx::tmem_relinquish2();
    }
    ptx::tc_fence_before();
    __syncwarp();
    ptx::cluster_sync();            // barriers of both CTAs initialised before any remote signal
    ptx::tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    int t_begin = 0, t_end = 0;
    bool in_turn = false;
    if constexpr (ALIGN) in_turn = p.count > 0;
    if (!in_turn) {
        t_begin = p.cta_start[cluster];
        t_end = p.cta_start[cluster + 1];
    } else if constexpr (ALIGN) {
        const int total = p.start[p.count], g = static_cast<int>(gridDim.x >> 1);
        t_end = total / g;
        t_end += t_end * g + (t_end & 1 ? g - 1 - cluster : cluster) < total;
    }
    // the cluster's tile t; slot: where the last one lay (in turn they go up)
    auto tile_of = [&](int t, int& slot) {
        if constexpr (ALIGN) {
            if (in_turn) {
                const int g = static_cast<int>(gridDim.x >> 1);
                const int e = t * g + (t & 1 ? g - 1 - cluster : cluster);
                while (e >= p.start[slot + 1]) ++slot;
                const int local = e - p.start[slot], nt = p.col_tiles[slot];
                return TcTile{p.mod[slot], slot, local / nt, local % nt};
            }
        }
        return p.tiles[t];
    };
    int slot = 0;
    long long limit = kWaitLimit;                     // of the waits that the diagnostic's roles share
    if constexpr (ALIGN) limit = p.wait_limit;
    // this CTA's copies of k-step kb of the tile at row i0, column n0 into a stage
    auto fill = [&](const CUtensorMap* amap, const CUtensorMap* bmap, const CUtensorMap* lmap, bool right, int i0, int n0,
                    int kb, int stage) {
        const uint32_t own = ptx::smem_u32(&ctl->full[stage]);
        const uint32_t fb = ptx::mapa(own, 0);
        if (crank == 0) ptx::mbar_arrive_expect_tx(own, 2 * STAGE_BYTES);
        const uint32_t a = ptx::smem_u32(smem + stage * STAGE_BYTES);
        const uint32_t b = a + K2_A_BYTES;
        ptx::tma_load_2d_pair(a, amap, fb, kb * K2_BK, i0);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = 2 * crank + h;
            ptx::tma_load_2d_pair(b + h * 8192, bmap, fb, n0 + 64 * c, kb * K2_BK);
            if (ALIGN && !right)
                ptx::tma_load_2d_pair(b + K2_B_BYTES + h * 8192, lmap, fb, n0 + 64 * c, kb * K2_BK);
        }
        if (right) ptx::tma_load_2d_pair(b + K2_B_BYTES, lmap, fb, kb * K2_BK, i0);
    };
    pdl_begin();

    if (warp == 0) {
        // ------------------------------------------------ operand TMA producer
        // P rows of this CTA's row tile and this CTA's half (128 columns) of
        // the N tile; both CTAs' copies complete on the even CTA's barrier.
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t issued = 0, last_par = 0, steps = 0;
            bool ok = true;
            for (int t = t_begin; t < t_end && ok; ++t) {
                const TcTile tl = tile_of(t, slot);
                const TcMod& md = p.mods[tl.mod];
                const CUtensorMap* amap = &p.maps[tl.mod * kMaps + 1];
                const CUtensorMap* bmap = &p.maps[tl.mod * kMaps + 2];
                const CUtensorMap* lmap = &p.maps[tl.mod * kMaps + 9];
                const bool right = ALIGN && md.right != 0;
                const int i0 = (2 * tl.t0 + crank) * K2_BM, n0 = tl.t1 * K2_BN;
                const int nk = (md.r + K2_BK - 1) / K2_BK;
                for (int kb = 0; kb < nk; ++kb) {
                    if (!ptx::mbar_wait(ptx::smem_u32(&ctl->empty[stage]), phase ^ 1, abort_flag, p.status,
                                        MOARA_ERR_DEVICE_TIMEOUT, limit)) { ok = false; break; }
                    fill(amap, bmap, lmap, right, i0, n0, kb, stage);
                    ++steps;
                    issued |= 1u << stage;
                    last_par = (last_par & ~(1u << stage)) | (phase << stage);
                    if (++stage == K2_STAGES) { stage = 0; phase ^= 1; }
                }
            }
            if (ALIGN) ctl->steps = steps;
            if (!ALIGN && !ok && crank == 0) {
                for (int s = 0; s < K2_STAGES; ++s)
                    if (issued & (1u << s)) wait_drain(ptx::smem_u32(&ctl->full[s]), (last_par >> s) & 1);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------ MMA issuer (even CTA)
        // M = 256 (both CTAs' row tiles), N = 256, K = 16 per MMA
        if (crank == 0 && lane == 0) {
            constexpr uint32_t idesc = ptx::idesc_bf16(256, K2_BN, 0, 1);
            int stage = 0;
            uint32_t phase = 0;
            int buf = 0;
            uint32_t acc_phase = 0;
            bool ok = true;
            for (int t = t_begin; t < t_end && ok; ++t) {
                const TcTile tl = tile_of(t, slot);
                const TcMod& md = p.mods[tl.mod];
                const int nk = (md.r + K2_BK - 1) / K2_BK;
                const bool right = ALIGN && md.right != 0;
                if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->acce[buf]), acc_phase ^ 1, abort_flag, p.status,
                                            MOARA_ERR_DEVICE_TIMEOUT, limit)) { ok = false; break; }
                ptx::tc_fence_after();
                const uint32_t d0 = tmem + buf * 256;
                for (int kb = 0; kb < nk; ++kb) {
                    if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->full[stage]), phase, abort_flag, p.status,
                                                MOARA_ERR_DEVICE_TIMEOUT, limit)) { ok = false; break; }
                    ptx::tc_fence_after();
                    const uint32_t a = ptx::smem_u32(smem + stage * STAGE_BYTES);
                    const uint32_t b = a + K2_A_BYTES;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const uint64_t adesc = ptx::smem_desc_sw128(a + kk * 32, 16, 1024);
                        const uint64_t bdesc = ptx::smem_desc_sw128(b + kk * 2048, 8192, 1024);
                        ptx::mma2_f16(d0, adesc, bdesc, idesc, (kb | kk) != 0);
                        if constexpr (ALIGN) {   // the residual plane, of N (K-major rows with a right projector)
                            if (!right)
                                ptx::mma2_f16(d0, adesc, ptx::smem_desc_sw128(b + K2_B_BYTES + kk * 2048, 8192, 1024),
                                              idesc, 1);
                            else
                                ptx::mma2_f16(d0, ptx::smem_desc_sw128(b + K2_B_BYTES + kk * 32, 16, 1024), bdesc,
                                              idesc, 1);
                        }
                    }
                    ptx::mma2_commit_mc(ptx::smem_u32(&ctl->empty[stage]), 0x3);
                    if (++stage == K2_STAGES) { stage = 0; phase ^= 1; }
                }
                if (!ok) break;
                ptx::mma2_commit_mc(ptx::smem_u32(&ctl->accf[buf]), 0x3);
                if (++buf == 2) { buf = 0; acc_phase ^= 1; }
            }
            ptx::mma2_commit_mc(ptx::smem_u32(&ctl->drain), 0x1);
            wait_drain(ptx::smem_u32(&ctl->drain), 0);
        }
    } else if (warp == 2) {
        // ------------------------------------------- W chunk loader (TMA in)
        // (bf16 W only: an fp32 W is updated by reduce-add, never loaded)
        if (SB && !ALIGN && lane == 0) {
            uint32_t g = 0;
            uint32_t issued = 0, last_par = 0;
            bool ok = true;
            for (int t = t_begin; t < t_end && ok; ++t) {
                const TcTile tl = p.tiles[t];
                const TcMod& md = p.mods[tl.mod];
                const CUtensorMap* wmap = &p.maps[tl.mod * kMaps + 3];
                const int i0 = (2 * tl.t0 + crank) * K2_BM, n0 = tl.t1 * K2_BN;
                const int nc = min(K2_BN / WC, (md.n - n0 + WC - 1) / WC);
                for (int c = 0; c < nc; ++c, ++g) {
                    const int b = g % K2_WBUF;
                    const uint32_t ph = (g / K2_WBUF) & 1;
                    if (!ptx::mbar_wait(ptx::smem_u32(&ctl->wempty[b]), ph ^ 1, abort_flag, p.status,
                                        MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit)) { ok = false; break; }
                    const uint32_t fb = ptx::smem_u32(&ctl->wfull[b]);
                    ptx::mbar_arrive_expect_tx(fb, K2_WBYTES);
                    ptx::tma_load_2d(ptx::smem_u32(wring + b * K2_WBYTES), wmap, fb, n0 + c * WC, i0);
                    issued |= 1u << b;
                    last_par = (last_par & ~(1u << b)) | (ph << b);
                }
            }
            if (!ok) {
                for (int b = 0; b < K2_WBUF; ++b)
                    if (issued & (1u << b)) wait_drain(ptx::smem_u32(&ctl->wfull[b]), (last_par >> b) & 1);
            }
        }
    } else if (warp == 3) {
        // ------------------------------ W chunk storer (TMA store / reduce-add)
        if (!ALIGN && lane == 0) {
            uint32_t g = 0;
            bool ok = true;
            for (int t = t_begin; t < t_end && ok; ++t) {
                const TcTile tl = p.tiles[t];
                const TcMod& md = p.mods[tl.mod];
                const CUtensorMap* wmap = &p.maps[tl.mod * kMaps + 3];
                const int i0 = (2 * tl.t0 + crank) * K2_BM, n0 = tl.t1 * K2_BN;
                const bool w3 = W3D && md.w3d;
                const int nc = w3 ? 2 * min(K2_BN / 64, (md.n - n0) / 64) : min(K2_BN / WC, (md.n - n0 + WC - 1) / WC);
                for (int c = 0; c < nc; ++c, ++g) {
                    const int b = g % K2_WBUF;
                    const uint32_t ph = (g / K2_WBUF) & 1;
                    if (!ptx::mbar_wait(ptx::smem_u32(&ctl->wdone[b]), ph, abort_flag, p.status,
                                        MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit)) { ok = false; break; }
                    const uint32_t src = ptx::smem_u32(wring + b * K2_WBYTES);
                    if constexpr (SB) ptx::tma_store_2d(wmap, src, n0 + c * WC, i0);
                    else if (w3) ptx::tma_reduce_add_3d(&p.maps[tl.mod * kMaps + 8], src, 0,
                                                        (n0 + 64 * (c % (nc / 2))) / 32, i0 + 64 * (c / (nc / 2)));
                    else ptx::tma_reduce_add_2d(wmap, src, n0 + c * WC, i0);
                    ptx::bulk_commit_group();
                    ptx::bulk_wait_read_all();            // the chunk may be refilled once read
                    ptx::mbar_arrive(ptx::smem_u32(&ctl->wempty[b]));
                }
            }
            ptx::bulk_wait_all();
        }
    } else if constexpr (ALIGN) {
        // ------------------------------------ epilogue warps (alignment)
        // 8 warps: TMEM lane quarter q = warp % 4, column half ch of the tile
        const int q = warp & 3, ch = (warp - 4) >> 2;
        const int il = q * 32 + lane;
        int buf = 0;
        uint32_t acc_phase = 0;
        for (int t = t_begin; t < t_end; ++t) {
            const TcTile tl = tile_of(t, slot);
            const TcMod& md = p.mods[tl.mod];
            const int nn = md.n, mkb = md.kb;
            const int i = (2 * tl.t0 + crank) * K2_BM + il, c0 = tl.t1 * K2_BN + ch * (K2_BN / 2);
            const bool row_ok = i < md.m;
            const uint16_t* const grow = p.G[tl.slot] + (long long)i * nn;
            const float* const mrow = md.mag + (long long)i * mkb;
            // 16 entries of this row of G and the norms of their blocks (n is
            // a multiple of 8; zero past n)
            constexpr int NM = BLK >= 16 ? 1 : 16 / BLK;
            auto load = [&](int c, uint4 (&g)[2], float (&mg)[NM]) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    g[h] = make_uint4(0u, 0u, 0u, 0u);
                    if (row_ok && c + 8 * h < nn) g[h] = __ldg(reinterpret_cast<const uint4*>(grow + c + 8 * h));
                }
#pragma unroll
                for (int d = 0; d < NM; ++d)
                    mg[d] = row_ok && c + d * BLK < nn ? __ldg(mrow + (c + d * BLK) / BLK) : 0.0f;
            };
            uint4 g[2], gn[2];
            float mg[NM], mgn[NM];
            load(c0, g, mg);
            const bool got = ptx::mbar_wait(ptx::smem_u32(&ctl->accf[buf]), acc_phase, abort_flag, p.status,
                                            MOARA_ERR_DEVICE_TIMEOUT, limit);
            if (!__all_sync(0xffffffffu, got)) break;
            ptx::tc_fence_after();
            float dot = 0.0f, na = 0.0f, gg = 0.0f;
#pragma unroll 1
            for (int c = 0; c < K2_BN / 2; c += 16) {
                if (c0 + c >= nn) break;                   // warp-uniform
                load(c0 + c + 16, gn, mgn);                // zeros past the tile's half are not used
                float v[16];
                __syncwarp();
                ptx::tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) + buf * 256 + ch * (K2_BN / 2) + c, v);
                const uint32_t w[8] = {g[0].x, g[0].y, g[0].z, g[0].w, g[1].x, g[1].y, g[1].z, g[1].w};
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float x = bf_lo(w[e]), y = bf_hi(w[e]);
                    const float m = mg[NM == 1 ? 0 : 2 * e / BLK];
                    // columns past n: G and the product's columns are zero
                    const float a0 = m * v[2 * e], a1 = m * v[2 * e + 1];
                    dot = fmaf(x, a0, dot);
                    dot = fmaf(y, a1, dot);
                    na = fmaf(a0, a0, na);
                    na = fmaf(a1, a1, na);
                    gg = fmaf(x, x, gg);
                    gg = fmaf(y, y, gg);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) g[h] = gn[h];
#pragma unroll
                for (int d = 0; d < NM; ++d) mg[d] = mgn[d];
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) {   // the even CTA's issuer waits for both CTAs' epilogues
                if (crank == 0) ptx::mbar_arrive(ptx::smem_u32(&ctl->acce[buf]));
                else ptx::mbar_arrive_remote(ptx::mapa(ptx::smem_u32(&ctl->acce[buf]), 0));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                dot += __shfl_xor_sync(0xffffffffu, dot, o);
                na += __shfl_xor_sync(0xffffffffu, na, o);
                gg += __shfl_xor_sync(0xffffffffu, gg, o);
            }
            if (lane == 0) {
                double* acc = p.acc + 3 * (in_turn ? p.call_idx[tl.slot] : tl.slot);
                atomicAdd(acc + 0, static_cast<double>(dot));
                atomicAdd(acc + 1, static_cast<double>(na));
                atomicAdd(acc + 2, static_cast<double>(gg));
            }
            if (++buf == 2) { buf = 0; acc_phase ^= 1; }
        }
    } else {
        // ------------------------------------------------- epilogue warps
        // 8 warps: TMEM lane quarter q = warp % 4, column half ch of each
        // chunk (32 fp32 / 64 bf16 columns); each thread handles 16 / 32
        // values of its W row in the swizzled shared-memory chunk: the update
        // dW = -lr * alpha * dM * (P N) for an fp32 W (added to W by the
        // storer's reduce), or W - lr * alpha * dM * (P N) rounded to bf16.
        const int ew = warp - 4;                        // 0..7
        const int q = warp & 3;
        const int ch = ew >> 2;
        const int il = q * 32 + lane;                   // row within the tile
        constexpr int NDM = BLK >= 16 ? 1 : 16 / BLK;   // dM values per thread and chunk
        constexpr bool HOIST = BLK >= 32 && K2_BN % BLK == 0;
        int buf = 0;
        uint32_t acc_phase = 0;
        uint32_t g = 0;
        bool ok = true;
        for (int t = t_begin; t < t_end && ok; ++t) {
            const TcTile tl = p.tiles[t];
            const TcMod& md = p.mods[tl.mod];
            const int mm = md.m, nn = md.n, mkb = md.kb;
            const float* const dMp = md.dM;
            const int i0 = (2 * tl.t0 + crank) * K2_BM, n0 = tl.t1 * K2_BN;
            const int i = i0 + il;
            const bool row_ok = i < mm;
            const bool w3 = W3D && md.w3d;
            const int nc = w3 ? 2 * min(K2_BN / 64, (nn - n0) / 64) : min(K2_BN / WC, (nn - n0 + WC - 1) / WC);
            // blocks of B >= 32 columns: the tile's dM values of this row are
            // loaded once, before the wait for the accumulator
            float dmt[HOIST ? K2_BN / BLK : 1];
            if (HOIST) {
#pragma unroll
                for (int d = 0; d < K2_BN / BLK; ++d) {
                    const int jb = n0 / BLK + d;
                    dmt[d] = (p.decompose && row_ok && jb < mkb) ? dMp[(long long)i * mkb + jb] : 1.0f;
                }
            }
            const bool got = ptx::mbar_wait(ptx::smem_u32(&ctl->accf[buf]), acc_phase, abort_flag, p.status,
                                            MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit);
            if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
            ptx::tc_fence_after();
            for (int c = 0; c < nc; ++c, ++g) {
                const int b = g % K2_WBUF;
                const uint32_t ph = (g / K2_WBUF) & 1;
                if constexpr (W3D) {
                    if (w3) {
                        // chunk c: rows 64 hq .. + 63 and columns 64 cq .. + 63 of the
                        // tile, hq = c / (nc / 2), cq = c % (nc / 2): a row half's chunks
                        // go out one after the other, so the reduces of a tile's rows
                        // cover their whole width in turn (K2 per two 7B layers 0.701 ->
                        // 0.690 ms against alternating row halves).  The four warps of
                        // that row half write it (warp ch: the 32-column group ch, one
                        // 128-byte line per row; two lines of a warp's store share a
                        // bank group); the other four only pass the chunk's barriers
                        const int ncq = nc / 2;
                        const bool mine = (c / ncq) == (q >> 1);
                        const int cb = (c % ncq) * 64 + ch * 32;
                        float v[32];
                        if (mine) {
                            __syncwarp();
                            const uint32_t ta = tmem + (static_cast<uint32_t>(q * 32) << 16) + buf * 256 + cb;
                            ptx::tmem_ld16(ta, *reinterpret_cast<float(*)[16]>(v));
                            ptx::tmem_ld16(ta + 16, *reinterpret_cast<float(*)[16]>(v + 16));
                        }
                        const bool gotw = ptx::mbar_wait(ptx::smem_u32(&ctl->wempty[b]), ph ^ 1, abort_flag, p.status,
                                                         MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit);
                        if (!__all_sync(0xffffffffu, gotw)) { ok = false; break; }
                        if (mine) {
                            float d0 = dmt[0];
#pragma unroll
                            for (int d = 1; d < K2_BN / BLK; ++d) d0 = (cb >= d * BLK) ? dmt[d] : d0;
                            const float ms = -p.step_scale;
                            const int ln = (32 * (q & 1) + lane) * 2 + ch;    // box line: row * 2 + group
                            uint8_t* line = wring + b * K2_WBYTES + ln * 128;
                            const uint32_t x = static_cast<uint32_t>(ln & 7);
#pragma unroll
                            for (int u = 0; u < 8; ++u)
                                *reinterpret_cast<uint4*>(line + ((u ^ x) << 4)) =
                                    make_uint4(__float_as_uint(ms * (d0 * v[4 * u + 0])),
                                               __float_as_uint(ms * (d0 * v[4 * u + 1])),
                                               __float_as_uint(ms * (d0 * v[4 * u + 2])),
                                               __float_as_uint(ms * (d0 * v[4 * u + 3])));
                        }
                        ptx::fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&ctl->wdone[b]));
                        continue;
                    }
                }
                const int j0 = n0 + c * WC + ch * HC;
                float dm[NDM];
                if (HOIST) {
                    // the thread's 16 (32) columns of the chunk lie in one block
                    const int cb = c * WC + ch * HC;
                    dm[0] = dmt[0];
#pragma unroll
                    for (int d = 1; d < K2_BN / BLK; ++d) dm[0] = (cb >= d * BLK) ? dmt[d] : dm[0];
                } else {
#pragma unroll
                    for (int d = 0; d < NDM; ++d) {
                        const int jb = (j0 + 8 * d) / BLK;
                        dm[d] = (p.decompose && row_ok && jb < mkb) ? dMp[(long long)i * mkb + jb] : 1.0f;
                    }
                }
                float v[HC];
                __syncwarp();
#pragma unroll
                for (int h = 0; h < HC / 16; ++h)
                    ptx::tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) + buf * 256 + c * WC + ch * HC + 16 * h,
                                   *reinterpret_cast<float(*)[16]>(v + 16 * h));
                // bf16 W: the loaded chunk; fp32 W: a free staging chunk
                const bool gotw = SB ? ptx::mbar_wait(ptx::smem_u32(&ctl->wfull[b]), ph, abort_flag, p.status,
                                                      MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit)
                                     : ptx::mbar_wait(ptx::smem_u32(&ctl->wempty[b]), ph ^ 1, abort_flag, p.status,
                                                      MOARA_ERR_DEVICE_TIMEOUT, kWaitLimit);
                if (!__all_sync(0xffffffffu, gotw)) { ok = false; break; }
                uint8_t* wrow = wring + b * K2_WBYTES + il * 128;
                const uint32_t x = static_cast<uint32_t>(il & 7);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    uint4* w4 = reinterpret_cast<uint4*>(wrow + (((ch * 4 + u) ^ x) << 4));
                    if constexpr (SB) {
                        const uint4 wv = *w4;
                        const float d0 = dm[0];
                        const uint32_t ww[4] = {wv.x, wv.y, wv.z, wv.w};
                        uint32_t out[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const float lo = bf_lo(ww[k]) - p.step_scale * (d0 * v[8 * u + 2 * k]);
                            const float hi = bf_hi(ww[k]) - p.step_scale * (d0 * v[8 * u + 2 * k + 1]);
                            out[k] = pack_bf16x2(lo, hi);
                        }
                        *w4 = make_uint4(out[0], out[1], out[2], out[3]);
                    } else {
                        const float d0 = dm[NDM == 1 ? 0 : (u * 4) / BLK];
                        const float ms = -p.step_scale;
                        *w4 = make_uint4(__float_as_uint(ms * (d0 * v[4 * u + 0])),
                                         __float_as_uint(ms * (d0 * v[4 * u + 1])),
                                         __float_as_uint(ms * (d0 * v[4 * u + 2])),
                                         __float_as_uint(ms * (d0 * v[4 * u + 3])));
                    }
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&ctl->wdone[b]));
            }
            if (!ok) break;
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) {   // the even CTA's issuer waits for both CTAs' epilogues
                if (crank == 0) ptx::mbar_arrive(ptx::smem_u32(&ctl->acce[buf]));
                else ptx::mbar_arrive_remote(ptx::mapa(ptx::smem_u32(&ctl->acce[buf]), 0));
            }
            if (++buf == 2) { buf = 0; acc_phase ^= 1; }
        }
    }

    ptx::tc_fence_before();
    __syncwarp();
    if (ALIGN) pair_abort(ctl, crank);
    __syncwarp();
    ptx::cluster_sync();            // no CTA leaves while its peer may still signal or fill it
    if (ALIGN && *abort_flag) {     // the same in both CTAs
        if (threadIdx.x == 0) {
            // the copies of any k-step do: every stage takes as many bytes
            pair_settle<K2_STAGES>(ctl, crank, [&](int, int stage) {
                int first = 0;
                const TcTile tl = tile_of(t_begin, first);
                const CUtensorMap* maps = &p.maps[tl.mod * kMaps];
                fill(maps + 1, maps + 2, maps + 9, p.mods[tl.mod].right != 0, (2 * tl.t0 + crank) * K2_BM, tl.t1 * K2_BN, 0,
                     stage);
            });
        }
        __syncwarp();
        ptx::cluster_sync();
    }
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc2(tmem, 512);
    }
}

// ---------------------------------------------------------------- host side
// ===========================================================================
// KR: bf16 tensor-core GEMM of the projector refresh (the TruncatedSVD of
// Algorithm 1, computed by randomized subspace iteration after Halko,
// Martinsson and Tropp, 2011 -- this library's choice of method, not the
// paper's): out (M x N) = op(A) B with fp32 accumulation,
// written in fp32 and/or bf16.  A is read K-major (stored M x K) or MN-major
// (stored K x M); A or B may come as two planes hi + lo (two MMAs per k-step
// keep ~16 significant bits, used for V); B is stored K x N (MN-major).
// Used for V^T Q, V Z, the Gram matrices X^T X and the triangular factor
// products X R^-1.  Tile 256 x 256 (two 128-row accumulators in TMEM), BK =
// 64, one tile per CTA: the contractions are long enough that the epilogue
// need not overlap the next tile.  The last column tile issues the MMA with
// N = 64 * ceil(cols / 64), so a ragged N costs at most 48 columns; with
// `ktri` the K loop of column tile n0 stops at n0 + 256 (B upper triangular).
// ===========================================================================
constexpr int KR_BM = 256, KR_BN = 256, KR_BK = 64;
constexpr int KR_PLANE = KR_BM * KR_BK * 2;               // 32 KB: one A plane or the B tile
template <int LO> struct KrCfg {
    static constexpr int STAGES = LO ? 2 : 3;
    static constexpr int STAGE_BYTES = (LO ? 3 : 2) * KR_PLANE;
};
constexpr int KR_WARPS = 10;                              // 0 TMA, 1 MMA, 2-9 epilogue
constexpr int KR_THREADS = KR_WARPS * 32;
constexpr int KR_SMEM = 1024 + 6 * KR_PLANE + 2048;
constexpr int kKrGroup = 64;                              // problems per launch (three maps each in the parameters)

struct KrParams {
    CUtensorMap amap[kKrGroup];        // A_hi, box {64, 64}
    CUtensorMap lmap[kKrGroup];        // A_lo or B_lo (the geometry of A or B), unused without LO
    CUtensorMap bmap[kKrGroup];        // B ({N, K}), box {64, 64}
    float* out[kKrGroup];              // M x N fp32 or null
    uint16_t* out_bf[kKrGroup];        // M x N bf16 or null
    uint16_t* out_lo[kKrGroup];        // M x N bf16 residual (out - bf16(out)) or null
    int M[kKrGroup], N[kKrGroup], K[kKrGroup];
    int ktri[kKrGroup];
    int lower[kKrGroup];               // tiles above the diagonal are skipped
    int tiles_n[kKrGroup];
    int tile_start[kKrGroup + 1];
    int count;
    int* status;
    long long wait_limit;              // clock cycles of a bounded wait before it gives up
};

static_assert(sizeof(KrParams) <= 32764, "KR's parameter block fits the kernel parameter space");

// Columns j0 .. j0 + 15 of one output row (offset ro) in fp32, bf16 and / or as
// a bf16 residual.
__device__ __forceinline__ void kr_store16(float* of, uint16_t* ob, uint16_t* ol, long long ro, int j0, int N,
                                           const float (&v)[16]) {
    if (j0 + 16 <= N) {                       // N % 8 == 0: 16-byte aligned rows
        if (of != nullptr) {
            float4* o4 = reinterpret_cast<float4*>(of + ro + j0);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                o4[e] = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
        }
        if (ob != nullptr) {
            uint4* b4 = reinterpret_cast<uint4*>(ob + ro + j0);
            b4[0] = make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]),
                               pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
            b4[1] = make_uint4(pack_bf16x2(v[8], v[9]), pack_bf16x2(v[10], v[11]),
                               pack_bf16x2(v[12], v[13]), pack_bf16x2(v[14], v[15]));
        }
        if (ol != nullptr) {
            float rl[16];
#pragma unroll
            for (int e = 0; e < 16; ++e)
                rl[e] = v[e] - __bfloat162float(__float2bfloat16_rn(v[e]));
            uint4* l4 = reinterpret_cast<uint4*>(ol + ro + j0);
            l4[0] = make_uint4(pack_bf16x2(rl[0], rl[1]), pack_bf16x2(rl[2], rl[3]),
                               pack_bf16x2(rl[4], rl[5]), pack_bf16x2(rl[6], rl[7]));
            l4[1] = make_uint4(pack_bf16x2(rl[8], rl[9]), pack_bf16x2(rl[10], rl[11]),
                               pack_bf16x2(rl[12], rl[13]), pack_bf16x2(rl[14], rl[15]));
        }
    } else {
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            if (j0 + e >= N) continue;
            if (of != nullptr) of[ro + j0 + e] = v[e];
            const __nv_bfloat16 hb = __float2bfloat16_rn(v[e]);
            if (ob != nullptr) ob[ro + j0 + e] = *reinterpret_cast<const uint16_t*>(&hb);
            if (ol != nullptr) {
                const __nv_bfloat16 lb = __float2bfloat16_rn(v[e] - __bfloat162float(hb));
                ol[ro + j0 + e] = *reinterpret_cast<const uint16_t*>(&lb);
            }
        }
    }
}

// LO: 1 adds the MMA with A's residual plane, 2 with B's.
template <bool KMAJOR, int LO>
__global__ void __launch_bounds__(KR_THREADS, 1) kr_product(const __grid_constant__ KrParams p) {
    constexpr int STAGES = KrCfg<LO>::STAGES;
    constexpr int STAGE_BYTES = KrCfg<LO>::STAGE_BYTES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    SmemCtl* ctl = reinterpret_cast<SmemCtl*>(smem + 6 * KR_PLANE);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &ctl->abort;

    // locate (problem, tile)
    const int tile = blockIdx.x;
    int lo = 0, hi = p.count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.tile_start[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    const int pi = lo;
    const int local = tile - p.tile_start[pi];
    const int M = p.M[pi], N = p.N[pi], K = p.K[pi];
    const int i0 = (local / p.tiles_n[pi]) * KR_BM;
    const int n0 = (local % p.tiles_n[pi]) * KR_BN;
    if (p.lower[pi] && n0 >= i0 + KR_BM) return;     // whole CTA, before any barrier or TMEM
    const int nch = min(4, (N - n0 + 63) / 64);            // 64-column chunks of B in this tile
    const int halves = (M - i0) > 128 ? 2 : 1;
    const int kend = p.ktri[pi] ? min(K, n0 + KR_BN) : K;
    const int nk = (kend + KR_BK - 1) / KR_BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(ptx::smem_u32(&ctl->full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctl->empty[s]), 1);
        }
        ptx::mbar_init(ptx::smem_u32(&ctl->accf[0]), 1);
        ptx::mbar_init(ptx::smem_u32(&ctl->drain), 1);
        ctl->abort = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(&ctl->tmem_base), 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    pdl_begin();

    if (warp == 0) {
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t issued = 0, last_par = 0;
            const uint32_t bytes = (LO == 1 ? 2 : 1) * KR_PLANE + (LO == 2 ? 2 : 1) * nch * 8192;
            for (int kb = 0; kb < nk; ++kb) {
                if (!ptx::mbar_wait(ptx::smem_u32(&ctl->empty[stage]), phase ^ 1, abort_flag, p.status,
                                    MOARA_ERR_DEVICE_TIMEOUT, p.wait_limit))
                    break;
                const uint32_t fb = ptx::smem_u32(&ctl->full[stage]);
                ptx::mbar_arrive_expect_tx(fb, bytes);
                const uint32_t a = ptx::smem_u32(smem + stage * STAGE_BYTES);
                const uint32_t b = a + (LO == 1 ? 2 : 1) * KR_PLANE;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int x = KMAJOR ? kb * KR_BK : i0 + 64 * c;
                    const int y = KMAJOR ? i0 + 64 * c : kb * KR_BK;
                    ptx::tma_load_2d(a + c * 8192, &p.amap[pi], fb, x, y);
                    if (LO == 1) ptx::tma_load_2d(a + KR_PLANE + c * 8192, &p.lmap[pi], fb, x, y);
                }
                for (int c = 0; c < nch; ++c) {
                    ptx::tma_load_2d(b + c * 8192, &p.bmap[pi], fb, n0 + 64 * c, kb * KR_BK);
                    if (LO == 2) ptx::tma_load_2d(b + KR_PLANE + c * 8192, &p.lmap[pi], fb, n0 + 64 * c, kb * KR_BK);
                }
                issued |= 1u << stage;
                last_par = (last_par & ~(1u << stage)) | (phase << stage);
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
            // every copy issued has landed before the CTA may leave (after a
            // wait that gave up elsewhere the MMA may not have consumed them)
            for (int s = 0; s < STAGES; ++s)
                if (issued & (1u << s)) wait_drain(ptx::smem_u32(&ctl->full[s]), (last_par >> s) & 1);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = ptx::idesc_bf16(128, nch * 64, KMAJOR ? 0 : 1, 1);
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = 0; kb < nk; ++kb) {
                if (!ptx::mbar_wait(ptx::smem_u32(&ctl->full[stage]), phase, abort_flag, p.status,
                                    MOARA_ERR_DEVICE_TIMEOUT, p.wait_limit)) break;
                ptx::tc_fence_after();
                const uint32_t a = ptx::smem_u32(smem + stage * STAGE_BYTES);
                const uint32_t b = a + (LO == 1 ? 2 : 1) * KR_PLANE;
                for (int h = 0; h < halves; ++h) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const uint32_t ao = a + h * 16384 + (KMAJOR ? kk * 32 : kk * 2048);
                        const uint64_t adesc = KMAJOR ? ptx::smem_desc_sw128(ao, 16, 1024)
                                                      : ptx::smem_desc_sw128(ao, 8192, 1024);
                        const uint64_t bdesc = ptx::smem_desc_sw128(b + kk * 2048, 8192, 1024);
                        ptx::mma_f16(tmem + h * 256, adesc, bdesc, idesc, (kb | kk) != 0);
                        if (LO == 1) {
                            const uint32_t lo_addr = ao + KR_PLANE;
                            const uint64_t ldesc = KMAJOR ? ptx::smem_desc_sw128(lo_addr, 16, 1024)
                                                          : ptx::smem_desc_sw128(lo_addr, 8192, 1024);
                            ptx::mma_f16(tmem + h * 256, ldesc, bdesc, idesc, 1);
                        } else if (LO == 2) {
                            ptx::mma_f16(tmem + h * 256, adesc,
                                         ptx::smem_desc_sw128(b + KR_PLANE + kk * 2048, 8192, 1024), idesc, 1);
                        }
                    }
                }
                ptx::mma_commit(ptx::smem_u32(&ctl->empty[stage]));
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
            ptx::mma_commit(ptx::smem_u32(&ctl->accf[0]));
            ptx::mma_commit(ptx::smem_u32(&ctl->drain));
            wait_drain(ptx::smem_u32(&ctl->drain), 0);
        }
    } else {
        // 8 epilogue warps: lane quarter q = warp % 4, accumulator half h.
        const int ew = warp - 2;
        const int q = warp & 3;
        const int h = ew >> 2;
        const bool got = ptx::mbar_wait(ptx::smem_u32(&ctl->accf[0]), 0, abort_flag, p.status,
                                        MOARA_ERR_DEVICE_TIMEOUT, p.wait_limit);
        if (__all_sync(0xffffffffu, got) && h < halves) {
            ptx::tc_fence_after();
            const int row = i0 + h * 128 + q * 32 + lane;
            uint16_t* const ol = p.out_lo[pi];
            float* const of = p.out[pi];
            uint16_t* const ob = p.out_bf[pi];
            const long long ro = (long long)row * N;
            for (int c = 0; c < nch * 4; ++c) {
                const int j0 = n0 + c * 16;
                if (j0 >= N) break;                       // warp-uniform
                float v[16];
                __syncwarp();
                ptx::tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) + h * 256 + c * 16, v);
                if (row < M) kr_store16(of, ob, ol, ro, j0, N, v);
            }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, 512);
    }
}

// The same product on 2-CTA pairs: an output tile of 256 x 256 with 128 rows and
// half of B's columns per CTA, so that a k-step takes half as long and each
// operand is fetched once per pair.  For launches that one tile's K outlasts
// (few tiles): 199 Gram tiles of seven modules (K up to 11008) take 81 us
// instead of 110, the products of a 1024 / 2816 layer 25 and 14 instead of 40
// and 21.
// With more tiles than SMs the fixed costs per tile (barriers, TMEM, an
// epilogue that overlaps no MMAs) weigh twice and the single CTA is as fast.
template <int LO> struct KpCfg {
    static constexpr int STAGE_BYTES = (LO ? 3 : 2) * (KR_PLANE / 2);
    static constexpr int STAGES = 6 * KR_PLANE / STAGE_BYTES;
};

template <bool KMAJOR, int LO>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(KR_THREADS, 1) kr_pair(const __grid_constant__ KrParams p) {
    constexpr int STAGES = KpCfg<LO>::STAGES, STAGE_BYTES = KpCfg<LO>::STAGE_BYTES;
    constexpr int PLANE = KR_PLANE / 2;                      // 128 rows of A, or 128 columns of B
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    SmemCtl* ctl = reinterpret_cast<SmemCtl*>(smem + 6 * KR_PLANE);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int crank = static_cast<int>(ptx::cluster_ctarank());
    volatile int* abort_flag = &ctl->abort;

    const int tile = blockIdx.x >> 1;
    int lo = 0, hi = p.count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.tile_start[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    const int pi = lo;
    const int local = tile - p.tile_start[pi];
    const int M = p.M[pi], N = p.N[pi], K = p.K[pi];
    const int i0 = (local / p.tiles_n[pi]) * KR_BM;
    const int n0 = (local % p.tiles_n[pi]) * KR_BN;
    if (p.lower[pi] && n0 >= i0 + KR_BM) return;     // the whole pair, before any barrier or TMEM
    const int r0 = i0 + 128 * crank;
    const int nb = N - n0 > 128 ? 2 : 1;             // 64-column chunks of B per CTA
    const int kend = p.ktri[pi] ? min(K, n0 + KR_BN) : K;
    const int nk = (kend + KR_BK - 1) / KR_BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(ptx::smem_u32(&ctl->full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctl->empty[s]), 1);
        }
        ptx::mbar_init(ptx::smem_u32(&ctl->accf[0]), 1);
        ptx::mbar_init(ptx::smem_u32(&ctl->drain), 1);
        ctl->abort = 0;
        ctl->steps = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 1) {                // collective: one warp of each CTA of the pair
        ptx::tmem_alloc2(ptx::smem_u32(&ctl->tmem_base), 256);
        ptx::tmem_relinquish2();
    }
    ptx::tc_fence_before();
    __syncwarp();
    ptx::cluster_sync();            // barriers of both CTAs initialised before any remote signal
    ptx::tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    pdl_begin();

    // this CTA's copies of k-step kb into a stage
    const uint32_t bytes = (LO == 1 ? 2 : 1) * PLANE + (LO == 2 ? 2 : 1) * nb * 8192;
    auto fill = [&](int kb, int stage) {
        const uint32_t own = ptx::smem_u32(&ctl->full[stage]);
        const uint32_t fb = ptx::mapa(own, 0);
        if (crank == 0) ptx::mbar_arrive_expect_tx(own, 2 * bytes);
        const uint32_t a = ptx::smem_u32(smem + stage * STAGE_BYTES);
        const uint32_t b = a + (LO == 1 ? 2 : 1) * PLANE;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int x = KMAJOR ? kb * KR_BK : r0 + 64 * c;
            const int y = KMAJOR ? r0 + 64 * c : kb * KR_BK;
            ptx::tma_load_2d_pair(a + c * 8192, &p.amap[pi], fb, x, y);
            if (LO == 1) ptx::tma_load_2d_pair(a + PLANE + c * 8192, &p.lmap[pi], fb, x, y);
        }
        for (int c = 0; c < nb; ++c) {
            const int x = n0 + 64 * (nb * crank + c);
            ptx::tma_load_2d_pair(b + c * 8192, &p.bmap[pi], fb, x, kb * KR_BK);
            if (LO == 2) ptx::tma_load_2d_pair(b + PLANE + c * 8192, &p.lmap[pi], fb, x, kb * KR_BK);
        }
    };

    if (warp == 0) {
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0, steps = 0;
            for (int kb = 0; kb < nk; ++kb) {
                if (!ptx::mbar_wait(ptx::smem_u32(&ctl->empty[stage]), phase ^ 1, abort_flag, p.status,
                                    MOARA_ERR_DEVICE_TIMEOUT, p.wait_limit)) break;
                fill(kb, stage);
                ++steps;
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
            ctl->steps = steps;
        }
    } else if (warp == 1) {
        if (crank == 0 && lane == 0) {
            const uint32_t idesc = ptx::idesc_bf16(256, nb * 128, KMAJOR ? 0 : 1, 1);
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = 0; kb < nk; ++kb) {
                if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->full[stage]), phase, abort_flag, p.status,
                                            MOARA_ERR_DEVICE_TIMEOUT, p.wait_limit)) break;
                ptx::tc_fence_after();
                const uint32_t a = ptx::smem_u32(smem + stage * STAGE_BYTES);
                const uint32_t b = a + (LO == 1 ? 2 : 1) * PLANE;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint32_t ao = a + (KMAJOR ? kk * 32 : kk * 2048);
                    const uint64_t adesc = KMAJOR ? ptx::smem_desc_sw128(ao, 16, 1024)
                                                  : ptx::smem_desc_sw128(ao, 8192, 1024);
                    const uint64_t bdesc = ptx::smem_desc_sw128(b + kk * 2048, 8192, 1024);
                    ptx::mma2_f16(tmem, adesc, bdesc, idesc, (kb | kk) != 0);
                    if (LO == 1) {
                        const uint64_t ldesc = KMAJOR ? ptx::smem_desc_sw128(ao + PLANE, 16, 1024)
                                                      : ptx::smem_desc_sw128(ao + PLANE, 8192, 1024);
                        ptx::mma2_f16(tmem, ldesc, bdesc, idesc, 1);
                    } else if (LO == 2) {
                        ptx::mma2_f16(tmem, adesc, ptx::smem_desc_sw128(b + PLANE + kk * 2048, 8192, 1024), idesc, 1);
                    }
                }
                ptx::mma2_commit_mc(ptx::smem_u32(&ctl->empty[stage]), 0x3);
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
            ptx::mma2_commit_mc(ptx::smem_u32(&ctl->accf[0]), 0x3);
            ptx::mma2_commit_mc(ptx::smem_u32(&ctl->drain), 0x1);
            wait_drain(ptx::smem_u32(&ctl->drain), 0);
        }
    } else {
        // 8 epilogue warps: lane quarter q = warp % 4, every other 16-column chunk
        const int q = warp & 3;
        const bool got = ptx::mbar_wait(ptx::smem_u32(&ctl->accf[0]), 0, abort_flag, p.status,
                                        MOARA_ERR_DEVICE_TIMEOUT, p.wait_limit);
        if (__all_sync(0xffffffffu, got)) {
            ptx::tc_fence_after();
            const int row = r0 + q * 32 + lane;
            uint16_t* const ol = p.out_lo[pi];
            float* const of = p.out[pi];
            uint16_t* const ob = p.out_bf[pi];
            const long long ro = (long long)row * N;
            for (int c = (warp - 2) >> 2; c < nb * 8; c += 2) {
                const int j0 = n0 + c * 16;
                if (j0 >= N) break;                       // warp-uniform
                float v[16];
                __syncwarp();
                ptx::tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) + c * 16, v);
                if (row < M) kr_store16(of, ob, ol, ro, j0, N, v);
            }
        }
    }

    ptx::tc_fence_before();
    __syncwarp();
    pair_abort(ctl, crank);
    __syncwarp();
    ptx::cluster_sync();            // no CTA leaves while its peer may still signal or fill it
    if (*abort_flag) {              // the same in both CTAs
        if (threadIdx.x == 0) pair_settle<STAGES>(ctl, crank, fill);
        __syncwarp();
        ptx::cluster_sync();
    }
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc2(tmem, 256);
    }
}

// ===========================================================================
// KS: fp32-accurate GEMM of the Rayleigh-Ritz step on tensor cores.  Both
// operands arrive as three bf16 planes (x = hi + mid + lo, 24 significant
// bits); six MMAs per k-step (hi.hi, hi.mid, mid.hi, hi.lo, mid.mid, lo.hi)
// leave out terms of relative size 2^-24 and below.  out (M x N, fp32) =
// A B with A stored K x M and B stored K x N (both MN-major), tile 256 x 256
// (two 128-row accumulators in TMEM) or 128 x 256, BK = 32, two stages of
// 96 KB; `ktri` stops the K loop of column tile n0 at n0 + 256 (B upper
// triangular).
// ===========================================================================
constexpr int KS_BM = 256, KS_BN = 256, KS_BK = 32;
constexpr int KS_PLANE = KS_BM * KS_BK * 2;               // 16 KB: one plane of A (or B)
constexpr int KS_RING = 12 * KS_PLANE;                    // 192 KB of stages
constexpr int KS_SMEM = 1024 + KS_RING + 2048;
// NP = 3 planes: six products per k-step, two stages of 96 KB.  NP = 2
// (hi + mid, 16 significant bits; for iterates that a later fp32-accurate
// pass corrects): three products (hi.hi, hi.mid, mid.hi), three stages of 64 KB.
template <int NP> struct KsCfg {
    static constexpr int STAGE = 2 * NP * KS_PLANE;
    static constexpr int STAGES = KS_RING / STAGE;
    static constexpr int PRODUCTS = NP == 3 ? 6 : 3;
};
constexpr int kKsGroup = 38;                              // problems per launch (six maps each in the parameters)

struct KsParams {
    CUtensorMap amap[kKsGroup][3];     // A planes ({M, K}, box {64, 32})
    CUtensorMap bmap[kKsGroup][3];     // B planes ({N, K}, box {64, 32})
    float* out[kKsGroup];
    int M[kKsGroup], N[kKsGroup], K[kKsGroup];
    int ktri[kKsGroup];
    int ldo[kKsGroup];                 // row pitch of out
    int sub[kKsGroup];                 // out -= A B
    int lower[kKsGroup];               // tiles above the diagonal are skipped
    int tiles_n[kKsGroup];
    int tile_start[kKsGroup + 1];
    int count;
    int bm;                            // tile rows: 256 or 128
    int* status;
    long long wait_limit;              // clock cycles of a bounded wait before it gives up
};

static_assert(sizeof(KsParams) <= 32764, "KS's parameter block fits the kernel parameter space");

template <int NP>
__global__ void __launch_bounds__(KR_THREADS, 1) ks_product(const __grid_constant__ KsParams p) {
    constexpr int KS_STAGE = KsCfg<NP>::STAGE, KS_STAGES = KsCfg<NP>::STAGES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    SmemCtl* ctl = reinterpret_cast<SmemCtl*>(smem + KS_RING);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &ctl->abort;

    const int tile = blockIdx.x;
    int lo = 0, hi = p.count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.tile_start[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    const int pi = lo;
    const int local = tile - p.tile_start[pi];
    const int M = p.M[pi], N = p.N[pi], K = p.K[pi];
    const int i0 = (local / p.tiles_n[pi]) * p.bm;
    const int n0 = (local % p.tiles_n[pi]) * KS_BN;
    if (p.lower[pi] && n0 >= i0 + p.bm) return;      // whole CTA, before any barrier or TMEM
    const int nch = min(4, (N - n0 + 63) / 64);
    const int halves = p.bm > 128 && (M - i0) > 128 ? 2 : 1;
    const int kend = p.ktri[pi] ? min(K, n0 + KS_BN) : K;
    const int nk = (kend + KS_BK - 1) / KS_BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < KS_STAGES; ++s) {
            ptx::mbar_init(ptx::smem_u32(&ctl->full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctl->empty[s]), 1);
        }
        ptx::mbar_init(ptx::smem_u32(&ctl->accf[0]), 1);
        ptx::mbar_init(ptx::smem_u32(&ctl->drain), 1);
        ctl->abort = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(&ctl->tmem_base), 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    pdl_begin();

    if (warp == 0) {
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t issued = 0, last_par = 0;
            const int ach = p.bm / 64;                     // 64-row chunks of A
            const uint32_t bytes = NP * (ach + nch) * 4096;
            for (int kb = 0; kb < nk; ++kb) {
                if (!ptx::mbar_wait(ptx::smem_u32(&ctl->empty[stage]), phase ^ 1, abort_flag, p.status,
                                    MOARA_ERR_DEVICE_TIMEOUT, p.wait_limit))
                    break;
                const uint32_t fb = ptx::smem_u32(&ctl->full[stage]);
                ptx::mbar_arrive_expect_tx(fb, bytes);
                const uint32_t a = ptx::smem_u32(smem + stage * KS_STAGE);
                const uint32_t b = a + NP * KS_PLANE;
#pragma unroll
                for (int q = 0; q < NP; ++q) {
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (c < ach)
                            ptx::tma_load_2d(a + q * KS_PLANE + c * 4096, &p.amap[pi][q], fb, i0 + 64 * c, kb * KS_BK);
                    for (int c = 0; c < nch; ++c)
                        ptx::tma_load_2d(b + q * KS_PLANE + c * 4096, &p.bmap[pi][q], fb, n0 + 64 * c, kb * KS_BK);
                }
                issued |= 1u << stage;
                last_par = (last_par & ~(1u << stage)) | (phase << stage);
                if (++stage == KS_STAGES) { stage = 0; phase ^= 1; }
            }
            // every copy issued has landed before the CTA may leave (after a
            // wait that gave up elsewhere the MMA may not have consumed them)
            for (int s = 0; s < KS_STAGES; ++s)
                if (issued & (1u << s)) wait_drain(ptx::smem_u32(&ctl->full[s]), (last_par >> s) & 1);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = ptx::idesc_bf16(128, nch * 64, 1, 1);
            // plane pairs (A, B) of the six products
            constexpr int PA[6] = {0, 0, 1, 0, 1, 2};
            constexpr int PB[6] = {0, 1, 0, 2, 1, 0};
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = 0; kb < nk; ++kb) {
                if (!ptx::mbar_wait(ptx::smem_u32(&ctl->full[stage]), phase, abort_flag, p.status,
                                    MOARA_ERR_DEVICE_TIMEOUT, p.wait_limit)) break;
                ptx::tc_fence_after();
                const uint32_t a = ptx::smem_u32(smem + stage * KS_STAGE);
                const uint32_t b = a + NP * KS_PLANE;
#pragma unroll
                for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
                    for (int e = 0; e < KsCfg<NP>::PRODUCTS; ++e) {
                        const uint64_t bdesc = ptx::smem_desc_sw128(b + PB[e] * KS_PLANE + kk * 2048, 4096, 1024);
                        for (int h = 0; h < halves; ++h) {
                            const uint64_t adesc =
                                ptx::smem_desc_sw128(a + PA[e] * KS_PLANE + h * 8192 + kk * 2048, 4096, 1024);
                            ptx::mma_f16(tmem + h * 256, adesc, bdesc, idesc, (kb | kk | e) != 0);
                        }
                    }
                }
                ptx::mma_commit(ptx::smem_u32(&ctl->empty[stage]));
                if (++stage == KS_STAGES) { stage = 0; phase ^= 1; }
            }
            ptx::mma_commit(ptx::smem_u32(&ctl->accf[0]));
            ptx::mma_commit(ptx::smem_u32(&ctl->drain));
            wait_drain(ptx::smem_u32(&ctl->drain), 0);
        }
    } else {
        const int ew = warp - 2;
        const int q = warp & 3;
        // row half of the tile, or with one half every other 16-column chunk
        const int h = halves == 2 ? ew >> 2 : 0, cfirst = halves == 2 ? 0 : ew >> 2, cstep = halves == 2 ? 1 : 2;
        const bool got = ptx::mbar_wait(ptx::smem_u32(&ctl->accf[0]), 0, abort_flag, p.status,
                                        MOARA_ERR_DEVICE_TIMEOUT, p.wait_limit);
        if (__all_sync(0xffffffffu, got)) {
            ptx::tc_fence_after();
            const int row = i0 + h * 128 + q * 32 + lane;
            float* const of = p.out[pi];
            const long long ro = (long long)row * p.ldo[pi];
            const bool sub = p.sub[pi] != 0;
            for (int c = cfirst; c < nch * 4; c += cstep) {
                const int j0 = n0 + c * 16;
                if (j0 >= N) break;                       // warp-uniform
                float v[16];
                __syncwarp();
                ptx::tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) + h * 256 + c * 16, v);
                if (row >= M) continue;
                if (j0 + 16 <= N) {
                    float4* o4 = reinterpret_cast<float4*>(of + ro + j0);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float4 w = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
                        if (sub) {
                            const float4 o = o4[e];
                            w = make_float4(o.x - w.x, o.y - w.y, o.z - w.z, o.w - w.w);
                        }
                        o4[e] = w;
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        if (j0 + e < N) of[ro + j0 + e] = sub ? of[ro + j0 + e] - v[e] : v[e];
                }
            }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, 512);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

bool encode_2d(EncodeTiledFn enc, CUtensorMap* map, CUtensorMapDataType dt, int esize, const void* ptr,
               uint64_t inner, uint64_t outer, uint32_t box_inner, uint32_t box_outer) {
    const cuuint64_t dims[2] = {inner, outer};
    const cuuint64_t strides[1] = {inner * esize};
    const cuuint32_t box[2] = {box_inner, box_outer};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, dt, 2, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_bf16_2d(EncodeTiledFn enc, CUtensorMap* map, const void* ptr, uint64_t inner, uint64_t outer,
                    uint32_t box_inner, uint32_t box_outer) {
    return encode_2d(enc, map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ptr, inner, outer, box_inner, box_outer);
}

// Largest number of 2-CTA clusters of `fn` resident at once (at most `cap`).
int max_clusters(const void* fn, int threads, int smem, int cap) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * cap, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess || n < 1) {
        cudaGetLastError();
        return cap;
    }
    return std::min(n, cap);
}

template <int BLK>
void set_smem_attrs() {
    cudaFuncSetAttribute(k2_backproject<BLK, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, K2_SMEM);
    cudaFuncSetAttribute(k2_backproject<BLK, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, K2_SMEM);
    if constexpr (BLK >= 32)
        cudaFuncSetAttribute(k2_backproject<BLK, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, K2_SMEM);
}

}  // namespace

struct TcState {
    int device = 0;
    int* d_status = nullptr;
    int sms = 148;
    EncodeTiledFn encode = nullptr;
    std::string err;
    std::vector<TcMod> mods;               // indexed by module id (unsupported ones left zero)
    std::vector<CUtensorMap> maps;         // kMaps per module id
    TcMod* d_mods = nullptr;
    CUtensorMap* d_maps = nullptr;
    int cap = 0;
    bool dirty = false;
    // Per-CTA work lists of one launch (CSR: start offsets, then tiles).
    struct Tiles {
        void* mem = nullptr;
        const int* k1_start = nullptr; const TcTile* k1 = nullptr; int g1 = 0; int bn1 = K1_BN;
        const int* k2_start = nullptr; const TcTile* k2 = nullptr; int g2 = 0;
    };
    std::map<std::vector<int>, Tiles> tiles;
    int align_lists = 0;                   // of them, made by alignment calls
    bool attrs_set = false;
    int k1_clusters = 1, k2_clusters = 1;  // co-resident 2-CTA clusters of K1 / K2
    K1Params p1;                           // parameter block of the next K1 launch
    K0Params p0;                           // parameter block of the next K0 launch
    KrParams pr;                           // parameter block of the next refresh GEMM launch
    bool kr_attrs = false;
    KsParams ps;                           // parameter block of the next split-precision GEMM launch
    bool ks_attrs = false;
    // decomposition of later module parts, overlapped with K1 / K2 of earlier ones
    cudaStream_t aux = nullptr;
    cudaEvent_t ev_start = nullptr;
    cudaEvent_t ev_part[32] = {};          // decomposition of part q done (auxiliary stream)
    cudaEvent_t ev_k1[32] = {};            // K1 of part q about to start (launching stream)
    long long wait_limit = kWaitLimit;     // bounded waits of the refresh / alignment products (KR, KS)
};

bool tc_supported(int m, int n, int r, int B, int dtype, int decompose, int state_dtype) {
    if (state_dtype == MOARA_DTYPE_BF16 && decompose && B < 32) return false;
    if (dtype != MOARA_DTYPE_BF16) return false;
    if (m < 1 || n < 8 || r < 8) return false;
    if ((n % 8) != 0 || (r % 8) != 0) return false;
    if (decompose && !(B == 8 || B == 16 || B == 32 || B == 64 || B == 128)) return false;
    if (!decompose && !(B >= 1)) return false;
    return true;
}

TcState* tc_create(int device, int* d_status) {
    TcState* st = new TcState();
    st->device = device;
    st->d_status = d_status;
    cudaDeviceProp prop{};
    if (cudaGetDeviceProperties(&prop, device) == cudaSuccess) {
        st->sms = prop.multiProcessorCount;
        if (prop.major != 10 || prop.minor != 3) {   // these kernels are built for sm_103a only
            delete st;
            return nullptr;
        }
    }
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess || q != cudaDriverEntryPointSuccess || fn == nullptr) {
        delete st;
        return nullptr;
    }
    st->encode = reinterpret_cast<EncodeTiledFn>(fn);
    return st;
}

void tc_destroy(TcState* st) {
    if (st == nullptr) return;
    if (st->d_mods) cudaFree(st->d_mods);
    if (st->d_maps) cudaFree(st->d_maps);
    for (auto& kv : st->tiles)
        if (kv.second.mem) cudaFree(kv.second.mem);
    if (st->aux) cudaStreamDestroy(st->aux);
    if (st->ev_start) cudaEventDestroy(st->ev_start);
    for (cudaEvent_t e : st->ev_part)
        if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : st->ev_k1)
        if (e) cudaEventDestroy(e);
    delete st;
}

int tc_register(TcState* st, int id, const ModDev& md, const moara_hparams& hp) {
    if (st == nullptr) return MOARA_OK;
    if (static_cast<int>(st->mods.size()) <= id) {
        st->mods.resize(id + 1, TcMod{});
        st->maps.resize(kMaps * (id + 1));
    }
    if (!tc_supported(md.m, md.n, md.r, hp.block_size, md.dtype, hp.decompose, hp.state_dtype) || md.Pb == nullptr)
        return MOARA_OK;
    // W and the direction moments: fp32, or bf16 (state_dtype); a ring chunk
    // is one 128-byte row wide either way
    const bool sb = hp.state_dtype == MOARA_DTYPE_BF16;
    const CUtensorMapDataType sdt = sb ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    const int ses = sb ? 2 : 4, scols = sb ? StateCols<true>::N : StateCols<false>::N;
    TcMod t{};
    t.m = md.m; t.n = md.n; t.r = md.r; t.kb = md.kb;
    t.Vhi = md.ws_Vhi; t.Vlo = md.ws_Vlo;
    t.W = md.W; t.exp_avg = md.exp_avg; t.exp_avg_sq = md.exp_avg_sq;
    t.mag = md.ws_inv;     // the block-scale buffer of the fp32 path holds the norms here
    t.mag_avg = md.mag_avg; t.mag_avg_sq = md.mag_avg_sq;
    t.Nb = reinterpret_cast<uint16_t*>(md.ws_N);
    t.dM = md.ws_dM;
    t.Pb = md.Pb;
    t.right = md.right;
    t.Qt = md.ws_Qt;
    CUtensorMap* mp = &st->maps[kMaps * id];
    bool ok;
    if (!md.right) {
        // K1: A = P^T (MN-major chunks of P), B = V (MN-major), moments r x n;
        // K2: A = P rows (K-major), B = N (MN-major)
        ok = encode_bf16_2d(st->encode, &mp[0], md.Pb, md.r, md.m, 64, 64) &&
             encode_bf16_2d(st->encode, &mp[1], md.Pb, md.r, md.m, 64, 128) &&
             encode_bf16_2d(st->encode, &mp[2], t.Nb, md.n, md.r, 64, 64) &&
             encode_bf16_2d(st->encode, &mp[4], t.Vhi, md.n, md.m, 64, 64) &&
             encode_bf16_2d(st->encode, &mp[5], t.Vlo, md.n, md.m, 64, 64) &&
             encode_2d(st->encode, &mp[6], sdt, ses, md.exp_avg, md.n, md.r, scols, K1_BM) &&
             encode_2d(st->encode, &mp[7], sdt, ses, md.exp_avg_sq, md.n, md.r, scols, K1_BM);
    } else {
        // right projector Q (n x r): K1 computes R = V Q with A = V rows
        // (K-major, 128 rows x 64 columns) and B = Q (MN-major chunks), moments
        // m x r; K2 computes dV = N Q^T with A = N rows (K-major) and
        // B = Q^T (r x n, MN-major)
        ok = md.ws_Qt != nullptr &&
             encode_bf16_2d(st->encode, &mp[0], md.Pb, md.r, md.n, 64, 64) &&
             encode_bf16_2d(st->encode, &mp[1], t.Nb, md.r, md.m, 64, 128) &&
             encode_bf16_2d(st->encode, &mp[2], md.ws_Qt, md.n, md.r, 64, 64) &&
             encode_bf16_2d(st->encode, &mp[4], t.Vhi, md.n, md.m, 64, 128) &&
             encode_bf16_2d(st->encode, &mp[5], t.Vlo, md.n, md.m, 64, 128) &&
             encode_2d(st->encode, &mp[6], sdt, ses, md.exp_avg, md.r, md.m, scols, K1_BM) &&
             encode_2d(st->encode, &mp[7], sdt, ses, md.exp_avg_sq, md.r, md.m, scols, K1_BM);
    }
    // residual plane of N for the alignment diagnostic, after its hi plane
    ok = ok && (md.right ? encode_bf16_2d(st->encode, &mp[9], t.Nb + (size_t)md.m * md.r, md.r, md.m, 64, 128)
                         : encode_bf16_2d(st->encode, &mp[9], t.Nb + (size_t)md.r * md.n, md.n, md.r, 64, 64));
    ok = ok && encode_2d(st->encode, &mp[3], sdt, ses, md.W, md.n, md.m, scols, K2_BM);
    if (!ok) {
        st->err = "cuTensorMapEncodeTiled failed";
        return MOARA_ERR_CUDA;
    }
    // An fp32 W whose rows split into 64-column pairs of 128-byte groups is
    // also viewed as (32 columns, n / 32 groups, m rows): a box of 32 x 2 x 64
    // adds 64 rows x 256 contiguous bytes per row with one reduce, traversed
    // row by row, while each 128-byte group stays one swizzled line of the
    // staging chunk (line = row * 2 + group).  The wider contiguous pieces per
    // row keep HBM pages open longer than the 128-byte pieces of the 2-D map
    // (K2 per two 7B layers 0.74 -> 0.70 ms; the group-outer box order, whose
    // lines are free of bank conflicts, gave 0.72 ms).
    t.w3d = 0;
    if (!sb && md.n % 64 == 0) {
        const cuuint64_t dims[3] = {32, static_cast<cuuint64_t>(md.n / 32), static_cast<cuuint64_t>(md.m)};
        const cuuint64_t strides[2] = {128, static_cast<cuuint64_t>(md.n) * 4};
        const cuuint32_t box[3] = {32, 2, 64};
        const cuuint32_t estr[3] = {1, 1, 1};
        t.w3d = st->encode(&mp[8], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, md.W, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    st->mods[id] = t;
    st->dirty = true;
    return MOARA_OK;
}

static int tc_upload(TcState* st) {
    if (!st->dirty) return MOARA_OK;
    const int n = static_cast<int>(st->mods.size());
    if (n > st->cap) {
        int ncap = std::max(64, st->cap);
        while (ncap < n) ncap *= 2;
        if (st->d_mods) cudaFree(st->d_mods);
        if (st->d_maps) cudaFree(st->d_maps);
        st->d_mods = nullptr;
        st->d_maps = nullptr;
        if (cudaMalloc(&st->d_mods, sizeof(TcMod) * ncap) != cudaSuccess ||
            cudaMalloc(&st->d_maps, sizeof(CUtensorMap) * kMaps * ncap) != cudaSuccess) {
            st->err = "cudaMalloc of the tensor-core module table failed";
            return MOARA_ERR_CUDA;
        }
        st->cap = ncap;
    }
    if (cudaMemcpy(st->d_mods, st->mods.data(), sizeof(TcMod) * n, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(st->d_maps, st->maps.data(), sizeof(CUtensorMap) * kMaps * n, cudaMemcpyHostToDevice) !=
            cudaSuccess) {
        st->err = "upload of the tensor-core module table failed";
        return MOARA_ERR_CUDA;
    }
    st->dirty = false;
    return MOARA_OK;
}

// Longest-processing-time assignment of weighted tiles to `grid` persistent
// CTAs: tiles in descending cost, each to the CTA with the least work so far;
// each CTA runs its tiles in that (descending) order.
static void lpt_assign(const std::vector<TcTile>& tiles, const std::vector<double>& cost, int grid,
                       std::vector<int>& start, std::vector<TcTile>& out) {
    std::vector<int> order(tiles.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = static_cast<int>(i);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return cost[a] > cost[b]; });
    std::vector<std::vector<int>> per(grid);
    std::vector<std::pair<double, int>> heap;
    for (int c = 0; c < grid; ++c) heap.push_back({0.0, c});
    auto cmp = [](const std::pair<double, int>& a, const std::pair<double, int>& b) {
        return a.first > b.first || (a.first == b.first && a.second > b.second);
    };
    std::make_heap(heap.begin(), heap.end(), cmp);
    for (int i : order) {
        std::pop_heap(heap.begin(), heap.end(), cmp);
        auto& top = heap.back();
        per[top.second].push_back(i);
        top.first += cost[i];
        std::push_heap(heap.begin(), heap.end(), cmp);
    }
    start.assign(grid + 1, 0);
    out.clear();
    for (int c = 0; c < grid; ++c) {
        start[c] = static_cast<int>(out.size());
        for (int i : per[c]) out.push_back(tiles[i]);
    }
    start[grid] = static_cast<int>(out.size());
}

// Shared-memory limits of the step kernels and their resident grids.
static void tc_init(TcState* st) {
    if (!st->attrs_set) {
        constexpr int W = K1_BN, N = K1_BN_NARROW;
        for (auto fn : {k1_project<true, false, false, W>, k1_project<false, false, false, W>,
                        k1_project<true, true, false, W>, k1_project<false, true, false, W>,
                        k1_project<true, false, true, W>, k1_project<false, false, true, W>,
                        k1_project<true, true, true, W>, k1_project<false, true, true, W>,
                        k1_project<true, false, false, N>, k1_project<false, false, false, N>,
                        k1_project<true, true, false, N>, k1_project<false, true, false, N>,
                        k1_project<true, false, true, N>, k1_project<false, false, true, N>,
                        k1_project<true, true, true, N>, k1_project<false, true, true, N>})
            cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, K1_SMEM);
        set_smem_attrs<8>(); set_smem_attrs<16>(); set_smem_attrs<32>(); set_smem_attrs<64>();
        set_smem_attrs<128>();
        // clusters of two that fit on the GPU at once (persistent grids)
        st->k1_clusters = max_clusters(reinterpret_cast<const void*>(k1_project<false, false, false, K1_BN>), K1_THREADS,
                                       K1_SMEM,
                                       st->sms / 2);
        st->k2_clusters = max_clusters(reinterpret_cast<const void*>(k2_backproject<128, false>), K2_THREADS, K2_SMEM,
                                       st->sms / 2);
        st->attrs_set = true;
    }
}

// Work lists of one launch: K1 tiles (128-rank x 256-column) and K2 tiles
// (128-row x 256-column), cost-weighted in SM clocks: MMA time (8 clocks per
// K row of a 128 x 256 tile) against the epilogue's HBM traffic (K1: the two
// moments read and written and N stored, 18 bytes per entry; K2: W read and
// written, 8 bytes per entry; about 27 bytes per clock per SM).
static TcState::Tiles* tc_tiles(TcState* st, const std::vector<int>& ids) {
    auto it = st->tiles.find(ids);
    if (it != st->tiles.end()) return &it->second;
    // Work units are pair tiles: the two CTAs of a cluster take rank (K1) or
    // row (K2) tiles 2 t0 and 2 t0 + 1 of the same column tile t1.
    std::vector<TcTile> k1, k2;
    std::vector<double> c1, c2;
    // columns of a K1 tile (see K1_BN_NARROW)
    int wide = 0;
    for (int id : ids) {
        const TcMod& md = st->mods[id];
        const int rows = md.right ? md.m : md.r, cols = md.right ? md.r : md.n;
        wide += (rows + 2 * K1_BM - 1) / (2 * K1_BM) * ((cols + K1_BN - 1) / K1_BN);
    }
    const int bn = 2 * wide <= st->k1_clusters ? K1_BN_NARROW : K1_BN;
    for (size_t slot = 0; slot < ids.size(); ++slot) {
        const TcMod& md = st->mods[ids[slot]];
        // column tiles outer, rank pairs inner: clusters that start together
        // share the V panel of one column tile in L2
        // R: r x n (K = m), or m x r (K = n) with a right projector
        const int Rr = md.right ? md.m : md.r, Rc = md.right ? md.r : md.n, Rk = md.right ? md.n : md.m;
        const int nt = (Rc + bn - 1) / bn, rt = (Rr + K1_BM - 1) / K1_BM;
        for (int j = 0; j < nt; ++j)
            for (int i = 0; i < (rt + 1) / 2; ++i) {
                const int rows = std::min(K1_BM, Rr - 2 * i * K1_BM);
                const double mma = 8.0 * Rk * bn / K1_BN;
                const double epi = 0.66 * rows * std::min(bn, Rc - j * bn);
                k1.push_back({ids[slot], static_cast<int>(slot), i, j});
                c1.push_back(std::max(mma, epi));
            }
        const int mt = (md.m + K2_BM - 1) / K2_BM, nt2 = (md.n + K2_BN - 1) / K2_BN;
        for (int i = 0; i < (mt + 1) / 2; ++i)
            for (int j = 0; j < nt2; ++j) {
                const double mma = 8.0 * md.r;
                const double epi = 0.3 * std::min(K2_BM, md.m - 2 * i * K2_BM) * std::min(K2_BN, md.n - j * K2_BN);
                k2.push_back({ids[slot], static_cast<int>(slot), i, j});
                c2.push_back(std::max(mma, epi));
            }
    }
    TcState::Tiles t;
    t.bn1 = bn;
    t.g1 = std::max(1, std::min(static_cast<int>(k1.size()), st->k1_clusters));   // clusters
    t.g2 = std::max(1, std::min(static_cast<int>(k2.size()), st->k2_clusters));
    std::vector<int> s1, s2;
    std::vector<TcTile> o1, o2;
    lpt_assign(k1, c1, t.g1, s1, o1);
    lpt_assign(k2, c2, t.g2, s2, o2);
    auto pad = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t b_s1 = pad(sizeof(int) * s1.size()), b_o1 = pad(sizeof(TcTile) * std::max<size_t>(1, o1.size()));
    const size_t b_s2 = pad(sizeof(int) * s2.size()), b_o2 = pad(sizeof(TcTile) * std::max<size_t>(1, o2.size()));
    std::vector<char> host(b_s1 + b_o1 + b_s2 + b_o2, 0);
    std::memcpy(host.data(), s1.data(), sizeof(int) * s1.size());
    std::memcpy(host.data() + b_s1, o1.data(), sizeof(TcTile) * o1.size());
    std::memcpy(host.data() + b_s1 + b_o1, s2.data(), sizeof(int) * s2.size());
    std::memcpy(host.data() + b_s1 + b_o1 + b_s2, o2.data(), sizeof(TcTile) * o2.size());
    if (cudaMalloc(&t.mem, host.size()) != cudaSuccess) return nullptr;
    if (cudaMemcpy(t.mem, host.data(), host.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaFree(t.mem);
        return nullptr;
    }
    char* base = static_cast<char*>(t.mem);
    t.k1_start = reinterpret_cast<const int*>(base);
    t.k1 = reinterpret_cast<const TcTile*>(base + b_s1);
    t.k2_start = reinterpret_cast<const int*>(base + b_s1 + b_o1);
    t.k2 = reinterpret_cast<const TcTile*>(base + b_s1 + b_o1 + b_s2);
    return &(st->tiles[ids] = t);
}

// The decomposition without Optimizer_M for block size B.
static auto k0_plain(int B) {
    return B == 8    ? k0_decompose<8, false>
           : B == 16 ? k0_decompose<16, false>
           : B == 32 ? k0_decompose<32, false>
           : B == 64 ? k0_decompose<64, false>
                     : k0_decompose<128, false>;
}

// K0 and Optimizer_M of one module part.  `background`: a grid of short
// CTAs (about four row segments per warp) that fills the room K1 / K2 leave
// on each SM instead of a persistent grid that would hold SMs they need.
template <int BLK>
static cudaError_t launch_k0(TcState* st, const K0Params& p0, bool background, cudaStream_t s,
                             int64_t* launches, const TcProfile& prof, bool early, bool mag_adam) {
    const int phase = background ? MOARA_PHASE_TC_DECOMPOSE_OVERLAP : MOARA_PHASE_TC_DECOMPOSE;
    if (prof.on) prof.mark(prof.ctx, phase, s, true);
    const long long items = p0.start[p0.count];
    const int g0 = background ? static_cast<int>(std::max<long long>(1, std::min<long long>((items + 31) / 32, 1 << 30)))
                              : st->sms * 3;
    bool pass = mag_adam;                              // Optimizer_M as a pass of its own
    cudaError_t e = cudaSuccess;
    if constexpr (BLK >= 32) {
        if (mag_adam) e = launch_if(early && !background, k0_decompose<BLK, true>, g0, 256, 0, s, 1, p0);
        pass = false;
    }
    if (BLK < 32 || !mag_adam) e = launch_if(early && !background, k0_decompose<BLK, false>, g0, 256, 0, s, 1, p0);
    if (pass && e == cudaSuccess) e = launch_if(early && !background, k0_mag_adam, background ? st->sms : st->sms * 4, 256, 0, s, 1, p0);
    if (prof.on) prof.mark(prof.ctx, phase, s, false);
    *launches += pass ? 2 : 1;
    return e;
}

// which: 1 = K1, 2 = K2, 4 = early launches (of K1 only directly behind its decomposition on the stream)
template <int BLK, bool SB>
static cudaError_t launch_k12(TcState* st, const K1Params& p1, const K2Params& p2, int g1, int bn, int g2, bool hilo,
                              cudaStream_t s, int64_t* launches, const TcProfile& prof, int which, bool rt) {
    cudaError_t e;
    if (which & 1) {
        if (prof.on) prof.mark(prof.ctx, MOARA_PHASE_TC_PROJECT, s, true);
        constexpr int W = K1_BN, N = K1_BN_NARROW;
        auto fn = bn == W ? (rt ? (hilo ? k1_project<true, SB, true, W> : k1_project<false, SB, true, W>)
                                : (hilo ? k1_project<true, SB, false, W> : k1_project<false, SB, false, W>))
                          : (rt ? (hilo ? k1_project<true, SB, true, N> : k1_project<false, SB, true, N>)
                                : (hilo ? k1_project<true, SB, false, N> : k1_project<false, SB, false, N>));
        // of several parts, K1 waits for its part's decomposition on the other stream
        e = launch_if((which & 4) != 0 && !prof.on, fn, 2 * g1, K1_THREADS, K1_SMEM, s, 1, p1);
        if (prof.on) prof.mark(prof.ctx, MOARA_PHASE_TC_PROJECT, s, false);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    if (!(which & 2)) return cudaSuccess;
    if (prof.on) prof.mark(prof.ctx, MOARA_PHASE_TC_BACKPROJECT, s, true);
    e = launch_if((which & 4) != 0 && !prof.on, k2_backproject<BLK, SB>, 2 * g2, K2_THREADS, K2_SMEM, s, 1, p2);
    if (prof.on) prof.mark(prof.ctx, MOARA_PHASE_TC_BACKPROJECT, s, false);
    if (e != cudaSuccess) return e;
    ++*launches;
    return cudaSuccess;
}

static cudaError_t launch_k0_any(int B, TcState* st, const K0Params& p0, bool background, cudaStream_t s,
                                 int64_t* launches, const TcProfile& prof, bool early, bool mag_adam) {
    switch (B) {
        case 8: return launch_k0<8>(st, p0, background, s, launches, prof, early, mag_adam);
        case 16: return launch_k0<16>(st, p0, background, s, launches, prof, early, mag_adam);
        case 32: return launch_k0<32>(st, p0, background, s, launches, prof, early, mag_adam);
        case 64: return launch_k0<64>(st, p0, background, s, launches, prof, early, mag_adam);
        default: return launch_k0<128>(st, p0, background, s, launches, prof, early, mag_adam);
    }
}

static cudaError_t launch_k12_any(int B, bool sb, TcState* st, const K1Params& p1, const K2Params& p2, int g1,
                                  int bn, int g2, bool hilo, cudaStream_t s, int64_t* launches, const TcProfile& prof,
                                  int which, bool rt = false) {
    if (sb) {   // bf16 states: B >= 32 (tc_supported)
        switch (B) {
            case 32: return launch_k12<32, true>(st, p1, p2, g1, bn, g2, hilo, s, launches, prof, which, rt);
            case 64: return launch_k12<64, true>(st, p1, p2, g1, bn, g2, hilo, s, launches, prof, which, rt);
            default: return launch_k12<128, true>(st, p1, p2, g1, bn, g2, hilo, s, launches, prof, which, rt);
        }
    }
    switch (B) {
        case 8: return launch_k12<8, false>(st, p1, p2, g1, bn, g2, hilo, s, launches, prof, which, rt);
        case 16: return launch_k12<16, false>(st, p1, p2, g1, bn, g2, hilo, s, launches, prof, which, rt);
        case 32: return launch_k12<32, false>(st, p1, p2, g1, bn, g2, hilo, s, launches, prof, which, rt);
        case 64: return launch_k12<64, false>(st, p1, p2, g1, bn, g2, hilo, s, launches, prof, which, rt);
        default: return launch_k12<128, false>(st, p1, p2, g1, bn, g2, hilo, s, launches, prof, which, rt);
    }
}

// A launch group is split into parts (consecutive modules, about equal
// gradient bytes): the decomposition of part q + 1 runs on an auxiliary stream
// while K1 / K2 of part q run.  A part carries at least kPartBytes of
// gradients, two 4096 / 11008 layers: every part boundary ends two persistent
// grids and starts two, which costs more than the hidden decomposition gives
// where a part holds less.  Measured, us per step with 1 / 2 / 4 / 8 / 16 parts:
//   24 layers of 1024 / 2816 (0.6 GB)     1008   1023   1074   1132   1385
//    4 layers of 4096 / 11008 (1.6 GB)    3501   3465   3487   3599   3795
//    5 layers (2.0 GB)                    4405   4320   4336   4433   4627
//    8 layers (3.2 GB)                    7080   6863   6968   6902   7185
//   12 layers (4.9 GB)                   10755  10411  10428  10350  10536
constexpr int kOverlapParts = 16;
constexpr double kPartBytes = 0.8e9;
// Groups of up to so many gradient bytes, and every group without a
// decomposition, launch each kernel beside the end of the one in front.
// Larger decomposed groups lose by it when steps follow one another (us per
// step with / without: one layer of 1024 / 2816, 25 MB, 66.0 / 71.6; two 108.9 /
// 112.8; four 194.3 / 193.8; eight 361.8 / 352.1; thirty ragged weights of 0.63
// GB 1053 / 1011; a 4096 / 11008 layer 872 / 862; a layer without decomposition
// 730 / 742).
constexpr double kEarlyBytes = 6.4e7;
static_assert(kOverlapParts <= 32, "one event per part");

int tc_group_limit() { return kTcGroup; }

int tc_step(TcState* st, const moara_hparams& hp, int n_mod, const int* ids, const void* const* G, float bc1,
            float bc2, float lr, int first_step, const float* clip, const TcClipFuse* fuse, cudaStream_t s,
            int64_t* launches, const TcProfile& prof) {
    tc_init(st);
    int rc = tc_upload(st);
    if (rc != MOARA_OK) return rc;
    const bool dec = hp.decompose != 0;
    const bool hilo = dec && first_step;
    const int B = dec ? hp.block_size : 128;
    auto fail = [&](const char* what) {
        st->err = what;
        return MOARA_ERR_CUDA;
    };
    // clipping from the block norms: Optimizer_M and K2 wait for the norm of
    // every module, so they run once after all decompositions and K1s
    const bool fused = fuse != nullptr && dec;
    if (fused && n_mod > kTcGroup) {
        st->err = "fused clipping takes at most tc_group_limit() modules";
        return MOARA_ERR_UNSUPPORTED;
    }
    for (int c0 = 0; c0 < n_mod; c0 += kTcGroup) {
        const int cnt = std::min(kTcGroup, n_mod - c0);
        // parts of the group (consecutive modules, about equal G bytes)
        double tot = 0.0;
        for (int q = 0; q < cnt; ++q) tot += (double)st->mods[ids[c0 + q]].m * st->mods[ids[c0 + q]].n;
        const int nparts = dec ? std::max(1, static_cast<int>(std::min<double>(kOverlapParts, 2.0 * tot / kPartBytes))) : 1;
        const bool early = !dec || 2.0 * tot <= kEarlyBytes;
        std::vector<int> pstart{0};
        if (nparts > 1) {
            double acc = 0.0;
            for (int q = 0; q < cnt; ++q) {
                acc += (double)st->mods[ids[c0 + q]].m * st->mods[ids[c0 + q]].n;
                if ((int)pstart.size() < nparts && acc >= tot * pstart.size() / nparts && q + 1 < cnt)
                    pstart.push_back(q + 1);
            }
        }
        pstart.push_back(cnt);
        const int np = static_cast<int>(pstart.size()) - 1;
        if (np > 1) {
            if (st->aux == nullptr) {
                cudaError_t e = cudaStreamCreateWithFlags(&st->aux, cudaStreamNonBlocking);
                if (e == cudaSuccess) e = cudaEventCreateWithFlags(&st->ev_start, cudaEventDisableTiming);
                for (int q = 0; q < 32 && e == cudaSuccess; ++q) {
                    e = cudaEventCreateWithFlags(&st->ev_part[q], cudaEventDisableTiming);
                    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&st->ev_k1[q], cudaEventDisableTiming);
                }
                if (e != cudaSuccess) return fail("auxiliary stream / events");
            }
            // the auxiliary stream starts after everything queued on s so far
            if (cudaEventRecord(st->ev_start, s) != cudaSuccess ||
                cudaStreamWaitEvent(st->aux, st->ev_start, 0) != cudaSuccess)
                return fail("auxiliary stream ordering");
        }
        auto build_p0 = [&](int a, int b) {
            K0Params& p0 = st->p0;
            std::memset(&p0, 0, sizeof(p0));
            p0.count = b - a;
            p0.hilo = hilo ? 1 : 0;
            p0.do_mag = 1;
            p0.decomp_eps = hp.decomp_eps;
            p0.beta1 = hp.beta1; p0.beta2 = hp.beta2; p0.adam_eps = hp.adam_eps;
            p0.bc1 = bc1; p0.bc2 = bc2;
            p0.clip = clip;
            long long acc = 0, macc = 0;
            for (int q = 0; q < b - a; ++q) {
                const TcMod& md = st->mods[ids[c0 + a + q]];
                const int segs = (md.n + K0_SEG - 1) / K0_SEG;
                p0.start[q] = acc;
                p0.mstart[q] = macc;
                p0.p[q] = K0Item{static_cast<const uint16_t*>(G[c0 + a + q]), md.Vhi, md.Vlo, md.mag, md.mag_avg,
                                 md.mag_avg_sq, md.dM, md.m, md.n, md.kb, segs};
                acc += static_cast<long long>(md.m) * segs;
                macc += static_cast<long long>(md.m) * md.kb;
            }
            p0.start[b - a] = acc;
            p0.mstart[b - a] = macc;
            return &p0;
        };
        // decomposition: part 0 on s with the full grid; part q + 1 in the
        // background on the auxiliary stream, launched after K1 / K2 of part q
        // so that their persistent CTAs are placed first
        if (dec && launch_k0_any(B, st, *build_p0(pstart[0], pstart[1]), false, s, launches, prof, early, !fused) !=
                       cudaSuccess)
            return fail("decomposition launch failed");
        for (int q = 0; q < np; ++q) {
            const int a = pstart[q], b = pstart[q + 1];
            std::vector<int> chunk(ids + c0 + a, ids + c0 + b);
            TcState::Tiles* tl = tc_tiles(st, chunk);
            if (tl == nullptr) { st->err = "tile list allocation failed"; return MOARA_ERR_CUDA; }
            if (q > 0 && cudaStreamWaitEvent(s, st->ev_part[q], 0) != cudaSuccess) return fail("part wait");
            K1Params& p1 = st->p1;
            std::memset(&p1, 0, sizeof(p1));
            if (!dec) {
                for (int k = 0; k < b - a; ++k) {
                    const TcMod& md = st->mods[chunk[k]];
                    // G as K1's B operand (64 x 64 chunks), or as its A operand
                    // (128 rows x 64 columns) for a right projector
                    if (!encode_bf16_2d(st->encode, &p1.gmap[k], G[c0 + a + k], md.n, md.m, 64, md.right ? 128 : 64)) {
                        st->err = "cuTensorMapEncodeTiled failed for a gradient";
                        return MOARA_ERR_CUDA;
                    }
                }
            }
            p1.cta_start = tl->k1_start; p1.tiles = tl->k1;
            p1.mods = st->d_mods; p1.maps = st->d_maps; p1.status = st->d_status;
            p1.beta1 = hp.beta1; p1.beta2 = hp.beta2; p1.adam_eps = hp.adam_eps;
            p1.bc1 = bc1; p1.bc2 = bc2;
            p1.inv_bc1 = 1.0f / bc1; p1.inv_bc2 = 1.0f / bc2;
            p1.decompose = dec ? 1 : 0;
            p1.clip = dec ? nullptr : clip;
            K2Params p2{};
            p2.cta_start = tl->k2_start; p2.tiles = tl->k2;
            p2.mods = st->d_mods; p2.maps = st->d_maps; p2.status = st->d_status;
            p2.step_scale = lr * hp.scale;
            p2.decompose = hp.decompose;
            bool rt = false;
            for (int k = 0; k < b - a; ++k) rt = rt || st->mods[chunk[k]].right != 0;
            const bool sb = hp.state_dtype == MOARA_DTYPE_BF16;
            // The decomposition of part q + 1 starts when K1 of part q does:
            // K1 runs tensor-bound with HBM to spare, while K2, whose W
            // stream keeps HBM busy, loses most when it shares the memory
            // system.  (Also holding K2 back until the decomposition ends
            // left a gap after each K1 and was slower.)
            const bool bg = dec && q + 1 < np;
            if (bg && cudaEventRecord(st->ev_k1[q], s) != cudaSuccess) return fail("part event");
            cudaError_t e = launch_k12_any(B, sb, st, p1, p2, tl->g1, tl->bn1, tl->g2, hilo, s, launches, prof,
                                           np == 1 && early ? 5 : 1, rt);
            if (e != cudaSuccess) {
                st->err = cudaGetErrorString(e);
                return MOARA_ERR_CUDA;
            }
            if (bg) {
                if (cudaStreamWaitEvent(st->aux, st->ev_k1[q], 0) != cudaSuccess ||
                    launch_k0_any(B, st, *build_p0(pstart[q + 1], pstart[q + 2]), true, st->aux, launches, prof,
                                  false, !fused) != cudaSuccess ||
                    cudaEventRecord(st->ev_part[q + 1], st->aux) != cudaSuccess)
                    return fail("background decomposition launch failed");
            }
            if (!fused) {
                e = launch_k12_any(B, sb, st, p1, p2, tl->g1, tl->bn1, tl->g2, hilo, s, launches, prof, early ? 6 : 2, rt);
                if (e != cudaSuccess) {
                    st->err = cudaGetErrorString(e);
                    return MOARA_ERR_CUDA;
                }
            }
        }
        if (fused) {
            // total norm from every module's block norms, the coefficient,
            // Optimizer_M of the clipped magnitudes, then K2 over the group
            K0Params* pall = build_p0(0, cnt);
            pall->clip = fuse->state + 1;
            if (prof.on) prof.mark(prof.ctx, MOARA_PHASE_CLIP_NORM, s, true);
            k0_mag_sq<<<kNormParts, 256, 0, s>>>(*pall, fuse->partials);
            ++*launches;
            if (launch_clip_finish(fuse->partials, kNormParts, fuse->extra, fuse->max_norm, fuse->state, s,
                                   launches) != cudaSuccess)
                return fail("clipping coefficient launch failed");
            if (prof.on) prof.mark(prof.ctx, MOARA_PHASE_CLIP_NORM, s, false);
            if (prof.on) prof.mark(prof.ctx, MOARA_PHASE_TC_DECOMPOSE, s, true);
            if (launch_if(false, k0_mag_adam, st->sms * 4, 256, 0, s, 1, *pall) != cudaSuccess)
                return fail("clipped magnitude launch failed");
            ++*launches;
            if (prof.on) prof.mark(prof.ctx, MOARA_PHASE_TC_DECOMPOSE, s, false);
            std::vector<int> all(ids + c0, ids + c0 + cnt);
            TcState::Tiles* tl = tc_tiles(st, all);
            if (tl == nullptr) { st->err = "tile list allocation failed"; return MOARA_ERR_CUDA; }
            K2Params p2{};
            p2.cta_start = tl->k2_start; p2.tiles = tl->k2;
            p2.mods = st->d_mods; p2.maps = st->d_maps; p2.status = st->d_status;
            p2.step_scale = lr * hp.scale;
            p2.decompose = hp.decompose;
            const cudaError_t e = launch_k12_any(B, hp.state_dtype == MOARA_DTYPE_BF16, st, st->p1, p2, tl->g1, tl->bn1, tl->g2,
                                                 hilo, s, launches, prof, 2);
            if (e != cudaSuccess) {
                st->err = cudaGetErrorString(e);
                return MOARA_ERR_CUDA;
            }
        }
    }
    return MOARA_OK;
}

const char* tc_last_error(const TcState* st) { return st ? st->err.c_str() : "no tensor-core state"; }

void tc_set_wait_limit(TcState* st, long long cycles) {
    if (st != nullptr) st->wait_limit = cycles > 0 ? cycles : kWaitLimit;
}

int tc_gemm_bf16(TcState* st, int a_kmajor, const TcGemmItem* items, int count, cudaStream_t s,
                 int64_t* launches) {
    if (!st->kr_attrs) {
        for (auto fn : {kr_product<true, 0>, kr_product<true, 1>, kr_product<false, 0>, kr_product<false, 1>,
                        kr_product<false, 2>})
            cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, KR_SMEM);
        for (auto fn : {kr_pair<true, 0>, kr_pair<true, 1>, kr_pair<false, 0>, kr_pair<false, 1>, kr_pair<false, 2>})
            cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, KR_SMEM);
        st->kr_attrs = true;
    }
    for (int i = 0; i < count; ++i) {
        const TcGemmItem& x = items[i];
        const int a_inner = a_kmajor ? x.K : x.M;
        if (x.M < 1 || x.N < 1 || x.K < 1 || (a_inner % 8) != 0 || (x.N % 8) != 0) {
            st->err = "tensor-core refresh GEMM: row pitches must be multiples of 16 bytes";
            return MOARA_ERR_UNSUPPORTED;
        }
        if (x.B_lo != nullptr && (a_kmajor || x.A_lo != nullptr)) {
            st->err = "tensor-core refresh GEMM: B in two planes goes with one MN-major plane of A";
            return MOARA_ERR_UNSUPPORTED;
        }
    }
    // sub-launches: items without a residual plane, with A's, with B's
    auto kind = [](const TcGemmItem& x) { return x.A_lo != nullptr ? 1 : x.B_lo != nullptr ? 2 : 0; };
    for (int with_lo = 0; with_lo < 3; ++with_lo) {
        std::vector<int> sel;
        for (int i = 0; i < count; ++i)
            if (kind(items[i]) == with_lo) sel.push_back(i);
        // longest K first, so that the last CTAs to start are short ones
        std::stable_sort(sel.begin(), sel.end(), [&](int a, int b) { return items[a].K > items[b].K; });
        for (size_t c0 = 0; c0 < sel.size(); c0 += kKrGroup) {
            const int cnt = static_cast<int>(std::min<size_t>(kKrGroup, sel.size() - c0));
            KrParams& kp = st->pr;
            std::memset(&kp, 0, sizeof(kp));
            int total = 0;
            for (int q = 0; q < cnt; ++q) {
                const int it = sel[c0 + q];
                const TcGemmItem& x = items[it];
                const uint64_t a_cols = a_kmajor ? x.K : x.M, a_rows = a_kmajor ? x.M : x.K;
                bool ok = encode_bf16_2d(st->encode, &kp.amap[q], x.A, a_cols, a_rows, 64, 64);
                if (with_lo == 1) ok = ok && encode_bf16_2d(st->encode, &kp.lmap[q], x.A_lo, a_cols, a_rows, 64, 64);
                if (with_lo == 2) ok = ok && encode_bf16_2d(st->encode, &kp.lmap[q], x.B_lo, x.N, x.K, 64, 64);
                ok = ok && encode_bf16_2d(st->encode, &kp.bmap[q], x.B, x.N, x.K, 64, 64);
                if (!ok) {
                    st->err = "cuTensorMapEncodeTiled failed for a refresh operand";
                    return MOARA_ERR_CUDA;
                }
                kp.out[q] = x.out;
                kp.out_bf[q] = x.out_bf16;
                kp.out_lo[q] = x.out_lo;
                kp.M[q] = x.M; kp.N[q] = x.N; kp.K[q] = x.K;
                kp.ktri[q] = x.ktri;
                kp.lower[q] = x.lower;
                kp.tiles_n[q] = (x.N + KR_BN - 1) / KR_BN;
                kp.tile_start[q] = total;
                total += ((x.M + KR_BM - 1) / KR_BM) * kp.tiles_n[q];
            }
            kp.tile_start[cnt] = total;
            kp.count = cnt;
            kp.status = st->d_status;
            kp.wait_limit = st->wait_limit;
            if (total == 0) continue;
            // CTA pairs where one tile's K outlasts what all tiles take on every
            // SM (a pair works it off in half the time)
            double longest = 0.0, work = 0.0;
            for (int q = 0; q < cnt; ++q) {
                const TcGemmItem& x = items[sel[c0 + q]];
                longest = std::max(longest, 1.0 * x.K);
                for (int i0 = 0; i0 < x.M; i0 += KR_BM)
                    work += 1.0 * x.K * (((x.lower ? std::min(x.N, i0 + KR_BM) : x.N) + KR_BN - 1) / KR_BN);
            }
            work /= st->sms;
            const bool pair = std::max(0.5 * longest, 1.1 * work) < 0.95 * std::max(longest, work);
            auto single = a_kmajor ? (with_lo == 0 ? kr_product<true, 0> : kr_product<true, 1>)
                                   : (with_lo == 0 ? kr_product<false, 0>
                                                   : with_lo == 1 ? kr_product<false, 1> : kr_product<false, 2>);
            auto paired = a_kmajor ? (with_lo == 0 ? kr_pair<true, 0> : kr_pair<true, 1>)
                                   : (with_lo == 0 ? kr_pair<false, 0>
                                                   : with_lo == 1 ? kr_pair<false, 1> : kr_pair<false, 2>);
            auto fn = pair ? paired : single;
            // (the pairs' cluster shape is the kernel's own)
            const cudaError_t e = launch(fn, pair ? 2 * total : total, KR_THREADS, KR_SMEM, s, 1, kp);
            if (e != cudaSuccess) {
                st->err = cudaGetErrorString(e);
                return MOARA_ERR_CUDA;
            }
            ++*launches;
        }
    }
    return MOARA_OK;
}

// out (cols x ld_out, bf16) = in^T for in (rows x cols, bf16, row pitch
// cols); columns rows..ld_out-1 of the output are zero.  32 x 32 tiles.
__global__ void __launch_bounds__(256) k_transpose_pad_bf16(const uint16_t* __restrict__ in, uint16_t* out,
                                                           int rows, int cols, int ld_out) {
    __shared__ uint16_t t[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int tr = (ld_out + 31) / 32, tc = (cols + 31) / 32;
    for (int tile = blockIdx.x; tile < tr * tc; tile += gridDim.x) {
        const int bi = tile / tc, bj = tile - bi * tc;      // input rows 32 bi.., columns 32 bj..
        for (int r = ty; r < 32; r += 8) {
            const int i = bi * 32 + r, j = bj * 32 + tx;
            t[r][tx] = (i < rows && j < cols) ? in[(long long)i * cols + j] : static_cast<uint16_t>(0);
        }
        __syncthreads();
        for (int r = ty; r < 32; r += 8) {
            const int j = bj * 32 + r, i = bi * 32 + tx;    // output row j, column i
            if (j < cols && i < ld_out) out[(long long)j * ld_out + i] = t[tx][r];
        }
        __syncthreads();
    }
}

cudaError_t tc_transpose_bf16(const uint16_t* in, uint16_t* out, int rows, int cols, cudaStream_t s,
                              int64_t* launches) {
    const int tiles = ((rows + 31) / 32) * ((cols + 31) / 32);
    k_transpose_pad_bf16<<<std::max(1, std::min(tiles, 152 * 8)), 256, 0, s>>>(in, out, rows, cols, rows);
    ++*launches;
    return cudaGetLastError();
}

__global__ void k_align_finish(const double* acc, float* S, int n) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const double dot = acc[3 * q], na = acc[3 * q + 1], gg = acc[3 * q + 2];
    const double den = sqrt(na) * sqrt(gg);
    S[q] = den > 0.0 ? static_cast<float>(dot / den) : 0.0f;
}

int tc_alignment(TcState* st, const moara_hparams& hp, int n_mod, const int* ids, const void* const* G,
                 float* S_out, double* acc, cudaStream_t s, int64_t* launches) {
    const int B = hp.block_size;
    if (!(B == 8 || B == 16 || B == 32 || B == 64 || B == 128)) {
        st->err = "alignment on tensor cores needs a block size in {8, 16, 32, 64, 128}";
        return MOARA_ERR_UNSUPPORTED;
    }
    for (int q = 0; q < n_mod; ++q) {
        const int id = ids[q];
        const TcMod* md = (id >= 0 && id < static_cast<int>(st->mods.size())) ? &st->mods[id] : nullptr;
        if (md == nullptr || md->Vhi == nullptr || md->Vlo == nullptr || md->Pb == nullptr) {
            st->err = "alignment: module is not on the tensor-core path";
            return MOARA_ERR_UNSUPPORTED;
        }
    }
    tc_init(st);
    int rc = tc_upload(st);
    if (rc != MOARA_OK) return rc;
    // 1. block norms M (into the module's norm buffer) and V = V_hi + V_lo
    for (int c0 = 0; c0 < n_mod; c0 += kTcGroup) {
        const int cnt = std::min(kTcGroup, n_mod - c0);
        K0Params& p0 = st->p0;
        std::memset(&p0, 0, sizeof(p0));
        p0.count = cnt;
        p0.hilo = 1;
        p0.do_mag = 1;                   // writes the norms; Optimizer_M is not launched
        p0.decomp_eps = hp.decomp_eps;
        long long acc_items = 0;
        for (int q = 0; q < cnt; ++q) {
            const TcMod& md = st->mods[ids[c0 + q]];
            const int segs = (md.n + K0_SEG - 1) / K0_SEG;
            p0.start[q] = acc_items;
            p0.p[q] = K0Item{static_cast<const uint16_t*>(G[c0 + q]), md.Vhi, md.Vlo, md.mag, nullptr, nullptr,
                             nullptr, md.m, md.n, md.kb, segs};
            acc_items += static_cast<long long>(md.m) * segs;
        }
        p0.start[cnt] = acc_items;
        const cudaError_t e = launch(k0_plain(B), st->sms * 3, 256, 0, s, 1, p0);
        ++*launches;
        if (e != cudaSuccess) {
            st->err = "alignment decomposition launch failed";
            return MOARA_ERR_CUDA;
        }
    }
    // 2. R = P^T V (r x n), or V Q (m x r) with a right projector, V in two
    //    planes, as two bf16 planes in the module's N buffer
    std::vector<TcGemmItem> g1[2];
    for (int q = 0; q < n_mod; ++q) {
        const TcMod& md = st->mods[ids[q]];
        if (!md.right) {
            TcGemmItem g{md.Pb, nullptr, md.Vhi, nullptr, md.Nb, md.r, md.n, md.m, 0, md.Nb + (size_t)md.r * md.n};
            g.B_lo = md.Vlo;
            g1[0].push_back(g);
        } else {
            g1[1].push_back(TcGemmItem{md.Vhi, md.Vlo, md.Pb, nullptr, md.Nb, md.m, md.r, md.n, 0,
                                       md.Nb + (size_t)md.m * md.r});
        }
    }
    for (int side = 0; side < 2; ++side) {
        if (g1[side].empty()) continue;
        rc = tc_gemm_bf16(st, side, g1[side].data(), static_cast<int>(g1[side].size()), s, launches);
        if (rc != MOARA_OK) return rc;
    }
    // 3. P R, or R Q^T, reduced against G
    if (cudaMemsetAsync(acc, 0, sizeof(double) * 3 * (size_t)n_mod, s) != cudaSuccess) {
        st->err = "alignment accumulator reset failed";
        return MOARA_ERR_CUDA;
    }
    for (int c0 = 0; c0 < n_mod; c0 += kTcGroup) {
        const int cnt = std::min(kTcGroup, n_mod - c0);
        const std::vector<int> chunk(ids + c0, ids + c0 + cnt);
        K2AlignParams p2{};
        p2.wait_limit = st->wait_limit;
        p2.mods = st->d_mods; p2.maps = st->d_maps; p2.status = st->d_status;
        p2.acc = acc + 3 * (size_t)c0;
        int clusters = 0;
        TcState::Tiles* tl = nullptr;
        if (st->tiles.count(chunk) > 0) {
            tl = tc_tiles(st, chunk);
        } else if (st->align_lists < kAlignLists) {
            cudaStreamCaptureStatus cap = cudaStreamCaptureStatusActive;
            if (cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone)
                tl = tc_tiles(st, chunk);
            if (tl != nullptr) ++st->align_lists;
            else cudaGetLastError();            // not to be had now (another thread records a graph): in turn
        }
        if (tl != nullptr) {
            p2.cta_start = tl->k2_start; p2.tiles = tl->k2;
            clusters = tl->g2;
            for (int q = 0; q < cnt; ++q) p2.G[q] = static_cast<const uint16_t*>(G[c0 + q]);
        } else {
            std::vector<int> order(cnt);
            for (int q = 0; q < cnt; ++q) order[q] = q;
            std::stable_sort(order.begin(), order.end(),
                             [&](int a, int b) { return st->mods[chunk[a]].r > st->mods[chunk[b]].r; });
            p2.count = cnt;
            int tiles = 0;
            for (int q = 0; q < cnt; ++q) {
                const TcMod& md = st->mods[chunk[order[q]]];
                p2.G[q] = static_cast<const uint16_t*>(G[c0 + order[q]]);
                p2.mod[q] = chunk[order[q]];
                p2.call_idx[q] = order[q];
                p2.col_tiles[q] = (md.n + K2_BN - 1) / K2_BN;
                p2.start[q] = tiles;
                tiles += (md.m + 2 * K2_BM - 1) / (2 * K2_BM) * p2.col_tiles[q];
            }
            p2.start[cnt] = tiles;
            clusters = std::min(tiles, st->k2_clusters);
        }
        auto fn = B == 8    ? k2_backproject<8, false, true>
                  : B == 16 ? k2_backproject<16, false, true>
                  : B == 32 ? k2_backproject<32, false, true>
                  : B == 64 ? k2_backproject<64, false, true>
                            : k2_backproject<128, false, true>;
        const cudaError_t e = launch(fn, 2 * clusters, K2_THREADS, K2_SMEM, s, 1, p2);
        ++*launches;
        if (e != cudaSuccess) {
            st->err = "alignment product launch failed";
            return MOARA_ERR_CUDA;
        }
    }
    k_align_finish<<<(n_mod + 127) / 128, 128, 0, s>>>(acc, S_out, n_mod);
    ++*launches;
    if (cudaGetLastError() != cudaSuccess) {
        st->err = "alignment finish launch failed";
        return MOARA_ERR_CUDA;
    }
    return MOARA_OK;
}

int tc_split_v(TcState* st, const TcSplitItem* items, int count, int B, float decomp_eps, cudaStream_t s,
               int64_t* launches) {
    for (int c0 = 0; c0 < count; c0 += kTcGroup) {
        const int cnt = std::min(kTcGroup, count - c0);
        K0Params& p0 = st->p0;
        std::memset(&p0, 0, sizeof(p0));
        p0.count = cnt;
        p0.hilo = 1;
        p0.do_mag = 0;
        p0.decomp_eps = decomp_eps;
        long long acc = 0;
        for (int q = 0; q < cnt; ++q) {
            const TcSplitItem& x = items[c0 + q];
            const int segs = (x.n + K0_SEG - 1) / K0_SEG;
            p0.start[q] = acc;
            p0.p[q] = K0Item{static_cast<const uint16_t*>(x.G), x.Vhi, x.Vlo, nullptr, nullptr, nullptr, nullptr,
                             x.m, x.n, (x.n + B - 1) / B, segs};
            acc += static_cast<long long>(x.m) * segs;
        }
        p0.start[cnt] = acc;
        if (!(B == 8 || B == 16 || B == 32 || B == 64 || B == 128)) {
            st->err = "block size not supported on the tensor-core path";
            return MOARA_ERR_UNSUPPORTED;
        }
        const cudaError_t e = launch(k0_plain(B), st->sms * 3, 256, 0, s, 1, p0);
        if (e != cudaSuccess) {
            st->err = cudaGetErrorString(e);
            return MOARA_ERR_CUDA;
        }
        ++*launches;
    }
    return MOARA_OK;
}

int tc_gemm_split3(TcState* st, const TcSplitGemmItem* items, int count, int planes, cudaStream_t s,
                   int64_t* launches) {
    if (!st->ks_attrs) {
        cudaFuncSetAttribute(ks_product<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, KS_SMEM);
        cudaFuncSetAttribute(ks_product<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, KS_SMEM);
        st->ks_attrs = true;
    }
    if (planes != 2 && planes != 3) {
        st->err = "split-precision GEMM: 2 or 3 planes";
        return MOARA_ERR_INVALID_ARG;
    }
    for (int i = 0; i < count; ++i) {
        const TcSplitGemmItem& x = items[i];
        if (x.M < 1 || x.N < 1 || x.K < 1 || (x.M % 8) != 0 || (x.N % 8) != 0) {
            st->err = "split-precision GEMM: M and N must be multiples of 8";
            return MOARA_ERR_UNSUPPORTED;
        }
        const int ldo = x.ldo > 0 ? x.ldo : x.N;
        if (ldo < x.N || (ldo % 4) != 0 || (reinterpret_cast<uintptr_t>(x.out) & 15) != 0) {
            st->err = "split-precision GEMM: out must be 16-byte aligned with a row pitch >= N, a multiple of 4";
            return MOARA_ERR_UNSUPPORTED;
        }
    }
    // longest K first, so that the last CTAs to start are short ones
    std::vector<int> order(count);
    for (int i = 0; i < count; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return items[a].K > items[b].K; });
    for (int c0 = 0; c0 < count; c0 += kKsGroup) {
        const int cnt = std::min(kKsGroup, count - c0);
        // Tiles of 128 rows where the longest 256-row tile (its K) lasts longer
        // than all of them take on every SM: few tiles, or a tall Gram matrix
        // among short ones.  A 128-row tile costs about 5/8 of a 256-row one
        // (its operands are 3/4 of the bytes).  Seven tall three-plane Gram
        // matrices (132 tiles, K up to 11008) take 418 us instead of 572, a group of
        // l = 160 / 288 products 33 us instead of 48; 830 tiles 389 us with 128 rows,
        // 357 with 256.
        double longest = 0.0, total256 = 0.0, total128 = 0.0;
        for (int q = 0; q < cnt; ++q) {
            const TcSplitGemmItem& x = items[order[c0 + q]];
            longest = std::max(longest, 1.0 * x.K);
            for (int i0 = 0; i0 < x.M; i0 += 128) {
                const int c128 = x.lower ? std::min(x.N, i0 + 128) : x.N;
                total128 += 0.625 * x.K * ((c128 + KS_BN - 1) / KS_BN);
                if (i0 % 256 == 0) total256 += 1.0 * x.K * (((x.lower ? std::min(x.N, i0 + 256) : x.N) + KS_BN - 1) / KS_BN);
            }
        }
        const int bm = std::max(0.625 * longest, total128 / st->sms) < std::max(longest, total256 / st->sms) ? 128 : 256;
        KsParams& kp = st->ps;
        std::memset(&kp, 0, sizeof(kp));
        int total = 0;
        for (int q = 0; q < cnt; ++q) {
            const TcSplitGemmItem& x = items[order[c0 + q]];
            bool ok = true;
            for (int pl = 0; pl < 3; ++pl) {
                ok = ok && encode_bf16_2d(st->encode, &kp.amap[q][pl], x.A + (size_t)pl * x.a_plane, x.M, x.K, 64, 32);
                ok = ok && encode_bf16_2d(st->encode, &kp.bmap[q][pl], x.B + (size_t)pl * x.b_plane, x.N, x.K, 64, 32);
            }
            if (!ok) {
                st->err = "cuTensorMapEncodeTiled failed for a split-precision operand";
                return MOARA_ERR_CUDA;
            }
            kp.out[q] = x.out;
            kp.M[q] = x.M; kp.N[q] = x.N; kp.K[q] = x.K;
            kp.ktri[q] = x.ktri;
            kp.ldo[q] = x.ldo > 0 ? x.ldo : x.N;
            kp.sub[q] = x.sub;
            kp.lower[q] = x.lower;
            kp.tiles_n[q] = (x.N + KS_BN - 1) / KS_BN;
            kp.tile_start[q] = total;
            total += ((x.M + bm - 1) / bm) * kp.tiles_n[q];
        }
        kp.tile_start[cnt] = total;
        kp.count = cnt;
        kp.bm = bm;
        kp.status = st->d_status;
        kp.wait_limit = st->wait_limit;
        if (total == 0) continue;
        const cudaError_t e = launch(planes == 3 ? ks_product<3> : ks_product<2>, total, KR_THREADS, KS_SMEM, s, 1, kp);
        if (e != cudaSuccess) {
            st->err = cudaGetErrorString(e);
            return MOARA_ERR_CUDA;
        }
        ++*launches;
    }
    return MOARA_OK;
}

}  // namespace moara
