// Tensor-core (tcgen05) path of Eq. 19: every mode product runs as 128-row
// tiles of pencils (M) against the zero-padded n x n eigenvector block (K = N =
// n rounded up to 16) held in shared memory, accumulating in TMEM.
//
// Precision (KX_F16X3): both operands are split into fp16 hi + lo halves after
// scaling by a power of two (2^14 for V, |V| <= 1; per item for the data), and
// D = A_hi B_hi + A_hi B_lo + A_lo B_hi is accumulated in fp32.  Each half has
// 11 significant bits, so the product keeps ~22 bits; the power-of-two scales
// are undone exactly in the epilogue.
//
// Passes over a chunk of items (pair products or caller vectors), all in the
// natural grid layout (x1 fastest) of fp32 scratch:
//   X3F  rho = psi_i psi_j (prologue), contract x3 with V3   [A MN-major]
//   X2F  contract x2 with V2                                  [A MN-major]
//   X1   contract x1 with V1, scale by f(Lambda) (+ Parseval energy), contract
//        back with V1^T                                       [A K-major]
//   X2I  contract k2 with V2^T                                [A MN-major]
//   X3I  contract k3 with V3^T, write phi (pair mode) or f(L)b (vector mode)
// then acc_kernel adds g_j psi_j phi_ij and g_i psi_i phi_ij, group by group, one thread
// per four grid points with a block of orbitals and their sums resident.
//
// Each pass kernel is persistent (one CTA per SM) and warp-specialised:
//   warps 0-7   epilogue (TMEM lane quadrant = warp % 4, one tile row per
//               thread; warps 0-3 and 4-7 take alternate column blocks)
//   warps 8-17  producers: global fp32 -> scale -> fp16 hi/lo -> shared stage (20 warps
//               are what 96 registers a thread allow)
//   warp 18     TMEM allocation and MMA issue (one thread)
//   warp 19     tile metadata, ahead of both
// with an S-deep ring of shared A stages and two TMEM accumulator slots, so
// loads, MMAs and stores of consecutive tiles overlap.
#include "kx_internal.h"
#include "kx_conv.cuh"
#include "kx_tc_ptx.cuh"

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <string>

namespace kx {
namespace {

enum PassKind { P_X3F = 0, P_X2F = 1, P_X1 = 2, P_X2I = 3, P_X3I = 4 };

constexpr int kEpiWarps = 8;   // two per TMEM lane quadrant, alternate 16/32-column blocks
constexpr int kProdWarps = 10;
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kProdThreads = 32 * kProdWarps;
constexpr int kProdGroups = 2;                            // producer groups work on alternate tiles
constexpr int kGroupThreads = kProdThreads / kProdGroups;
constexpr int kMmaWarp = kEpiWarps + kProdWarps;
constexpr int kMetaWarp = kMmaWarp + 1;
constexpr int kThreads = 32 * (kEpiWarps + kProdWarps + 2);
constexpr int kMetaRing = 8;  // >= the tiles a producer can be ahead of the epilogue (stages + 2 slots) + 1
constexpr int kMaxStages = 4;
constexpr size_t kSmemBudget = 218 * 1024;  // dynamic; ~7 KB of static shared memory beside it

// Optional per-role cycle counters of the pass kernels (compile with -DKX_ROLE_CLOCKS): each
// CTA writes kClk counters to PassArgs::clk[blockIdx.x * kClk + k].
constexpr int kClk = 12;
#ifdef KX_ROLE_CLOCKS
long long *g_clkbuf = nullptr;
#define KX_CLK_NOW() clock64()
#define KX_CLK_ADD(k, t0) (clk_acc[(k)] += clock64() - (t0))
#else
#define KX_CLK_NOW() 0LL
#define KX_CLK_ADD(k, t0) ((void)(t0))
#endif

// Shared-memory layout of the A operand (no swizzle, 8x8 fp16 core matrices of
// 128 contiguous bytes).  Core matrices sit kCoreStride = 144 bytes apart
// (128 + 16 of padding) so that a warp writing one 16-byte row into each of
// eight neighbouring core matrices hits eight different bank groups.
//   MN-major (8 rows contiguous in a core-matrix row):
//     (m, k) at (m/8)*144 + (k/8)*(16*144) + (k%8)*16 + (m%8)*2
//     descriptor: K-direction offset 16*144, M-direction offset 144
//   K-major (8 k contiguous in a core-matrix row), nkc = np/8:
//     (m, k) at (m/8)*(nkc*144) + (k/8)*144 + (m%8)*16 + (k%8)*2
//     descriptor: K-direction offset 144, M-direction offset nkc*144
constexpr int kCoreStride = 144;
__host__ __device__ constexpr size_t a_half_bytes(int np) { return (size_t)np * 16 * kCoreStride / 8; }

struct PassArgs {
    int n1, n2, n3;
    int nc;                // contraction length of this pass
    int np;                // nc rounded up to 16 (MMA K and N)
    int stages;            // shared A stages in the ring
    long long rows_pp;     // rows (pencils) per item
    long long total_rows;  // items * rows_pp
    long long N;
    const float *in;
    float *out;
    const __half *Vs;      // [2][np*np]: hi block, lo block (8x8 core-matrix order)
    const int2 *pairs;     // pair mode: (i, j) of each item of the chunk
    const float *psi32;    // [n_orb][N]
    const float *orb_max;  // [n_orb] max |psi|
    const float *src_max;  // vector mode: per-item max |b|
    int rhs_mode;
    const float *in_max;   // per-item max |input| (passes after X3F)
    float *out_max;        // per-item max |output| (nullable)
    const float *f32;      // f(Lambda), natural layout
    float mid_bound;       // fmax * sqrt(n1)
    double *e_partial;     // per-CTA energy partial (nullable)
    int energy_only;
    const double *occ;
    double *xout;          // vector mode output of X3I (fp64)
    int *status;
    long long timeout_cycles;
    long long *clk;        // role counters (only with KX_ROLE_CLOCKS)
};

__device__ __forceinline__ void ld8(const float *p, float *v) {
    float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    float4 b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// One k-step leaves the second accumulator unwritten: the epilogues then add zeros
// (one branch per chunk; a select and a bound test per element made the last stage
// three times as long as the others at the same number of values).
__device__ __forceinline__ void zero16(float *v) {
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = 0.f;
}

// f(Lambda) of 8 columns of one row: the table holds [k3][k1 / 4][k2][k1 % 4], so that
// the lanes of a warp (rows k2) read neighbouring 16-byte pieces; `ld4` = 4 n2.
__device__ __forceinline__ void ld8f(const float *p, int ld4, float *v) {
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    const float4 b = __ldg(reinterpret_cast<const float4 *>(p + ld4));
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

template <int PASS>
__device__ __forceinline__ float item_in_max(const PassArgs &a, long long item) {
    if (PASS == P_X3F) {
        if (a.rhs_mode) return a.src_max[item];
        int2 ij = a.pairs[item];
        return a.orb_max[ij.x] * a.orb_max[ij.y];
    }
    return a.in_max[item];
}

// What the producers and the epilogue need to know about one tile, per group of
// 8 rows (a group never straddles two items: every n is a multiple of 8).  Finding
// it takes divisions and two or three dependent loads (item, pair, maxima),
// about 1.5 k cycles, and both the producers and the epilogue spent them per tile (24-28%
// of the epilogue's time at 96^3).  A warp of its own fetches it up to kMetaRing tiles
// ahead: X3F 3.31 -> 2.95 ms, X3I 2.85 -> 2.63 ms per apply at 96^3 / 64 orbitals.
// In the MN-major passes row (m, k) of group g reads p0[g] + k * kstride + m % 8, in
// the K-major one row m reads the n1 values at p0[g] + (m % 8) n1.
struct TileMeta {
    const float *p0[16];   // nullptr: rows past the end
    const float *p1[16];   // second orbital of the pair product (X3F pair mode)
    long long obase[16];   // first output element of the group's first row
    double w[16];          // X1: energy weight of the item
    int item[16];
    int foff[16];          // X1: offset of the group's first row in the f table
    float scale[16];       // power-of-two split scale of the source
    int exp_[16];          // its exponent
    float in_max[16];
};

// Lane g < 16 of the metadata warp: group g of a tile.
template <int PASS>
__device__ __forceinline__ void make_meta(const PassArgs &a, long long tile, TileMeta &d, int g) {
    const long long n12 = (long long)a.n1 * a.n2;
    const long long R0 = tile * 128 + 8 * g;  // < 2^31: 32-bit division below
    if (R0 >= a.total_rows) {
        d.p0[g] = nullptr;
        if (PASS == P_X3F) d.p1[g] = nullptr;
        d.obase[g] = 0;
        d.w[g] = 0.0;
        d.item[g] = 0;
        d.foff[g] = 0;
        d.scale[g] = 0.f;
        d.exp_[g] = 0;
        d.in_max[g] = 0.f;
        return;
    }
    const unsigned rpp = (unsigned)a.rows_pp;
    const long long item = (unsigned)R0 / rpp, local = (unsigned)R0 - (unsigned)item * rpp;
    const float mx = item_in_max<PASS>(a, item);
    const int e = scale_exp(mx);
    d.item[g] = (int)item;
    d.in_max[g] = mx;
    d.exp_[g] = e;
    d.scale[g] = pow2f(e);
    long long off;  // of the group's first row inside the item
    if (PASS == P_X1) {
        off = local * a.n1;
        const int k3 = (unsigned)local / (unsigned)a.n2, k2 = (unsigned)local % (unsigned)a.n2;  // rows (k3, k2)
        d.foff[g] = (k3 * (a.n1 >> 2) * a.n2 + k2) * 4;
        double w = 0.0;
        if (a.e_partial != nullptr && !a.rhs_mode) {
            const int2 ij = a.pairs[item];
            w = (ij.x == ij.y) ? 1.0 : 2.0;
            if (a.occ) w *= a.occ[ij.x] * a.occ[ij.y];
        }
        d.w[g] = w;
    } else if (PASS == P_X2F || PASS == P_X2I) {
        const long long k3 = (unsigned)local / (unsigned)a.n1, x1 = (unsigned)local % (unsigned)a.n1;  // rows (k3, x1)
        off = k3 * n12 + x1;
    } else {  // rows = positions
        off = local;
    }
    d.obase[g] = item * a.N + off;
    if (PASS == P_X3F && !a.rhs_mode) {
        const int2 ij = a.pairs[item];
        d.p0[g] = a.psi32 + (long long)ij.x * a.N + off;
        d.p1[g] = a.psi32 + (long long)ij.y * a.N + off;
    } else {
        d.p0[g] = a.in + item * a.N + off;
        if (PASS == P_X3F) d.p1[g] = nullptr;
    }
}

template <int PASS, int U, bool TWO>
__device__ __forceinline__ void produce_tile_u(const PassArgs &a, const TileMeta &d, uint8_t *Ahi, uint8_t *Alo,
                                               int ptid) {
    const int np = a.np;
    const int nkc = np >> 3;
    const int ntask = 16 * np;  // 128 rows x np columns / 8
    const unsigned magic = (65536u + (unsigned)nkc - 1u) / (unsigned)nkc;  // t / nkc == (t * magic) >> 16 for t < 2^11
    const int kstride = (PASS == P_X3F || PASS == P_X3I) ? a.n1 * a.n2 : a.n1;
    for (int t0 = ptid; t0 < ntask; t0 += kGroupThreads * U) {
        float v[U][8];
        float u[TWO ? U : 1][8];
        // issue every load of the batch first (padding tasks read nothing)
#pragma unroll
        for (int r = 0; r < U; ++r) {
            const int t = t0 + r * kGroupThreads;
            const float *p0 = nullptr;
            const float *p1 = nullptr;
            bool ok = false;
            if (t < ntask) {
                if (PASS == P_X1) {
                    // lanes walk the 8-value chunks of one row, then the next row: contiguous reads
                    const int m = (int)(((unsigned)t * magic) >> 16), kc = t - m * nkc;
                    p0 = d.p0[m >> 3];
                    ok = p0 != nullptr && kc * 8 < a.nc;
                    if (ok) p0 += (m & 7) * a.n1 + kc * 8;
                } else {
                    // lanes walk the 16 row groups at one k, then the next k: 16 x 32 contiguous bytes
                    const int g = t & 15, k = t >> 4;
                    p0 = d.p0[g];
                    ok = p0 != nullptr && k < a.nc;
                    if (ok) {
                        p0 += k * kstride;
                        if (TWO) p1 = d.p1[g] + k * kstride;
                    }
                }
            }
            if (ok) {
                ld8(p0, v[r]);
                if (TWO) ld8(p1, u[TWO ? r : 0]);
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c) v[r][c] = 0.f;
                if (TWO) {
#pragma unroll
                    for (int c = 0; c < 8; ++c) u[TWO ? r : 0][c] = 0.f;
                }
            }
        }
        // then scale, split and store (offsets and scales re-derived from t)
#pragma unroll
        for (int r = 0; r < U; ++r) {
            const int t = t0 + r * kGroupThreads;
            if (t >= ntask) continue;
            int off;
            float sc;
            if (PASS == P_X1) {
                const int m = (int)(((unsigned)t * magic) >> 16), kc = t - m * nkc;
                off = (m >> 3) * (nkc * kCoreStride) + kc * kCoreStride + (m & 7) * 16;
                sc = d.scale[m >> 3];
            } else {
                const int g = t & 15, k = t >> 4;
                off = g * kCoreStride + (k >> 3) * (16 * kCoreStride) + (k & 7) * 16;
                sc = d.scale[g];
            }
            float2 w[4];
            const float2 sc2 = make_float2(sc, sc);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                w[c] = make_float2(v[r][2 * c], v[r][2 * c + 1]);
                if (TWO) w[c] = mul2(w[c], make_float2(u[TWO ? r : 0][2 * c], u[TWO ? r : 0][2 * c + 1]));
                w[c] = mul2(w[c], sc2);
            }
            uint4 hi4, lo4;
            split8(w, hi4, lo4);
            *reinterpret_cast<uint4 *>(Ahi + off) = hi4;
            *reinterpret_cast<uint4 *>(Alo + off) = lo4;
        }
    }
}

// Producer side: stage one 128-row tile of the A operand (scaled, split).
// Task t covers 8 consecutive values: MN-major row group g = t%16 at k = t/16;
// K-major row m = t/nkc, chunk kc = t%nkc.  Consecutive lanes therefore read
// consecutive global addresses.  All loads of a batch of U tasks are issued before
// any is converted, so each thread keeps U*32 bytes in flight (twice that for the
// pair product's two orbitals, in batches of 4); U is what splits a thread's tasks
// into even batches (pass_batch).
template <int PASS, int U>
__device__ __forceinline__ void produce_tile(const PassArgs &a, const TileMeta &d, uint8_t *Ahi, uint8_t *Alo,
                                             int ptid) {
    if (PASS == P_X3F) {
        if (a.rhs_mode)
            produce_tile_u<PASS, 6, false>(a, d, Ahi, Alo, ptid);
        else
            produce_tile_u<PASS, 4, true>(a, d, Ahi, Alo, ptid);
    } else {
        produce_tile_u<PASS, U, false>(a, d, Ahi, Alo, ptid);
    }
}

// D = A_hi B_hi + A_hi B_lo + A_lo B_hi over K = np (single issuing thread).
// The tensor core rounds its fp32 accumulator toward zero at every instruction,
// so a long chain of large partial sums drifts low.  To keep that drift small
// the two small cross products are issued first into accumulator Da, and the
// hi*hi chain is split over Da (even k-steps) and Db (odd k-steps); the
// epilogue adds Da + Db with round-to-nearest.
template <int NKS>
__device__ __forceinline__ void issue_ksteps(uint32_t tmem_a, uint32_t tmem_b, uint32_t ah0, uint32_t al0, uint32_t a_up,
                                             uint32_t bh0, uint32_t bl0, uint32_t b_up, uint32_t a_inc, uint32_t b_inc,
                                             uint32_t idesc) {
#pragma unroll
    for (int ks = 0; ks < NKS; ++ks) {
        const uint32_t da = ks * a_inc, db = ks * b_inc;
        ptx::mma_f16_lo(tmem_a, ah0 + da, a_up, bl0 + db, b_up, idesc, ks > 0 ? 1u : 0u);
        ptx::mma_f16_lo(tmem_a, al0 + da, a_up, bh0 + db, b_up, idesc, 1u);
    }
#pragma unroll
    for (int ks = 0; ks < NKS; ++ks) {
        const uint32_t da = ks * a_inc, db = ks * b_inc;
        if (ks & 1)
            ptx::mma_f16_lo(tmem_b, ah0 + da, a_up, bh0 + db, b_up, idesc, ks > 1 ? 1u : 0u);
        else
            ptx::mma_f16_lo(tmem_a, ah0 + da, a_up, bh0 + db, b_up, idesc, 1u);
    }
}

__device__ __forceinline__ void issue_split_mma(uint32_t tmem_a, uint32_t tmem_b, uint32_t a_hi, uint32_t a_lo,
                                                bool a_kmajor, uint32_t v_hi, uint32_t v_lo, bool inverse, int np,
                                                int row_groups = 16) {
    const uint32_t idesc = ptx::idesc_f16(128, np, a_kmajor ? 0 : 1, inverse ? 0 : 1);
    const uint32_t a_lbo = a_kmajor ? (uint32_t)kCoreStride : (uint32_t)(row_groups * kCoreStride);
    const uint32_t a_sbo = a_kmajor ? (uint32_t)((np >> 3) * kCoreStride) : (uint32_t)kCoreStride;
    const uint32_t a_step = 2 * a_lbo;  // one k-step = two core matrices along K
    // V stored as 8x8 core matrices, row block of 8 x-rows = np*16 bytes.
    //   forward  (B[x][k] = V[x][k]): MN-major, K (=x) stride np*16, N (=k) stride 128
    //   inverse  (B[k][x] = V[x][k]): K-major,  K (=k) stride 128,   N (=x) stride np*16
    const uint32_t b_lbo = inverse ? 128u : (uint32_t)(np * 16);
    const uint32_t b_sbo = inverse ? (uint32_t)(np * 16) : 128u;
    const uint32_t b_step = inverse ? 256u : (uint32_t)(np * 32);
    // descriptors built once; a k-step advances the start-address field (16-byte units)
    const uint64_t ah = ptx::sdesc(a_hi, a_lbo, a_sbo), al = ptx::sdesc(a_lo, a_lbo, a_sbo);
    const uint64_t bh = ptx::sdesc(v_hi, b_lbo, b_sbo), bl = ptx::sdesc(v_lo, b_lbo, b_sbo);
    const uint32_t a_up = (uint32_t)(ah >> 32), b_up = (uint32_t)(bh >> 32);
    const uint32_t a_inc = a_step >> 4, b_inc = b_step >> 4;
#define KX_ISSUE(n)                                                                                               \
    case n:                                                                                                       \
        issue_ksteps<n>(tmem_a, tmem_b, (uint32_t)ah, (uint32_t)al, a_up, (uint32_t)bh, (uint32_t)bl, b_up, a_inc, \
                        b_inc, idesc);                                                                            \
        break;
    switch (np >> 4) {
        KX_ISSUE(1)
        KX_ISSUE(2)
        KX_ISSUE(3)
        KX_ISSUE(4)
        KX_ISSUE(5)
        KX_ISSUE(6)
        KX_ISSUE(7)
        KX_ISSUE(8)
        default: break;
    }
#undef KX_ISSUE
}

// One arrival for a warp, after everything its lanes did before (their own proxy
// fences included): 32 arrivals on one word would be served one by one.
__device__ __forceinline__ void warp_arrive(uint64_t *bar) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) ptx::mbar_arrive(bar);
}

// Bounded wait shared by all roles: gives up when the limit elapses or another
// role already gave up (then every role leaves its loop and the CTA exits).
__device__ __forceinline__ bool wait_bar(uint64_t *bar, uint32_t parity, const PassArgs &a, volatile int *abort) {
    const long long t0 = clock64();
    while (!ptx::mbar_try_wait(bar, parity)) {
        if (*abort) return false;
        if (clock64() - t0 > a.timeout_cycles) {
            *abort = 1;
            atomicExch(a.status, KX_ERR_TIMEOUT);
            return false;
        }
    }
    return true;
}

// Warp-uniform form for roles that follow the wait with warp-collective
// instructions (tcgen05.ld): every lane sees the same outcome.
__device__ __forceinline__ bool wait_bar_warp(uint64_t *bar, uint32_t parity, const PassArgs &a,
                                              volatile int *abort) {
    const bool ok = wait_bar(bar, parity, a, abort);
    return __all_sync(0xffffffffu, ok);
}

__device__ __forceinline__ void track_max(float *out_max, long long item, float m, bool valid) {
    if (out_max == nullptr) return;
    const long long item0 = __shfl_sync(0xffffffffu, item, 0);
    const bool same = __all_sync(0xffffffffu, !valid || item == item0);
    if (same) {
        float r = valid ? m : 0.f;
        for (int o = 16; o > 0; o >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
        if ((threadIdx.x & 31) == 0 && r > 0.f) atomicMax(reinterpret_cast<int *>(out_max + item0), __float_as_int(r));
    } else if (valid && m > 0.f) {
        atomicMax(reinterpret_cast<int *>(out_max + item), __float_as_int(m));
    }
}

struct Bars {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t tfull[2];
    uint64_t tempty[2];
    uint64_t tfull2[2];
    uint64_t mid_full[2];  // by tile parity: a warp may finish tile j + 1 before another arrives for tile j
    uint64_t drain;
    uint64_t meta_full[kMetaRing];
    uint64_t meta_empty[kMetaRing];
};

// X1 epilogue, inverse half of tile j: wait for its inverse MMA, unscale and
// store the row (float4 per 4 columns), track the maximum, release the slot.
__device__ __forceinline__ bool x1_inverse_half(const PassArgs &a, Bars &bars, uint32_t tmem, int q, int hcol, int j,
                                                int np, bool two_acc, const TileMeta &d, int m, volatile int *abort) {
    const int b = j & 1;
    if (!wait_bar_warp(&bars.tfull2[b], (uint32_t)((j >> 1) & 1), a, abort)) return false;
    ptx::tc_fence_after();
    const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * 2 * np);
    const uint32_t tb = ta + (uint32_t)np;
    const int g8 = m >> 3;
    const bool valid = d.p0[g8] != nullptr;
    float *orow = a.out + d.obase[g8] + (m & 7) * a.n1;
    const float unscale2 = pow2f(-(scale_exp(a.mid_bound * d.in_max[g8]) + kVScaleExp));
    float my_max = 0.f;
    for (int c = hcol; c < (np >> 4); c += 2) {
        float v[16], vb[16];
        ptx::tmem_ld16x2(ta + 16 * c, tb + 16 * c, v, vb);
        if (!two_acc) zero16(vb);
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) {  // store each 8-column half that lies inside the row
            if (!valid || 16 * c + 8 * h2 >= a.nc) continue;
            float wv[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                wv[k] = (v[8 * h2 + k] + vb[8 * h2 + k]) * unscale2;
                my_max = fmaxf(my_max, fabsf(wv[k]));
            }
            float4 *dst = reinterpret_cast<float4 *>(orow + 16 * c + 8 * h2);
            dst[0] = make_float4(wv[0], wv[1], wv[2], wv[3]);
            dst[1] = make_float4(wv[4], wv[5], wv[6], wv[7]);
        }
    }
    track_max(a.out_max, d.item[g8], my_max, valid);
    ptx::tc_fence_before();
    warp_arrive(&bars.tempty[b]);
    warp_arrive(&bars.meta_empty[j % kMetaRing]);
    return true;
}

template <int PASS, int U>
__global__ void __launch_bounds__(kThreads, 1) tc_pass_kernel(const PassArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int np = a.np;
    const int S = a.stages;
    const size_t half_bytes = a_half_bytes(np);
    const size_t stage_bytes = 2 * half_bytes;  // hi + lo
    uint8_t *Vhi = smem;
    uint8_t *Vlo = Vhi + np * np * 2;
    uint8_t *stage0 = Vlo + np * np * 2;
    __shared__ Bars bars;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_abort;
    __shared__ double s_red[kEpiWarps];
    __shared__ TileMeta smeta[kMetaRing];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool with_inv = (PASS == P_X1) && !a.energy_only;
#ifdef KX_ROLE_CLOCKS
    long long clk_acc[kClk] = {0};
#endif
    const uint32_t tcols = (4 * np <= 256) ? 256u : 512u;
    if (warp == kMmaWarp) {
        ptx::tmem_alloc(&tmem_slot, tcols);
        ptx::tmem_relinquish();
    }
    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            ptx::mbar_init(&bars.full[s], kGroupThreads / 32);
            ptx::mbar_init(&bars.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(&bars.tfull[b], 1);
            ptx::mbar_init(&bars.tempty[b], kEpiWarps);
            ptx::mbar_init(&bars.tfull2[b], 1);
        }
        for (int b = 0; b < 2; ++b) ptx::mbar_init(&bars.mid_full[b], kEpiWarps);
        ptx::mbar_init(&bars.drain, 1);
        for (int r = 0; r < kMetaRing; ++r) {
            ptx::mbar_init(&bars.meta_full[r], 16);
            ptx::mbar_init(&bars.meta_empty[r], kEpiWarps);
        }
        ptx::fence_mbar_init();
        s_abort = 0;
    }
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(a.Vs);
        uint4 *dst = reinterpret_cast<uint4 *>(Vhi);
        const int n16 = (2 * np * np * 2) / 16;
        for (int i = tid; i < n16; i += blockDim.x) dst[i] = __ldg(src + i);
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const long long n_tiles = (a.total_rows + 127) / 128;
    const int n_my = (int)((n_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x);  // tiles of this CTA
    const long long n12 = (long long)a.n1 * a.n2;
    const bool two_acc = (np >> 4) > 1;

    if (warp == kMmaWarp) {
        // ------------------------------------------------------------ MMA issue
        if (ptx::elect_one()) {
            const uint32_t sVhi = ptx::smem_u32(Vhi), sVlo = ptx::smem_u32(Vlo);
            const bool inv = (PASS == P_X2I || PASS == P_X3I);
            bool ok = true;
            const long long tm0 = KX_CLK_NOW();
            for (int it = 0; it <= n_my && ok; ++it) {
                if (it < n_my) {
                    const int s = it % S, b = it & 1;
                    long long tw = KX_CLK_NOW();
                    ok = wait_bar(&bars.full[s], (uint32_t)((it / S) & 1), a, &s_abort);
                    KX_CLK_ADD(5, tw);
                    tw = KX_CLK_NOW();
                    if (ok && it >= 2) ok = wait_bar(&bars.tempty[b], (uint32_t)(((it >> 1) - 1) & 1), a, &s_abort);
                    KX_CLK_ADD(6, tw);
                    if (!ok) break;
                    ptx::tc_fence_after();
                    const uint32_t sA = ptx::smem_u32(stage0 + s * stage_bytes);
                    const uint32_t da = tmem + (uint32_t)(b * 2 * np);
                    issue_split_mma(da, da + (uint32_t)np, sA, sA + (uint32_t)half_bytes, PASS == P_X1, sVhi,
                                    sVlo, inv, np);
                    if (!with_inv) ptx::mma_commit(&bars.empty[s]);  // X1 keeps the stage for its mid operand
                    ptx::mma_commit(&bars.tfull[b]);
                }
                if (with_inv && it >= 1) {
                    // inverse of tile j: its mid operand sits in tile j's own A stage
                    const int j = it - 1, b = j & 1, sj = j % S;
                    const long long tw = KX_CLK_NOW();
                    ok = wait_bar(&bars.mid_full[b], (uint32_t)((j >> 1) & 1), a, &s_abort);
                    KX_CLK_ADD(7, tw);
                    if (!ok) break;
                    ptx::tc_fence_after();
                    const uint32_t sM = ptx::smem_u32(stage0 + sj * stage_bytes);
                    const uint32_t da = tmem + (uint32_t)(b * 2 * np);
                    issue_split_mma(da, da + (uint32_t)np, sM, sM + (uint32_t)half_bytes, true, sVhi, sVlo, true,
                                    np);
                    ptx::mma_commit(&bars.empty[sj]);
                    ptx::mma_commit(&bars.tfull2[b]);
                }
            }
            KX_CLK_ADD(4, tm0);
            if (!ok) {
                // a wait gave up: one more bounded wait for the MMAs already issued
                ptx::mma_commit(&bars.drain);
                ptx::mbar_wait_bounded(&bars.drain, 0, a.timeout_cycles);
            }
        }
        __syncwarp();
    } else if (warp == kMetaWarp) {
        // ------------------------------------------------------------ tile metadata
        if (lane < 16) {
            for (int it = 0; it < n_my; ++it) {
                const int r = it % kMetaRing;
                if (it >= kMetaRing &&
                    !wait_bar(&bars.meta_empty[r], (uint32_t)((it / kMetaRing - 1) & 1), a, &s_abort))
                    break;
                make_meta<PASS>(a, blockIdx.x + (long long)it * gridDim.x, smeta[r], lane);
                ptx::mbar_arrive(&bars.meta_full[r]);
            }
        }
        __syncwarp();
    } else if (warp >= kEpiWarps) {
        // ------------------------------------------------------------ producers
        const int ptid = tid - kEpiThreads;
        const int grp = ptid / kGroupThreads, gtid = ptid % kGroupThreads;
        const long long tp0 = KX_CLK_NOW();
        for (int it = grp; it < n_my; it += kProdGroups) {  // groups take alternate tiles
            const int s = it % S, r = it % kMetaRing;
            long long tw = KX_CLK_NOW();
            if (!wait_bar_warp(&bars.meta_full[r], (uint32_t)((it / kMetaRing) & 1), a, &s_abort)) break;
            KX_CLK_ADD(2, tw);
            // the tile into L2 while its stage is still in use: the producers' loads start from
            // memory only then (X3I 2.59 -> 2.22 ms per apply at 96^3 / 64 orbitals, the separate
            // passes at 120 x 112 x 120 / 16: X2F 0.37 -> 0.31, X1, which holds a stage through
            // both of its products, 0.79 -> 0.72 ms).  X3F's orbitals are in L2 already.
            // Not for a first tile, which has no wait to hide it behind, and not unrolled (the
            // longer code cost calls of a few tiles 1 of 40 us).
            if (it < S) {
            } else if (PASS == P_X1) {
                const int row8 = 8 * a.n1;  // eight contiguous rows per group
#pragma unroll 1
                for (int e = 32 * gtid; e < 16 * row8; e += 32 * kGroupThreads) {
                    const int g = e / row8;
                    if (smeta[r].p0[g] != nullptr) ptx::prefetch_l2(smeta[r].p0[g] + (e - g * row8));
                }
            } else if (PASS != P_X3F || a.rhs_mode) {
                const int g = gtid & 15;  // one prefetch per line: at its start or where a run of groups begins
                const float *p = smeta[r].p0[g];
                const long long ks = (PASS == P_X2F || PASS == P_X2I) ? a.n1 : (long long)a.n1 * a.n2;
                if (p != nullptr && (g == 0 || p != smeta[r].p0[g - 1] + 8 ||
                                     (reinterpret_cast<uintptr_t>(p) & 127) == 0))
#pragma unroll 1
                    for (int k = gtid >> 4; k < a.nc; k += kGroupThreads / 16) ptx::prefetch_l2(p + k * ks);
            }
            tw = KX_CLK_NOW();
            if (it >= S && !wait_bar_warp(&bars.empty[s], (uint32_t)(((it / S) - 1) & 1), a, &s_abort)) break;
            KX_CLK_ADD(1, tw);
            tw = KX_CLK_NOW();
            uint8_t *Ahi = stage0 + s * stage_bytes;
            produce_tile<PASS, U>(a, smeta[r], Ahi, Ahi + half_bytes, gtid);
            ptx::fence_proxy_async_smem();
            warp_arrive(&bars.full[s]);
            KX_CLK_ADD(3, tw);
        }
        KX_CLK_ADD(0, tp0);
    } else {
        // ------------------------------------------------------------ epilogue
        const int q = warp & 3, hcol = warp >> 2;  // lane quadrant, column half
        const int m = 32 * q + lane;  // TMEM lane == tile row of this thread
        const int nch = np >> 4;      // 16-column chunks
        double e_acc = 0.0;
        bool aborted = false;
        const long long te0 = KX_CLK_NOW();
        for (int it = 0; it < n_my; ++it) {
            const int b = it & 1;
            // row information and the per-item scale do not depend on the MMA:
            // take them (and fetch X1's first f chunk) before waiting for it
            const int r = it % kMetaRing, g8 = m >> 3;
            if (!wait_bar_warp(&bars.meta_full[r], (uint32_t)((it / kMetaRing) & 1), a, &s_abort)) break;
            const bool valid = smeta[r].p0[g8] != nullptr;
            const int item = smeta[r].item[g8];
            const long long obase = smeta[r].obase[g8] + (PASS == P_X1 ? (m & 7) * a.n1 : (m & 7));
            const int e_in = smeta[r].exp_[g8];
            const float in_mx = smeta[r].in_max[g8];
            const double w_item = (PASS == P_X1) ? smeta[r].w[g8] : 0.0;
            const float *frow = (PASS == P_X1) ? a.f32 + smeta[r].foff[g8] + 4 * (m & 7) : nullptr;
            const int ld4 = 4 * a.n2;
            float fpre[16];
            if (PASS == P_X1) {
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) {
                    if (valid && 16 * hcol + 8 * h2 < a.nc) {
                        ld8f(frow + (4 * hcol + 2 * h2) * ld4, ld4, fpre + 8 * h2);
                    } else {
#pragma unroll
                        for (int k = 0; k < 8; ++k) fpre[8 * h2 + k] = 0.f;
                    }
                }
            }
            long long tw = KX_CLK_NOW();
            if (!wait_bar_warp(&bars.tfull[b], (uint32_t)((it >> 1) & 1), a, &s_abort)) break;
            // the tile's producers are done with its metadata as well (their stage fed this MMA)
            // (X1 needs it once more, in the tile's inverse half)
            if (!with_inv) warp_arrive(&bars.meta_empty[r]);
            KX_CLK_ADD(9, tw);
            tw = KX_CLK_NOW();
            ptx::tc_fence_after();
            const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * 2 * np);
            const uint32_t tb = ta + (uint32_t)np;
            const float unscale = pow2f(-(e_in + kVScaleExp));
            float my_max = 0.f;

            if (PASS == P_X1) {
                // forward half of tile it: energy, f scaling, mid operand into the tile's own A stage
                const int e_mid = scale_exp(a.mid_bound * in_mx);
                const float s_mid = pow2f(e_mid);
                const double w = w_item;  // 0 for rows past the end and without the energy sum
                uint8_t *midh = stage0 + (it % S) * stage_bytes;
                float e_row = 0.f;
                for (int c = hcol; c < nch; c += 2) {
                    float fk[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k) fk[k] = fpre[k];
                    // prefetch the next chunk's f while this one is processed
                    // (nc is a multiple of 8: each 8-column half is either in or out)
#pragma unroll
                    for (int h2 = 0; h2 < 2; ++h2) {
                        if (valid && 16 * (c + 2) + 8 * h2 < a.nc) {
                            ld8f(frow + (4 * (c + 2) + 2 * h2) * ld4, ld4, fpre + 8 * h2);
                        } else {
#pragma unroll
                            for (int k = 0; k < 8; ++k) fpre[8 * h2 + k] = 0.f;
                        }
                    }
                    float v[16], vb[16];
                    float2 mid[8];
                    ptx::tmem_ld16x2(ta + 16 * c, tb + 16 * c, v, vb);
                    if (!two_acc) zero16(vb);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float2 y = mul2(add2(pair(v, k), pair(vb, k)), make_float2(unscale, unscale));
                        const float2 fy = mul2(pair(fk, k), y);
                        e_row = fmaf(fy.x, y.x, e_row);
                        e_row = fmaf(fy.y, y.y, e_row);
                        mid[k] = mul2(fy, make_float2(s_mid, s_mid));
                    }
                    if (with_inv) {
#pragma unroll
                        for (int h2 = 0; h2 < 2; ++h2) {
                            uint4 hi, lo;
                            split8(mid + 4 * h2, hi, lo);
                            const int off = (m >> 3) * ((np >> 3) * kCoreStride) + (2 * c + h2) * kCoreStride + (m & 7) * 16;
                            *reinterpret_cast<uint4 *>(midh + off) = hi;
                            *reinterpret_cast<uint4 *>(midh + half_bytes + off) = lo;
                        }
                    }
                }
                e_acc += w * (double)e_row;
                if (with_inv) {
                    ptx::fence_proxy_async_smem();
                    ptx::tc_fence_before();
                    warp_arrive(&bars.mid_full[b]);
                    KX_CLK_ADD(10, tw);
                    tw = KX_CLK_NOW();
                    // inverse half of the previous tile (its MMA ran while this tile's forward half was processed)
                    if (it >= 1) {
                        if (!x1_inverse_half(a, bars, tmem, q, hcol, it - 1, np, two_acc,
                                             smeta[(it - 1) % kMetaRing], m, &s_abort))
                            break;
                    }
                    KX_CLK_ADD(11, tw);
                    continue;  // tile it's TMEM slot is released by its inverse half
                }
            } else {
                // transposed write: one column per store, consecutive lanes = consecutive rows;
                // row base and column stride are computed once per tile
                // output (row r, column c) at base(r) + c * ostride: [k3 or x3][position] or [k3][k2 or x2][x1]
                const long long ostride = (PASS == P_X3F || PASS == P_X3I) ? n12 : (long long)a.n1;
                for (int cb = 32 * hcol; cb < np; cb += 64) {
                    float v[32], vb[32];
                    const long long tl = KX_CLK_NOW();
                    if (cb + 32 <= np) {
                        ptx::tmem_ld32x2(ta + cb, tb + cb, v, vb);
                    } else {
                        ptx::tmem_ld16x2(ta + cb, tb + cb, v, vb);
                    }
                    KX_CLK_ADD(11, tl);
                    if (!two_acc) zero16(vb);  // np == 16
                    if (!valid) continue;
                    // (nc is a multiple of 8: whole groups of 8 columns, no test per element)
                    if (PASS == P_X3I && a.rhs_mode) {
                        double *o = a.xout + obase + (long long)cb * ostride;
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            if (cb + 8 * g >= a.nc) break;
#pragma unroll
                            for (int k = 8 * g; k < 8 * g + 8; ++k, o += ostride)
                                *o = (double)((v[k] + vb[k]) * unscale);
                        }
                    } else {
                        float *o = a.out + obase + (long long)cb * ostride;
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            if (cb + 8 * g >= a.nc) break;
#pragma unroll
                            for (int k = 4 * g; k < 4 * g + 4; ++k, o += 2 * ostride) {
                                const float2 y = mul2(add2(pair(v, k), pair(vb, k)), make_float2(unscale, unscale));
                                my_max = fmaxf(my_max, fmaxf(fabsf(y.x), fabsf(y.y)));
                                o[0] = y.x;
                                o[ostride] = y.y;
                            }
                        }
                    }
                }
                track_max(a.out_max, item, my_max, valid);
            }
            ptx::tc_fence_before();
            warp_arrive(&bars.tempty[b]);
            KX_CLK_ADD(10, tw);
        }
        KX_CLK_ADD(8, te0);
        if (PASS == P_X1 && with_inv && n_my >= 1 && !s_abort)
            aborted = !x1_inverse_half(a, bars, tmem, q, hcol, n_my - 1, np, two_acc, smeta[(n_my - 1) % kMetaRing], m,
                                       &s_abort);
        (void)aborted;
        if (a.e_partial != nullptr) {
            double e = e_acc;
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
            if (lane == 0) s_red[warp] = e;
            ptx::named_bar(1, kEpiThreads);
            if (tid == 0) {
                double sum = 0.0;
                for (int w = 0; w < kEpiWarps; ++w) sum += s_red[w];
                a.e_partial[blockIdx.x] = sum;
            }
        }
    }
#ifdef KX_ROLE_CLOCKS
    if (a.clk != nullptr) {
        long long *o = a.clk + (long long)blockIdx.x * kClk;
        if (warp == kMmaWarp && lane == 0) { o[4] = clk_acc[4]; o[5] = clk_acc[5]; o[6] = clk_acc[6]; o[7] = clk_acc[7]; }
        if (tid == kEpiThreads) { o[0] = clk_acc[0]; o[1] = clk_acc[1]; o[2] = clk_acc[2]; o[3] = clk_acc[3]; }
        if (tid == 0) { o[8] = clk_acc[8]; o[9] = clk_acc[9]; o[10] = clk_acc[10]; o[11] = clk_acc[11]; }
    }
#endif
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, tcols);
    }
}

// ---------------------------------------------------------------------------
// Slab kernel: the three middle mode products of Eq. 19 for one k3 slice (an
// n1 x n2 plane of one item) without leaving the SM.  Per unit (item, k3):
//   M1  A1[x1][x2] (MN-major, from global) x V2      -> D1[x1][k2]
//   B   D1 -> A2[k2][x1] (MN-major, written by the thread owning row x1)
//   M2  A2 x V1                                      -> D2[k2][k1]
//   C   energy sum f Y^2; mid = f Y -> A3[k2][k1] (K-major, own row)
//   M3  A3 x V1^T                                    -> D3[k2][x1]
//   D   D3 -> A4[x1][k2] (MN-major, written by the thread owning row k2)
//   M4  A4 x V2^T                                    -> D4[x1][x2]
//   E   D4 -> global slice [x2][x1] (coalesced), per-item maximum
// E_x alone (ENERGY) stops after C.
// Two units are in flight: unit j uses TMEM slot and epilogue group j & 1 and A
// buffer j mod nbuf, so the two groups run their stage chains independently and
// the single MMA thread serves whichever group is ready.  Split scales are
// powers of two from bounds: each orthogonal mode product grows max|.| by at
// most sqrt(n), the scaling by at most fmax.
//
// What bounds it is each group's chain: four products of 18 MMAs (1.0-1.3 k cycles
// each at 96^2, on one tensor pipe for both groups) and the four stages between them
// (1.5-2.9 k cycles), ~18 k cycles a unit.  A third A buffer takes the split of the
// next plane (3.3 k cycles) out of the chain, where it stood beside stage E:
// 6.24 -> 5.34 ms per apply at 96^3 / 64 orbitals, 10.4 -> 8.65 at 80^3 / 96.  Small
// planes share a unit (slab_planes): 0.29 -> 0.17 ms at 56x40x48 / 24 orbitals.
// ---------------------------------------------------------------------------
struct SlabArgs {
    int n1, n2, n3, np1, np2;
    long long N;
    long long total_units;  // items * n3 / pp
    int pp;                 // planes per unit: 1, or 2 (4) where a plane fits 64 (32) rows
    const float *in;
    float *out;
    const __half *V1s, *V2s;
    const float *in_max;    // per item
    float *out_max;         // per item (nullable)
    const float *f32;
    float fmax, sq1, sq2;   // fmax, sqrt(n1), sqrt(n2) (each with a small margin)
    double *e_partial;
    const int2 *pairs;
    const double *occ;
    int rhs_mode;
    int stage_in;           // the input plane is bulk-copied into shared memory before it is split
    int share_v;            // V2 == V1 (same size, spacing and boundary): one shared copy
    int nbuf;               // A buffers (2 or 3)
    int *status;
    long long timeout_cycles;
};

constexpr int kSlabU = 6;            // producer loads in flight per thread
// Warp roles: 16 epilogue warps (warp w reads TMEM lane quadrant w % 4, the
// TMEM access rule; column half (w / 4) % 2; group w / 8), then 3 producer
// warps, then the MMA warp.  A plane of at most 96 rows leaves one quadrant (32:
// three) without rows: those epilogue warps work as producers instead (the split
// of a plane runs beside the last epilogue stage and took as long as it: slab
// time 8.54 -> 8.12 ms per apply at 96^3 / 64 orbitals).
constexpr int kSlabEpiWarps = 16;
constexpr int kSlabProdWarps = 3;
constexpr int kSlabMmaWarp = kSlabEpiWarps + kSlabProdWarps;
constexpr int kSlabThreads = 32 * (kSlabMmaWarp + 1);
constexpr int kSlabMaxBuf = 3;
// Units whose constants are kept: a slot is refilled eight units on, when two later
// units of the same group have been through their stages.
constexpr int kSlabRing = 8;

// Planes of a unit: small ones share the 128 rows of a product (consecutive k3 of one
// item; n3 is a multiple of 8), plane p on the rows from 128 p / pp on.  Everything but
// the row offsets is per row, so stages and products serve all of them at once.
__host__ __device__ constexpr int slab_planes(int npm) { return npm <= 32 ? 4 : npm <= 64 ? 2 : 1; }
// An A buffer holds only the row groups (8 rows) of the quadrants in use, a product's
// remaining rows up to 128 read what lies behind (their results are never read):
// hi + lo 41.5 KB at 96^2 instead of 55.3.
__host__ __device__ constexpr int slab_quadrants(int npm) { return slab_planes(npm) > 1 ? 4 : (npm + 31) / 32; }
__host__ __device__ constexpr size_t slab_half_bytes(int npm) {
    return (size_t)(npm / 8) * 4 * slab_quadrants(npm) * kCoreStride;
}

struct SlabBars {
    uint64_t full[kSlabMaxBuf], empty[kSlabMaxBuf], tfull[2], ready[2], in_full, drain;
};

// Constants of one unit: unscale and rescale factors of its stages, output and f
// offsets, the item and its energy weight.
struct SlabUnit {
    float us2, u2, s3, us4, u4;
    int item, foff;
    double w;
    long long out0;
};

__device__ __forceinline__ bool slab_wait(uint64_t *bar, uint32_t parity, const SlabArgs &a, volatile int *abort) {
    const long long t0 = clock64();
    while (!ptx::mbar_try_wait(bar, parity)) {
        if (*abort) return false;
        if (clock64() - t0 > a.timeout_cycles) {
            *abort = 1;
            atomicExch(a.status, KX_ERR_TIMEOUT);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void store_split8(uint8_t *hi_base, uint8_t *lo_base, int off, const float2 *w) {
    uint4 h, l;
    split8(w, h, l);
    *reinterpret_cast<uint4 *>(hi_base + off) = h;
    *reinterpret_cast<uint4 *>(lo_base + off) = l;
}

// Epilogue stage B or D for one warp: D row m of a plane (a TMEM lane) becomes K
// column m of the next MN-major operand; 8 consecutive D columns (M values, from
// the plane's first row group gp on) per 16-byte store.  Rows m >= nrow (padding)
// give zeros; rows m >= nprow are not written.
__device__ __forceinline__ void slab_transpose_stage(uint32_t ta, uint32_t tb, int m, int gp, int h, int nrow,
                                                     int nprow, int ncol, bool two, float us, int kcore, uint8_t *Ahi,
                                                     uint8_t *Alo) {
    const int off_r = (m >> 3) * kcore + (m & 7) * 16 + gp * kCoreStride;
    if (m >= nrow) us = 0.f;  // padding rows hold zeros already: their operand rows were zero
    for (int c = 16 * h; c < ncol; c += 32) {
        float v[16], vb[16];
        ptx::tmem_ld16x2(ta + c, tb + c, v, vb);
        if (!two) zero16(vb);
        if (m < nprow) {
#pragma unroll
            for (int g8 = 0; g8 < 2; ++g8) {
                float2 w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    w[k] = mul2(add2(pair(v, 4 * g8 + k), pair(vb, 4 * g8 + k)), make_float2(us, us));
                store_split8(Ahi, Alo, ((c >> 3) + g8) * kCoreStride + off_r, w);
            }
        }
    }
}

template <bool ENERGY, bool MULTI>
__global__ void __launch_bounds__(kSlabThreads, 1) tc_slab_kernel(const SlabArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int np1 = a.np1, np2 = a.np2, npm = max(np1, np2);
    const int nbuf = a.nbuf;
    const int nq = slab_quadrants(npm);          // TMEM lane quadrants with rows
    const int rg = 4 * nq, kcore = rg * kCoreStride;
    const int pp = MULTI ? a.pp : 1;                      // planes per unit
    const int row_sh = !MULTI ? 7 : pp == 2 ? 6 : 5;      // log2 of the 128 / pp rows of each
    const size_t half_bytes = slab_half_bytes(npm);
    uint8_t *buf0 = smem;  // A buffers (hi | lo)
    uint8_t *V1hi = buf0 + nbuf * 2 * half_bytes;
    uint8_t *V1lo = V1hi + np1 * np1 * 2;
    uint8_t *V2hi = a.share_v ? V1hi : V1lo + np1 * np1 * 2;
    uint8_t *V2lo = V2hi + np2 * np2 * 2;
    float *sin = reinterpret_cast<float *>(V2lo + np2 * np2 * 2);  // input plane [x2][x1] (stage_in)
    __shared__ SlabBars bars;
    __shared__ SlabUnit units[kSlabRing];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_abort;
    __shared__ double s_red[kSlabEpiWarps];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n_help = 4 * (4 - nq);             // epilogue warps without rows
    const int helper = (warp < kSlabEpiWarps && (warp & 3) >= nq) ? (warp & 3) - nq + (4 - nq) * (warp >> 2) : -1;
    const int n_prod = 32 * (kSlabProdWarps + n_help);  // producer threads
    const int group_threads = 64 * nq;           // epilogue threads of a group
    if (warp == kSlabMmaWarp) {
        ptx::tmem_alloc(&tmem_slot, 512);
        ptx::tmem_relinquish();
    }
    if (tid == 0) {
        for (int b = 0; b < kSlabMaxBuf; ++b) {
            ptx::mbar_init(&bars.full[b], n_prod / 32);
            ptx::mbar_init(&bars.empty[b], 1);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(&bars.tfull[b], 1);
            ptx::mbar_init(&bars.ready[b], group_threads / 32);
        }
        ptx::mbar_init(&bars.in_full, 1);
        ptx::mbar_init(&bars.drain, 1);
        ptx::fence_mbar_init();
        s_abort = 0;
    }
    if (tid < kSlabEpiWarps) s_red[tid] = 0.0;
    {
        const uint4 *s1 = reinterpret_cast<const uint4 *>(a.V1s);
        const uint4 *s2 = reinterpret_cast<const uint4 *>(a.V2s);
        uint4 *d1 = reinterpret_cast<uint4 *>(V1hi);
        uint4 *d2 = reinterpret_cast<uint4 *>(V2hi);
        const int c1 = (4 * np1 * np1) / 16, c2 = (4 * np2 * np2) / 16;
        for (int i = tid; i < c1; i += blockDim.x) d1[i] = __ldg(s1 + i);
        if (!a.share_v)
            for (int i = tid; i < c2; i += blockDim.x) d2[i] = __ldg(s2 + i);
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const int n_my = (int)((a.total_units - blockIdx.x + gridDim.x - 1) / gridDim.x);
    const long long n12 = (long long)a.n1 * a.n2;
    constexpr int kLast = ENERGY ? 1 : 3;  // last product of a unit

    if (warp == kSlabMmaWarp) {
        // ---------------------------------------------------------------- MMA issue
        // Polls both slots and issues the next product of whichever is ready:
        // M1 of unit j needs its A1 (full) and the slot's previous unit through
        // its last stage; M2..M4 need the group's previous stage (ready).
        if (ptx::elect_one()) {
            const uint32_t sV1h = ptx::smem_u32(V1hi), sV1l = ptx::smem_u32(V1lo);
            const uint32_t sV2h = ptx::smem_u32(V2hi), sV2l = ptx::smem_u32(V2lo);
            int jn[2] = {0, 1}, sn[2] = {0, 0};
            int buf[2] = {0, 1}, par[2] = {0, 0};  // of unit jn[g]: A buffer and its use's parity
            bool ok = true;
            int idle = 0;
            long long last = clock64();
            while (ok && (jn[0] < n_my || jn[1] < n_my)) {
                bool progressed = false;
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    const int j = jn[g], st = sn[g];
                    if (j >= n_my) continue;
                    bool go;
                    if (st == 0)
                        go = ptx::mbar_test_wait(&bars.full[buf[g]], (uint32_t)par[g]) &&
                             (j < 2 || ptx::mbar_test_wait(&bars.ready[g], 1u));
                    else
                        go = ptx::mbar_test_wait(&bars.ready[g], (uint32_t)((st - 1) & 1));
                    if (!go) continue;
                    ptx::tc_fence_after();
                    const uint32_t sA = ptx::smem_u32(buf0 + buf[g] * 2 * half_bytes);
                    const uint32_t da = tmem + (uint32_t)(g * 2 * npm);
                    // M1: A1 (MN-major) x V2 forward; M2: A2 (MN-major) x V1 forward;
                    // M3: A3 (K-major) x V1^T; M4: A4 (MN-major) x V2^T
                    const bool ax2 = st == 0 || st == 3;
                    issue_split_mma(da, da + (uint32_t)npm, sA, sA + (uint32_t)half_bytes, st == 2, ax2 ? sV2h : sV1h,
                                    ax2 ? sV2l : sV1l, st >= 2, ax2 ? np2 : np1, rg);
                    ptx::mma_commit(&bars.tfull[g]);
                    if (st == kLast) {
                        ptx::mma_commit(&bars.empty[buf[g]]);
                        sn[g] = 0;
                        jn[g] += 2;
                        buf[g] += 2;
                        if (buf[g] >= nbuf) {
                            buf[g] -= nbuf;
                            par[g] ^= 1;
                        }
                    } else {
                        ++sn[g];
                    }
                    progressed = true;
                }
                if (progressed) {
                    idle = 0;
                } else if ((++idle & 31) == 0) {  // the clock and the abort flag now and then
                    const long long now = clock64();
                    if (idle == 32) last = now;
                    if (s_abort) {
                        ok = false;
                    } else if (now - last > a.timeout_cycles) {
                        s_abort = 1;
                        atomicExch(a.status, KX_ERR_TIMEOUT);
                        ok = false;
                    }
                }
            }
            if (!ok) {
                ptx::mma_commit(&bars.drain);
                ptx::mbar_wait_bounded(&bars.drain, 0, a.timeout_cycles);
            }
        }
        __syncwarp();
    } else if (warp >= kSlabEpiWarps || helper >= 0) {
        // ---------------------------------------------------------------- producers: A1 from global
        const int ptid = helper >= 0 ? 32 * (kSlabProdWarps + helper) + lane : tid - kSlabEpiWarps * 32;
        const int ngrp = np1 >> 3;            // row groups (x1) of a plane
        const int ptask = ngrp * np2;         // x np2 columns (x2)
        const int ntask = ptask * pp;         // x planes
        const unsigned gmagic = (65536u + (unsigned)ngrp - 1u) / (unsigned)ngrp;  // t / ngrp for t < 2^11
        const int nlines = (int)((n12 * 4 * pp) >> 7);  // 128-byte lines of a unit's planes (n1 % 8 == 0)
        const uint32_t plane_bytes = (uint32_t)(n12 * 4 * pp);
        const unsigned n3u = (unsigned)(a.n3 / pp);  // units per item
        // task t: plane, 8-row group and column; source offset (0 with `in` false: padding) and A offset
        auto task = [&](int t, bool &in, int &src, int &off) {
            int pl = 0;
            if (MULTI) {
                pl = t >= ptask ? 1 : 0;
                if (pp > 2) pl += (t >= 2 * ptask ? 1 : 0) + (t >= 3 * ptask ? 1 : 0);
                t -= pl * ptask;
            }
            const int k = (int)(((unsigned)t * gmagic) >> 16), g = t - k * ngrp;
            in = 8 * g < a.n1 && k < a.n2;
            src = in ? pl * (int)n12 + k * a.n1 + 8 * g : 0;
            off = (g + (pl << (row_sh - 3))) * kCoreStride + (k >> 3) * kcore + (k & 7) * 16;
        };
        auto unit_item = [&](int it) { return (unsigned)(blockIdx.x + (long long)it * gridDim.x) / n3u; };
        auto plane_off = [&](int it) {
            const long long u = blockIdx.x + (long long)it * gridDim.x;
            const long long item = (unsigned)u / n3u, k3 = (unsigned)u % n3u;
            return item * a.N + k3 * pp * n12;
        };
        // stage_in: one thread copies the plane of the next unit into shared memory
        // (pieces of at most 16 KB) as soon as the previous plane has been split
        auto issue_plane = [&](int it) {
            ptx::fence_proxy_async_smem();
            ptx::mbar_arrive_expect_tx(&bars.in_full, plane_bytes);
            const char *src = reinterpret_cast<const char *>(a.in + plane_off(it));
            char *dst = reinterpret_cast<char *>(sin);
            for (uint32_t o = 0; o < plane_bytes; o += 16384u)
                ptx::bulk_load(dst + o, src + o, min(16384u, plane_bytes - o), &bars.in_full);
        };
        // item maxima and pairs are loaded one unit ahead, occupations with the unit
        const bool want_e = a.e_partial != nullptr && !a.rhs_mode;
        float next_max = 0.f;
        int2 next_ij = make_int2(0, 0);
        auto fetch = [&](int it) {
            const unsigned item = unit_item(it);
            next_max = __ldg(a.in_max + item);
            if (want_e && ptid == 0) next_ij = __ldg(a.pairs + item);
        };
        if (n_my > 0) fetch(0);
        int inflight = -1;  // unit whose plane copy thread 0 issued and has not yet waited for
        if (a.stage_in && ptid == 0 && n_my > 0) {
            issue_plane(0);
            inflight = 0;
        }
        int buf = 0, round = 0;  // A buffer of unit it, and how often it was used before
        for (int it = 0; it < n_my; ++it) {
            if (it + 2 < n_my) {
                // pull the plane of unit it+2 into L2 while this unit waits for its buffer
                const char *src = reinterpret_cast<const char *>(a.in + plane_off(it + 2));
                for (int l = ptid; l < nlines; l += n_prod) ptx::prefetch_l2(src + ((long long)l << 7));
            }
            bool ok = round == 0 || slab_wait(&bars.empty[buf], (uint32_t)((round - 1) & 1), a, &s_abort);
            if (ok && a.stage_in) ok = slab_wait(&bars.in_full, (uint32_t)(it & 1), a, &s_abort);
            if (ok && ptid == 0) inflight = -1;
            ok = ok && !s_abort;
            // with stage_in the producers meet at a named barrier below, so they leave together
            ok = a.stage_in ? ptx::named_bar_and(2, n_prod, ok) : (bool)__all_sync(0xffffffffu, ok);
            if (!ok) break;
            const float b1 = next_max;
            const int2 ij = next_ij;
            if (it + 1 < n_my) fetch(it + 1);
            const int e1 = scale_exp(b1);
            const float sc = pow2f(e1);
            uint8_t *Ahi = buf0 + buf * 2 * half_bytes;
            uint8_t *Alo = Ahi + half_bytes;
            if (ptid == 0) {
                // the unit's constants for the epilogue (it reads them after this unit's M1)
                SlabUnit &d = units[it % kSlabRing];
                const float b2 = b1 * a.sq2, b3 = a.fmax * a.sq1 * b2, b4 = a.sq1 * b3;
                const int e2 = scale_exp(b2), e3 = scale_exp(b3), e4 = scale_exp(b4);
                d.us2 = pow2f(e2 - e1 - kVScaleExp);
                d.u2 = pow2f(-(e2 + kVScaleExp));
                d.s3 = pow2f(e3);
                d.us4 = pow2f(e4 - e3 - kVScaleExp);
                d.u4 = pow2f(-(e4 + kVScaleExp));
                const unsigned u = (unsigned)(blockIdx.x + (long long)it * gridDim.x);
                const int item = (int)(u / n3u), k3 = (int)(u - (unsigned)item * n3u) * pp;
                d.item = item;
                d.foff = k3 * (int)n12;
                d.out0 = item * a.N + k3 * n12;
                double w = 0.0;
                if (want_e) {
                    w = (ij.x == ij.y) ? 1.0 : 2.0;
                    if (a.occ) w *= a.occ[ij.x] * a.occ[ij.y];
                }
                d.w = w;
            }
            if (a.stage_in) {
                // task: 8 rows x1 at one x2.  Two tasks' loads first, without branches between them
                // (batches of 3, 4 and 6 measured 1, 3 and 3% slower): a task past the end
                // repeats the last one, a padding one reads the plane's first values and scales them to
                // zero (an infinity or NaN there reaches the padding too; its item is lost with or without
                // that).  Row groups past np1 are never read (see the quadrants above).
                for (int t0 = ptid; t0 < ntask; t0 += 2 * n_prod) {
                    float4 x[2][2];
                    int off[2];
                    float scl[2];
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        bool in;
                        int so;
                        task(min(t0 + r * n_prod, ntask - 1), in, so, off[r]);
                        const float4 *src = reinterpret_cast<const float4 *>(sin + so);
                        x[r][0] = src[0];
                        x[r][1] = src[1];
                        scl[r] = in ? sc : 0.f;
                    }
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        if (t0 + r * n_prod >= ntask) break;
                        const float2 s2 = make_float2(scl[r], scl[r]);
                        const float2 w[4] = {mul2(make_float2(x[r][0].x, x[r][0].y), s2),
                                             mul2(make_float2(x[r][0].z, x[r][0].w), s2),
                                             mul2(make_float2(x[r][1].x, x[r][1].y), s2),
                                             mul2(make_float2(x[r][1].z, x[r][1].w), s2)};
                        store_split8(Ahi, Alo, off[r], w);
                    }
                }
                ptx::fence_proxy_async_smem();
                warp_arrive(&bars.full[buf]);
                // every producer has finished reading the plane: it may be overwritten
                ptx::named_bar(2, n_prod);
                if (ptid == 0 && it + 1 < n_my) {
                    issue_plane(it + 1);
                    inflight = it + 1;
                }
            } else {
                const float *slice = a.in + plane_off(it);
                for (int t0 = ptid; t0 < ntask; t0 += n_prod * kSlabU) {
                    float v[kSlabU][8];
#pragma unroll
                    for (int r = 0; r < kSlabU; ++r) {
                        bool in;
                        int so, off;
                        task(min(t0 + r * n_prod, ntask - 1), in, so, off);
                        if (in) {
                            ld8(slice + so, v[r]);
                        } else {
#pragma unroll
                            for (int c = 0; c < 8; ++c) v[r][c] = 0.f;
                        }
                    }
#pragma unroll
                    for (int r = 0; r < kSlabU; ++r) {
                        const int t = t0 + r * n_prod;
                        if (t >= ntask) continue;
                        bool in;
                        int so, off;
                        task(t, in, so, off);
                        float2 w[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) w[c] = mul2(pair(v[r], c), make_float2(sc, sc));
                        store_split8(Ahi, Alo, off, w);
                    }
                }
                ptx::fence_proxy_async_smem();
                warp_arrive(&bars.full[buf]);
            }
            if (++buf == nbuf) {
                buf = 0;
                ++round;
            }
        }
        // a plane copy still in flight after an early exit must land before the CTA leaves
        if (inflight >= 0) ptx::mbar_wait_bounded(&bars.in_full, (uint32_t)(inflight & 1), a.timeout_cycles);
    } else {
        // ---------------------------------------------------------------- epilogue: group g = warp / 8
        // Warp w of a group reads TMEM lanes 32*(w%4).. (its D rows) and the
        // 16-column chunks c = 16*h + 32*i, h = (w/4)%2.  tcgen05.ld is
        // warp-collective: every lane loads, only the stores are predicated per row.
        const int g = warp >> 3, q = warp & 3, h = (warp >> 2) & 1;
        const int row = 32 * q + lane;                      // TMEM lane == D row
        const int pl = MULTI ? row >> row_sh : 0, m = MULTI ? row & ((1 << row_sh) - 1) : row;  // plane, row of it
        const int m0 = m - lane;                            // the warp's first row of the plane
        const int gp = pl << (row_sh - 3);                  // the plane's first row group
        const bool two1 = (np1 >> 4) > 1, two2 = (np2 >> 4) > 1;
        const int nkc1 = np1 >> 3;
        const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(g * 2 * npm);
        const uint32_t tb = ta + (uint32_t)npm;
        const int ld4 = 4 * a.n2;
        double e_acc = 0.0;
        bool ok = true;
        int buf = g;
        for (int j = g; j < n_my && ok; j += 2) {
            const SlabUnit &U = units[j % kSlabRing];
            uint8_t *Ahi = buf0 + buf * 2 * half_bytes;
            uint8_t *Alo = Ahi + half_bytes;
            buf += 2;
            if (buf >= nbuf) buf -= nbuf;
            // ---- B: D1[x1][k2] -> A2[k2][x1]
            ok = __all_sync(0xffffffffu, slab_wait(&bars.tfull[g], 0u, a, &s_abort));
            if (!ok) break;
            ptx::tc_fence_after();
            if (m0 < np1)
                slab_transpose_stage(ta, tb, m, gp, h, a.n1, np1, np2, two2, U.us2, kcore, Ahi, Alo);
            ptx::fence_proxy_async_smem();
            ptx::tc_fence_before();
            warp_arrive(&bars.ready[g]);
            // ---- C: D2[k2][k1] = Y: energy sum f Y^2, mid = f Y -> A3[k2][k1] (K-major, own row)
            {
                const bool rowC = m < a.n2;
                const float *frow = a.f32 + U.foff + pl * (int)n12 + 4 * m;
                // f(Lambda) of this warp's first chunk; each further chunk's is fetched
                // while the previous one is processed
                float fr[2][16];
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const int c0 = 16 * h + 8 * hh;
                    if (rowC && c0 < a.n1) {
                        ld8f(frow + (c0 >> 2) * ld4, ld4, fr[0] + 8 * hh);
                    } else {
#pragma unroll
                        for (int k = 0; k < 8; ++k) fr[0][8 * hh + k] = 0.f;
                    }
                }
                ok = __all_sync(0xffffffffu, slab_wait(&bars.tfull[g], 1u, a, &s_abort));
                if (!ok) break;
                ptx::tc_fence_after();
                const float u2 = U.u2, s3 = U.s3;
                const int off_r = (row >> 3) * (nkc1 * kCoreStride) + (row & 7) * 16;
                float e_row = 0.f;
#pragma unroll
                for (int r = 0; r < kMaxN / 32; ++r) {
                    const int c = 16 * h + 32 * r;
                    if (c >= np1) break;
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const int c0 = c + 32 + 8 * hh;
                        if (rowC && c0 < a.n1) {
                            ld8f(frow + (c0 >> 2) * ld4, ld4, fr[(r + 1) & 1] + 8 * hh);
                        } else {
#pragma unroll
                            for (int k = 0; k < 8; ++k) fr[(r + 1) & 1][8 * hh + k] = 0.f;
                        }
                    }
                    float v[16], vb[16];
                    ptx::tmem_ld16x2(ta + c, tb + c, v, vb);
                    if (!two1) zero16(vb);
                    // (rows past n2 are never read back: no select for them)
                    float2 mid[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float2 y = mul2(add2(pair(v, k), pair(vb, k)), make_float2(u2, u2));
                        const float2 fy = mul2(pair(fr[r & 1], k), y);
                        e_row = fmaf(fy.x, y.x, e_row);
                        e_row = fmaf(fy.y, y.y, e_row);
                        if (!ENERGY) mid[k] = mul2(fy, make_float2(s3, s3));
                    }
                    if (!ENERGY) {
#pragma unroll
                        for (int hh = 0; hh < 2; ++hh)
                            store_split8(Ahi, Alo, off_r + ((c >> 3) + hh) * kCoreStride, mid + 4 * hh);
                    }
                }
                if (!ENERGY) ptx::fence_proxy_async_smem();
                ptx::tc_fence_before();
                const double w = U.w;
                warp_arrive(&bars.ready[g]);
                if (rowC) e_acc += w * (double)e_row;
            }
            if (ENERGY) continue;
            // ---- D: D3[k2][x1] -> A4[x1][k2]
            ok = __all_sync(0xffffffffu, slab_wait(&bars.tfull[g], 0u, a, &s_abort));
            if (!ok) break;
            ptx::tc_fence_after();
            if (m0 < np2)
                slab_transpose_stage(ta, tb, m, gp, h, a.n2, np2, np1, two1, U.us4, kcore, Ahi, Alo);
            ptx::fence_proxy_async_smem();
            ptx::tc_fence_before();
            warp_arrive(&bars.ready[g]);
            // ---- E: D4[x1][x2] -> slice [x2][x1] of the output, coalesced over x1
            ok = __all_sync(0xffffffffu, slab_wait(&bars.tfull[g], 1u, a, &s_abort));
            if (!ok) break;
            ptx::tc_fence_after();
            {
                const float u4 = U.u4;
                const int item = U.item;
                const bool valid = m < a.n1;
                float my_max = 0.f;
                if (m0 < a.n1) {
                    float *orow = a.out + U.out0 + pl * (int)n12 + m + (long long)(16 * h) * a.n1;
                    for (int c = 16 * h; c < np2; c += 32, orow += 32 * a.n1) {
                        float v[16], vb[16];
                        ptx::tmem_ld16x2(ta + c, tb + c, v, vb);
                        if (!two2) zero16(vb);
                        if (!valid) continue;
                        float *o = orow;
                        // (n2 is a multiple of 8: each half of the chunk is in or out)
#pragma unroll
                        for (int g8 = 0; g8 < 2; ++g8) {
                            if (c + 8 * g8 >= a.n2) break;
#pragma unroll
                            for (int k = 4 * g8; k < 4 * g8 + 4; ++k, o += 2 * a.n1) {
                                const float2 y = mul2(add2(pair(v, k), pair(vb, k)), make_float2(u4, u4));
                                my_max = fmaxf(my_max, fmaxf(fabsf(y.x), fabsf(y.y)));
                                o[0] = y.x;
                                o[a.n1] = y.y;
                            }
                        }
                    }
                }
                ptx::tc_fence_before();
                warp_arrive(&bars.ready[g]);
                track_max(a.out_max, item, my_max, valid);
            }
        }
        if (a.e_partial != nullptr) {
            double e = e_acc;
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
            if (lane == 0) s_red[warp] = e;
            ptx::named_bar(1, 2 * group_threads);
            if (tid == 0) {
                double sum = 0.0;
                for (int w = 0; w < kSlabEpiWarps; ++w) sum += s_red[w];
                a.e_partial[blockIdx.x] = sum;
            }
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kSlabMmaWarp) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, 512);
    }
}

// Accumulation of one chunk, group by group: one thread per W grid points visits a
// group's items in order, adding g_j psi_j phi_ij to orbital i and g_i psi_i phi_ij to
// orbital j in partial sums (one per orbital of the group's two blocks), then adds
// those to the orbitals' running sums.  Every sum is owned by one thread per launch
// and groups and chunks run in a fixed order, so the result is deterministic.
//
// Bound by memory traffic.  Consecutive groups share one of their two orbital
// blocks (the pair list walks rows or columns of block pairs), so a thread keeps two
// blocks, orbitals and running sums, in its own column of shared memory and exchanges
// only the block that changes: per pair 4N bytes of phi and 3N of orbitals and sums
// (with both blocks exchanged 6N).  An orbital's sum starts from zero at its first
// group and leaves negated, as Vx psi, after its last (no fill before, no pass after).
// The state lives in the thread, so groups need no barrier; the 16 phi loads of a
// group and those of a new block are issued together.  96^3, 64 orbitals: 2.15 ms
// an apply (7N bytes a pair: 13 GB, 6.0 TB/s) against 3.20 ms with both blocks
// exchanged per group and 0.29 ms for the fills and the negating pass.  W = 4 where
// rows are whole 16-byte pieces, else 1.
constexpr int kAccThreads = 128;
constexpr int kGroupItems = kOrbBlock * kOrbBlock;

template <int W> struct alignas(4 * W) Pts {
    float v[W];
};
template <int W> __device__ __forceinline__ Pts<W> ld_pts(const float *p) {
    return *reinterpret_cast<const Pts<W> *>(p);
}

struct AccArgs {
    const float *phi;
    const Group *groups;
    int g0, g1, item0, n_orb;
    const int2 *item_slot;
    const int2 *orb_span;   // first and last group of each orbital
    const float *psi32;
    const double *occ;
    float *acc;
    double *vx;
    int vx_vec;             // vx rows are 16-byte aligned
    int acc_init;           // the sums start from acc (multipole correction), not from zero
    long long N;
    const double *e_partial;  // energy partials of the chunk, added by the first CTA (nullable)
    int e_count;
    double e_factor;
    double *ex;
};

template <int W>
__global__ void __launch_bounds__(kAccThreads, 3) acc_kernel(const AccArgs a) {
    using P = Pts<W>;
    extern __shared__ __align__(16) unsigned char acc_sm[];
    P(*ps)[kAccThreads] = reinterpret_cast<P(*)[kAccThreads]>(acc_sm);  // orbitals of the two blocks
    P(*av)[kAccThreads] = ps + kGroupSlots;                             // their running sums
    P(*as)[kAccThreads] = av + kGroupSlots;                             // a partial group's sums
    const int tid = threadIdx.x, lane = tid & 31;
    const long long x = (blockIdx.x * (long long)kAccThreads + tid) * W;
    const bool valid = x < a.N;
    if (blockIdx.x == 0 && a.e_count > 0) {
        __shared__ double red[kAccThreads / 32];
        double s = 0.0;
        for (int b = tid; b < a.e_count; b += kAccThreads) s += a.e_partial[b];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) red[tid >> 5] = s;
        __syncthreads();
        if (tid == 0) *a.ex += a.e_factor * ((red[0] + red[1]) + (red[2] + red[3]));
    }
    int cur[2] = {-1, -1};  // blocks held in the halves [0, 4) and [4, 8)
    float gl = 1.f;         // occupation of slot `lane`
    // running sums of half h back to memory before group g: Vx psi if the orbital is done
    auto evict = [&](int h, int g) {
        if (cur[h] < 0) return;
#pragma unroll
        for (int s = 0; s < kOrbBlock; ++s) {
            const int o = cur[h] * kOrbBlock + s;
            if (o >= a.n_orb) break;
            const P v = av[4 * h + s][tid];
            if (!valid) continue;
            if (__ldg(a.orb_span + o).y < g) {
                double *d = a.vx + (long long)o * a.N + x;
                if (W == 4 && a.vx_vec) {
                    reinterpret_cast<double2 *>(d)[0] = make_double2(-(double)v.v[0], -(double)v.v[W > 1 ? 1 : 0]);
                    reinterpret_cast<double2 *>(d)[1] =
                        make_double2(-(double)v.v[W > 2 ? 2 : 0], -(double)v.v[W > 3 ? 3 : 0]);
                } else {
#pragma unroll
                    for (int c = 0; c < W; ++c) d[c] = -(double)v.v[c];
                }
            } else {
                *reinterpret_cast<P *>(a.acc + (long long)o * a.N + x) = v;
            }
        }
    };
    auto load = [&](int h, int blk, int g) {
        cur[h] = blk;
        P p[kOrbBlock], q[kOrbBlock];
#pragma unroll
        for (int s = 0; s < kOrbBlock; ++s) {
            const int o = blk * kOrbBlock + s;
#pragma unroll
            for (int c = 0; c < W; ++c) p[s].v[c] = q[s].v[c] = 0.f;
            if (o < a.n_orb && valid) {
                p[s] = ld_pts<W>(a.psi32 + (long long)o * a.N + x);
                if (a.acc_init || __ldg(a.orb_span + o).x != g) q[s] = ld_pts<W>(a.acc + (long long)o * a.N + x);
            }
        }
#pragma unroll
        for (int s = 0; s < kOrbBlock; ++s) {
            ps[4 * h + s][tid] = p[s];
            av[4 * h + s][tid] = q[s];
        }
        const int o = blk * kOrbBlock + (lane & 3);
        if ((lane >> 2) == h) gl = (a.occ && o < a.n_orb) ? (float)a.occ[o] : 1.f;
    };
    int4 next = __ldg(reinterpret_cast<const int4 *>(a.groups + a.g0));
    for (int g = a.g0; g < a.g1; ++g) {
        const int fi = next.x, ni = next.y, bi = next.z, bj = next.w;
        if (g + 1 < a.g1) next = __ldg(reinterpret_cast<const int4 *>(a.groups + g + 1));
        P f[kGroupItems];
#pragma unroll
        for (int k = 0; k < kGroupItems; ++k) {
            if (k < ni && valid) {
                f[k] = ld_pts<W>(a.phi + (long long)(fi + k - a.item0) * a.N + x);
            } else {
#pragma unroll
                for (int c = 0; c < W; ++c) f[k].v[c] = 0.f;
            }
        }
        // halves of I and J: where they already are, if anywhere
        int hi;
        if (bj < 0)
            hi = cur[1] == bi ? 1 : 0;
        else
            hi = (cur[1] == bi || cur[0] == bj) && !(cur[0] == bi || cur[1] == bj) ? 1 : 0;
        const int hj = 1 - hi;
        if (cur[hi] != bi) {
            evict(hi, g);
            load(hi, bi, g);
        }
        if (bj >= 0 && cur[hj] != bj) {
            evict(hj, g);
            load(hj, bj, g);
        }
        if (bj >= 0 && ni == kGroupItems) {
            // a whole block pair: the partial sums stay in registers
            P si[kOrbBlock], sj[kOrbBlock], pj[kOrbBlock];
#pragma unroll
            for (int s = 0; s < kOrbBlock; ++s) {
                const float gj = __shfl_sync(0xffffffffu, gl, 4 * hj + s);
                pj[s] = ps[4 * hj + s][tid];
#pragma unroll
                for (int c = 0; c < W; ++c) {
                    si[s].v[c] = sj[s].v[c] = 0.f;
                    pj[s].v[c] = gj * pj[s].v[c];
                }
            }
#pragma unroll
            for (int i = 0; i < kOrbBlock; ++i) {
                const float gi = __shfl_sync(0xffffffffu, gl, 4 * hi + i);
                P pi = ps[4 * hi + i][tid];
#pragma unroll
                for (int c = 0; c < W; ++c) pi.v[c] = gi * pi.v[c];
#pragma unroll
                for (int j = 0; j < kOrbBlock; ++j) {
#pragma unroll
                    for (int c = 0; c < W; ++c) {
                        si[i].v[c] = fmaf(pj[j].v[c], f[4 * i + j].v[c], si[i].v[c]);
                        sj[j].v[c] = fmaf(pi.v[c], f[4 * i + j].v[c], sj[j].v[c]);
                    }
                }
            }
#pragma unroll
            for (int s = 0; s < kOrbBlock; ++s) {
                P u = av[4 * hi + s][tid], v = av[4 * hj + s][tid];
#pragma unroll
                for (int c = 0; c < W; ++c) {
                    u.v[c] += si[s].v[c];
                    v.v[c] += sj[s].v[c];
                }
                av[4 * hi + s][tid] = u;
                av[4 * hj + s][tid] = v;
            }
        } else {
            // diagonal, ragged or cut block pairs: slots from the item table
            const int mi = 4 * hi, mj = bj >= 0 ? 4 * hj - kOrbBlock : 4 * hi;  // slots of J count on from 4
            P z;
#pragma unroll
            for (int c = 0; c < W; ++c) z.v[c] = 0.f;
#pragma unroll
            for (int s = 0; s < kGroupSlots; ++s) as[s][tid] = z;
#pragma unroll
            for (int k = 0; k < kGroupItems; ++k) {
                if (k >= ni) break;
                const int2 sl = __ldg(a.item_slot + fi + k);
                const int ii = mi + sl.x, jj = mj + sl.y;
                const float gj = __shfl_sync(0xffffffffu, gl, jj), gi = __shfl_sync(0xffffffffu, gl, ii);
                const P pj = ps[jj][tid];
                P u = as[ii][tid];
#pragma unroll
                for (int c = 0; c < W; ++c) u.v[c] = fmaf(gj * pj.v[c], f[k].v[c], u.v[c]);
                as[ii][tid] = u;
                if (ii != jj) {
                    const P pi = ps[ii][tid];
                    P v = as[jj][tid];
#pragma unroll
                    for (int c = 0; c < W; ++c) v.v[c] = fmaf(gi * pi.v[c], f[k].v[c], v.v[c]);
                    as[jj][tid] = v;
                }
            }
#pragma unroll
            for (int s = 0; s < kGroupSlots; ++s) {
                P u = av[s][tid];
                const P d = as[s][tid];
#pragma unroll
                for (int c = 0; c < W; ++c) u.v[c] += d.v[c];
                av[s][tid] = u;
            }
        }
    }
    evict(0, a.g1);
    evict(1, a.g1);
}
template <int W> constexpr size_t acc_smem() { return 3 * kGroupSlots * kAccThreads * sizeof(Pts<W>); }

// psi (fp64) -> psi32 and per-vector max |value|.
// *zero (nullable, the energy of the call) starts from 0.
__global__ void prep_kernel(const double *__restrict__ src, float *__restrict__ dst, float *__restrict__ vmax,
                            int n_vec, long long N, double *__restrict__ zero) {
    const int v = blockIdx.y;
    if (zero && blockIdx.x == 0 && v == 0 && threadIdx.x == 0) *zero = 0.0;
    float m = 0.f;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < N; x += (long long)gridDim.x * blockDim.x) {
        const float f = (float)src[(long long)v * N + x];
        dst[(long long)v * N + x] = f;
        m = fmaxf(m, fabsf(f));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > 0.f) atomicMax(reinterpret_cast<int *>(vmax + v), __float_as_int(m));
}

// Vx psi = -acc over n values (n % 4 == 0; both pointers 16-byte aligned).
__global__ void finalize_kernel(const float *__restrict__ acc, double *__restrict__ vx, long long n) {
    const float4 *a4 = reinterpret_cast<const float4 *>(acc);
    double2 *v2 = reinterpret_cast<double2 *>(vx);
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (n >> 2);
         e += (long long)gridDim.x * blockDim.x) {
        const float4 x = __ldg(a4 + e);
        v2[2 * e] = make_double2(-(double)x.x, -(double)x.y);
        v2[2 * e + 1] = make_double2(-(double)x.z, -(double)x.w);
    }
}

// The same for an output that is only 8-byte aligned.
__global__ void finalize_scalar_kernel(const float *__restrict__ acc, double *__restrict__ vx, long long n) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
        vx[e] = -(double)acc[e];
}

// e_x += factor sum partial[0 .. n), n <= 1024: strided partial sums and a fixed tree
// (one thread adding them took 10 us, a fifth of the smallest apply).
__global__ void __launch_bounds__(128) energy_add_kernel(const double *__restrict__ partial, int n, double factor,
                                                         double *e_x) {
    __shared__ double red[4];
    double s = 0.0;
    for (int b = threadIdx.x; b < n; b += 128) s += partial[b];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) *e_x += factor * ((red[0] + red[1]) + (red[2] + red[3]));
}

// Failure-path self-test: wait on an mbarrier phase that nothing completes; the
// bounded wait gives up and the status word records KX_ERR_TIMEOUT.
__global__ void selftest_wait_kernel(long long max_cycles, int *status) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        ptx::mbar_init(&bar, 1);
        ptx::fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0 && !ptx::mbar_wait_bounded(&bar, 0, max_cycles)) atomicExch(status, KX_ERR_TIMEOUT);
}

size_t stage_bytes_of(int np) { return 2 * a_half_bytes(np); }
constexpr size_t kStagingBytes = 0;

int pass_stages(int np, bool with_mid) {
    const size_t v = (size_t)4 * np * np;
    const size_t avail = kSmemBudget - v - kStagingBytes - (with_mid ? stage_bytes_of(np) : 0);
    return (int)std::max<size_t>(1, std::min<size_t>(kMaxStages, avail / stage_bytes_of(np)));
}

size_t pass_smem(int np, int stages, bool with_mid) {
    return (size_t)4 * np * np + (size_t)(stages + (with_mid ? 1 : 0)) * stage_bytes_of(np) + kStagingBytes + 1024;
}

// Producer batch of a pass kernel: a thread has ceil(16 np / kGroupThreads) tasks a
// tile; at np = 96 its 10 tasks take 2.60 ms as 5 + 5 and 2.70 as 8 + 2 (X3I per apply
// at 96^3 / 64 orbitals), at np = 80 its 8 are one batch.  Calls of a few tiles take the same
// either way (one or two vectors at 72^3 42 us with the rule, 43-45 with batches of 7 or 5;
// 80^3 to 128 x 128 x 64 within 1 us of the best).
int pass_batch(int np) {
    const int tasks = (16 * np + kGroupThreads - 1) / kGroupThreads;
    if (tasks == 9 || tasks == 10) return 5;
    return tasks == 8 || tasks <= 6 ? 8 : 7;
}

template <int PASS, int U>
int launch_pass_u(kx_plan *p, const PassArgs &a, int grid, size_t smem, cudaStream_t s) {
    if (int rc = raise_smem(p, reinterpret_cast<const void *>(tc_pass_kernel<PASS, U>), kSmemBudget + 1024)) return rc;
    tc_pass_kernel<PASS, U><<<grid, kThreads, smem, s>>>(a);
    KX_LAUNCH_CHECK("tc_pass_kernel launch");
    return KX_OK;
}

template <int PASS>
int launch_pass(kx_plan *p, PassArgs a, int axis, cudaStream_t s, int *grid_out) {
    a.nc = p->n[axis];
    a.np = p->np[axis];
    a.Vs = p->d_Vs[axis];
    a.n1 = p->n[0];
    a.n2 = p->n[1];
    a.n3 = p->n[2];
    a.N = (long long)p->N;
    a.status = p->d_status;
    a.timeout_cycles = 4000000000LL;  // ~2 s at the SM clock
#ifdef KX_ROLE_CLOCKS
    if (!g_clkbuf) cudaMallocManaged(&g_clkbuf, sizeof(long long) * kClk * 4096 * 5);
    a.clk = g_clkbuf + (long long)PASS * kClk * 4096;
#endif
    a.stages = pass_stages(a.np, false);  // X1's mid operand reuses its tile's A stage
    if (p->tune.pass_stages > 0) a.stages = std::min(a.stages, p->tune.pass_stages);
    const size_t smem = pass_smem(a.np, a.stages, false);
    const long long n_tiles = (a.total_rows + 127) / 128;
    const int grid = (int)std::max(1LL, std::min<long long>(n_tiles, (long long)p->num_sms));
    if (grid_out) *grid_out = grid;
    if (int rc = prof_begin(p, PK_X3F + PASS, s)) return rc;
    const int u = PASS == P_X3F ? 8 : pass_batch(a.np);  // X3F has its own batches
    int rc;
    if (PASS == P_X3F || u == 8) rc = launch_pass_u<PASS, 8>(p, a, grid, smem, s);
    else if (u == 7) rc = launch_pass_u<PASS, PASS == P_X3F ? 8 : 7>(p, a, grid, smem, s);
    else rc = launch_pass_u<PASS, PASS == P_X3F ? 8 : 5>(p, a, grid, smem, s);
    if (rc) return rc;
    return prof_end(p, s);
}

// axes 1 and 2 of the same size, spacing and boundary have the same eigenvectors
bool same_axes12(const kx_plan *p) { return p->n[0] == p->n[1] && p->h[0] == p->h[1] && p->bc[0] == p->bc[1]; }

// The slab kernel runs where V1, V2 and two full (128-row) A buffers fit in shared memory
// (planes up to ~104 x 104); what it needs is no more than that.
constexpr size_t kSlabSmemMax = 227 * 1024 - 1024;  // opt-in maximum less static shared memory
bool slab_fits(const kx_plan *p) {
    const int np1 = p->np[0], np2 = p->np[1], npm = std::max(np1, np2);
    return (size_t)4 * np1 * np1 + (size_t)4 * np2 * np2 + 4 * a_half_bytes(npm) + 1024 <= kSlabSmemMax;
}

// E_x alone through the slab kernel: its two products cost a unit nearly the same
// whatever the planes hold, the two passes it replaces go with their values.  Per call
// (40 orbitals), slab against passes: 48^3 0.48 / 0.45 ms, (80, 48, 64) 1.03 / 0.86 at
// 4608 and 3840 values a unit; (64, 48, 80) 0.84 / 0.86, 80^3 1.58 / 1.78, 96^3
// 2.57 / 3.12 at 6144, 6400 and 9216.  With one to nine orbitals the slab is ahead on every
// plane, by launches (four orbitals: 16^3 23 / 30 us, (80, 48, 64) 41 / 45, 96^3 67 / 82);
// the line is drawn where the calls are long.
bool slab_for_energy(const kx_plan *p) {
    return slab_planes(std::max(p->np[0], p->np[1])) * p->np[0] * p->np[1] >= 6000;
}

bool use_slab(const kx_plan *p) {
    if (const char *e = std::getenv("KX_SLAB")) return std::atoi(e) != 0;  // tuning override
    return p->tune.fuse_slab != 0;
}

// Mode 2 forward, mode 1 forward, f(Lambda) scaling (+ energy), mode 1 inverse
// and mode 2 inverse of R items in one launch; `in` holds the mode-3 forward
// output, `out` receives the input of the mode-3 inverse (both natural layout).
int launch_slab(kx_plan *p, long R, const float *in, const float *in_max, float *out, float *out_max,
                double *e_partial, const int2 *pairs, const double *occ, int rhs_mode, bool energy_only,
                cudaStream_t s, int *grid_out) {
    SlabArgs a{};
    a.n1 = p->n[0];
    a.n2 = p->n[1];
    a.n3 = p->n[2];
    a.np1 = p->np[0];
    a.np2 = p->np[1];
    a.N = (long long)p->N;
    a.pp = slab_planes(std::max(a.np1, a.np2));
    a.total_units = (long long)R * (a.n3 / a.pp);
    a.in = in;
    a.out = out;
    a.V1s = p->d_Vs[0];
    a.V2s = p->d_Vs[1];
    a.in_max = in_max;
    a.out_max = out_max;
    a.f32 = p->d_f32;
    a.fmax = (float)(p->fmax * 1.0001);
    a.sq1 = (float)(std::sqrt((double)a.n1) * 1.0001);
    a.sq2 = (float)(std::sqrt((double)a.n2) * 1.0001);
    a.e_partial = e_partial;
    a.pairs = pairs;
    a.occ = occ;
    a.rhs_mode = rhs_mode;
    a.status = p->d_status;
    a.timeout_cycles = 4000000000LL;  // ~2 s at the SM clock
    a.share_v = same_axes12(p) ? 1 : 0;
    const size_t base = (size_t)4 * a.np1 * a.np1 + (a.share_v ? 0 : (size_t)4 * a.np2 * a.np2) + 1024;
    const size_t buffer = 2 * slab_half_bytes(std::max(a.np1, a.np2));
    const size_t plane = (size_t)a.n1 * a.n2 * 4 * a.pp;
    // a third buffer first, then the staged input plane
    a.nbuf = base + 3 * buffer <= kSlabSmemMax ? 3 : 2;
    size_t smem = base + a.nbuf * buffer;
    a.stage_in = smem + plane <= kSlabSmemMax ? 1 : 0;
    if (a.stage_in) smem += plane;
    // at least 120 KB so that one CTA (and one 512-column TMEM allocation) sits on each SM
    smem = std::max<size_t>(smem, 120 * 1024);
    const int grid = (int)std::max(1LL, std::min<long long>(a.total_units, (long long)p->num_sms));
    if (grid_out) *grid_out = grid;
    int rc;
    if ((rc = prof_begin(p, PK_SLAB, s))) return rc;
    auto kernel = energy_only ? (a.pp > 1 ? tc_slab_kernel<true, true> : tc_slab_kernel<true, false>)
                              : (a.pp > 1 ? tc_slab_kernel<false, true> : tc_slab_kernel<false, false>);
    if ((rc = raise_smem(p, reinterpret_cast<const void *>(kernel), kSlabSmemMax))) return rc;
    kernel<<<grid, kSlabThreads, smem, s>>>(a);
    KX_LAUNCH_CHECK("tc_slab_kernel launch");
    return prof_end(p, s);
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

struct TcLayout {
    float *psi32, *acc, *T0, *T1, *orb_max, *mx;
    double *partial;
};

TcLayout carve(kx_plan *p, int n_vec, long chunk, bool with_acc) {
    TcLayout L{};
    uint8_t *b = reinterpret_cast<uint8_t *>(p->ws.ptr);
    size_t off = 0;
    auto take = [&](size_t bytes) { uint8_t *r = b + off; off += align256(bytes); return r; };
    L.psi32 = (float *)take(sizeof(float) * (size_t)n_vec * p->N);
    L.acc = with_acc ? (float *)take(sizeof(float) * (size_t)n_vec * p->N) : nullptr;
    const bool fft = p->precision == KX_FFT32;  // T1 holds complex values, more energy partials
    L.T0 = (float *)take(sizeof(float) * (size_t)chunk * p->N);
    L.T1 = (float *)take(sizeof(float) * (fft ? 2 : 1) * (size_t)chunk * p->N);
    L.orb_max = (float *)take(sizeof(float) * (size_t)n_vec);
    L.mx = (float *)take(sizeof(float) * 4 * (size_t)chunk);
    L.partial = (double *)take(sizeof(double) * (fft ? fft_partial_count(p, chunk) : 4096));
    return L;
}

float fmax_sqrt(const kx_plan *p) {
    // bound of |f(Lambda) (V1^T y)| / max|y| used for the mid-pass split scale
    return (float)(p->fmax * std::sqrt((double)p->n[0]) * 1.0001);
}

// ex += the energy of `grid` partials, now or, with e_count, later by acc_kernel.
int add_energy(kx_plan *p, const double *partial, int grid, double *ex, int *e_count, cudaStream_t s) {
    if (e_count) {
        *e_count = grid;
        return KX_OK;
    }
    if (int rc = prof_begin(p, PK_FINAL, s)) return rc;
    energy_add_kernel<<<1, 128, 0, s>>>(partial, grid, -0.5 * p->dV, ex);
    KX_LAUNCH_CHECK("energy_add_kernel launch");
    return prof_end(p, s);
}

// The five passes over R items: X3F writes T0, X2F T0->T1, X1 T1->T0, X2I
// T0->T1, X3I T1->T0 (or xout in vector mode).  mx holds four rows of per-item
// maxima, mx_stride apart.
int run_passes(kx_plan *p, PassArgs a, long R, float *T0, float *T1, float *mx, long mx_stride, double *ex,
               double *partial, bool energy_only, double *xout, cudaStream_t s, int *e_count = nullptr) {
    int rc;
    float *mx1 = mx, *mx2 = mx + mx_stride, *mx3 = mx + 2 * mx_stride, *mx4 = mx + 3 * mx_stride;
    a.rows_pp = (long long)p->n[0] * p->n[1];
    a.total_rows = R * a.rows_pp;
    a.out = T0;
    a.out_max = mx1;
    if ((rc = launch_pass<P_X3F>(p, a, 2, s, nullptr))) return rc;

    if (slab_fits(p) && use_slab(p) && (!energy_only || slab_for_energy(p))) {
        // X2F, X1 and X2I fused: T0 -> T1 without the intermediate round trips (E_x
        // alone: X2F and the forward half of X1)
        int grid = 0;
        if ((rc = launch_slab(p, R, T0, mx1, T1, mx4, ex ? partial : nullptr, a.pairs, a.occ, a.rhs_mode, energy_only,
                              s, &grid)))
            return rc;
        if (ex && (rc = add_energy(p, partial, grid, ex, energy_only ? nullptr : e_count, s))) return rc;
        if (energy_only) return KX_OK;
        a.e_partial = nullptr;
        a.energy_only = 0;
        a.rows_pp = (long long)p->n[0] * p->n[1];
        a.total_rows = R * a.rows_pp;
        a.in = T1;
        a.in_max = mx4;
        a.out = T0;
        a.out_max = nullptr;
        a.xout = xout;
        return launch_pass<P_X3I>(p, a, 2, s, nullptr);
    }

    a.rows_pp = (long long)p->n[2] * p->n[0];
    a.total_rows = R * a.rows_pp;
    a.in = T0;
    a.in_max = mx1;
    a.out = T1;
    a.out_max = mx2;
    if ((rc = launch_pass<P_X2F>(p, a, 1, s, nullptr))) return rc;

    a.rows_pp = (long long)p->n[2] * p->n[1];
    a.total_rows = R * a.rows_pp;
    a.in = T1;
    a.in_max = mx2;
    a.out = T0;
    a.out_max = mx3;
    a.e_partial = ex ? partial : nullptr;
    a.energy_only = energy_only ? 1 : 0;
    int grid = 0;
    if ((rc = launch_pass<P_X1>(p, a, 0, s, &grid))) return rc;
    if (ex && (rc = add_energy(p, partial, grid, ex, energy_only ? nullptr : e_count, s))) return rc;
    a.e_partial = nullptr;
    a.energy_only = 0;
    if (energy_only) return KX_OK;

    a.rows_pp = (long long)p->n[2] * p->n[0];
    a.total_rows = R * a.rows_pp;
    a.in = T0;
    a.in_max = mx3;
    a.out = T1;
    a.out_max = mx4;
    if ((rc = launch_pass<P_X2I>(p, a, 1, s, nullptr))) return rc;

    a.rows_pp = (long long)p->n[0] * p->n[1];
    a.total_rows = R * a.rows_pp;
    a.in = T1;
    a.in_max = mx4;
    a.out = T0;
    a.out_max = nullptr;
    a.xout = xout;
    return launch_pass<P_X3I>(p, a, 2, s, nullptr);
}

}  // namespace

long tc_default_chunk(const kx_plan *p, int n_orb) {
    (void)n_orb;
    if (p->tune.chunk_pairs > 0) return p->tune.chunk_pairs;
    if (const char *e = std::getenv("KX_CHUNK_PAIRS")) {  // tuning override (pairs per chunk)
        const long v = std::atol(e);
        if (v > 0) return v;
    }
    const size_t budget = (size_t)4 << 30;  // both chunk buffers together
    long c = (long)std::max<size_t>(1, budget / (2 * p->N * sizeof(float)));
    return std::max(1L, std::min<long>(c, 2048));
}

size_t tc_workspace_bytes(const kx_plan *p, int n_vec, long chunk) {
    const bool fft = p->precision == KX_FFT32;
    return align256(sizeof(float) * (size_t)n_vec * p->N) * 2 + align256(sizeof(float) * (size_t)chunk * p->N) +
           align256(sizeof(float) * (fft ? 2 : 1) * (size_t)chunk * p->N) + align256(sizeof(float) * n_vec) +
           align256(sizeof(float) * 4 * chunk) + align256(sizeof(double) * (fft ? fft_partial_count(p, chunk) : 4096)) +
           4096;
}

// Vx psi rows [o0, o1) = -acc (rows no group touches, with a multipole correction).
int finalize_rows(kx_plan *p, const float *acc, double *vx, int o0, int o1, cudaStream_t s) {
    if (o1 <= o0) return KX_OK;
    const long long n = (long long)(o1 - o0) * (long long)p->N;
    const size_t off = (size_t)o0 * p->N;
    if (int rc = prof_begin(p, PK_FINAL, s)) return rc;
    if ((reinterpret_cast<uintptr_t>(vx + off) & 15) == 0)
        finalize_kernel<<<(unsigned)std::min<long long>((n / 4 + 255) / 256, 8LL * p->num_sms), 256, 0, s>>>(
            acc + off, vx + off, n);
    else
        finalize_scalar_kernel<<<(unsigned)std::min<long long>((n + 255) / 256, 8LL * p->num_sms), 256, 0, s>>>(
            acc + off, vx + off, n);
    KX_LAUNCH_CHECK("finalize_kernel launch");
    return prof_end(p, s);
}

int tc_vx(kx_plan *p, int n_orb, const double *psi, const double *occ, double *vx, double *ex, bool energy_only,
          cudaStream_t s, long pair_begin, long pair_end) {
    int rc = ensure_pairs(p, n_orb, s, pair_begin, pair_end);
    if (rc) return rc;
    const std::vector<int> &first = p->h_group_first;  // n_groups + 1 entries
    const int n_groups = (int)first.size() - 1;
    const long P = first.back();
    long cap = tc_default_chunk(p, n_orb);
    for (int g = 0; g < n_groups; ++g) cap = std::max<long>(cap, first[g + 1] - first[g]);  // a group never splits
    const long chunk = std::max(1L, std::min<long>(cap, std::max(P, 1L)));
    rc = ensure_workspace(p, tc_workspace_bytes(p, n_orb, chunk));
    if (rc) return rc;
    TcLayout L = carve(p, n_orb, chunk, !energy_only);
    const long long N = (long long)p->N;

    // maxima of the orbitals and of the first chunk's items (neighbours in the workspace)
    KX_CUDA_TRY(cudaMemsetAsync(L.orb_max, 0, (size_t)((char *)(L.mx + 4 * chunk) - (char *)L.orb_max), s));
    // fp64 -> fp32 copies and maxima of orbitals [o0, o1)
    auto prep_range = [&](int o0, int o1) -> int {
        if (o1 <= o0) return KX_OK;
        dim3 g((unsigned)std::min<long long>((N + 255) / 256, 64), (unsigned)(o1 - o0));
        if (int r = prof_begin(p, PK_PREP, s)) return r;
        prep_kernel<<<g, 256, 0, s>>>(psi + (size_t)o0 * N, L.psi32 + (size_t)o0 * N, L.orb_max + o0, o1 - o0, N,
                                      o0 == 0 ? ex : nullptr);
        KX_LAUNCH_CHECK("prep_kernel launch");
        return prof_end(p, s);
    };
    // orbitals arriving in pieces: each is waited for and converted before the
    // first chunk that needs it (the multipole correction needs all of them first)
    const InputPieces &pc = p->in_pieces;
    const bool pieces = !pc.end.empty() && !energy_only && !mp_tc_eligible(p, n_orb, psi);
    int prepped = 0;  // pieces converted so far
    auto need = [&](int o_need) -> int {
        while (prepped < (int)pc.end.size() && (prepped == 0 ? 0 : pc.end[prepped - 1]) < o_need) {
            KX_CUDA_TRY(cudaStreamWaitEvent(s, pc.ready[prepped], 0));
            if (int r = prep_range(prepped == 0 ? 0 : pc.end[prepped - 1], pc.end[prepped])) return r;
            ++prepped;
        }
        return KX_OK;
    };
    if (pieces) {
        if (!pc.end.empty() && pc.end.back() < n_orb) return set_error(KX_ERR_ARG, "input pieces do not cover the orbitals");
    } else {
        for (size_t k = 0; k < pc.ready.size(); ++k) KX_CUDA_TRY(cudaStreamWaitEvent(s, pc.ready[k], 0));
        if ((rc = prep_range(0, n_orb))) return rc;
    }
    auto piece_of = [&](int o) {
        int k = 0;
        while (k + 1 < (int)pc.end.size() && pc.end[k] <= o) ++k;
        return k;
    };
    const std::vector<int> &maxorb = p->h_group_maxorb;
    // with multipole boundary values the accumulator starts from the boundary
    // correction (tensor-core form), otherwise from zero
    const bool acc_init = !energy_only && mp_tc_eligible(p, n_orb, psi);
    if (acc_init && (rc = mp_correct_into_acc(p, n_orb, psi, occ, L.acc, ex, s))) return rc;
    if (pieces && n_groups == 0 && ex) KX_CUDA_TRY(cudaMemsetAsync(ex, 0, sizeof(double), s));
    // rows [o0, o1) are final once the work queued so far has run: those no group
    // touches are filled here, the others were written by acc_kernel
    auto finish_rows = [&](int o0, int o1) -> int {
        for (int o = o0; o < o1;) {
            int e = o;
            while (e < o1 && p->h_orb_last[e] < 0) ++e;
            if (e > o) {
                if (acc_init) {
                    if (int r = finalize_rows(p, L.acc, vx, o, e, s)) return r;
                } else {
                    KX_CUDA_TRY(cudaMemsetAsync(vx + (size_t)o * N, 0, sizeof(double) * (size_t)(e - o) * N, s));
                }
            }
            o = e + 1;
        }
        if (o1 > o0 && p->final_hook.fn) p->final_hook.fn(p->final_hook.ctx, o0, o1, s);
        return KX_OK;
    };
    const int2 *pairs = reinterpret_cast<const int2 *>(p->d_pairs);
    const float mid_bound = fmax_sqrt(p);

    // pairs a chunk of a host-buffer call holds before it may end at a finished
    // row block (KX_ROW_CHUNK overrides: comparison runs)
    int row_chunk = 384;
    if (const char *e = std::getenv("KX_ROW_CHUNK")) row_chunk = std::max(1, std::atoi(e));
    // row_end[g]: groups [0, g) finish a row block (group g - 1 is the last one of
    // some orbital); tail: that row block is among the last three
    std::vector<char> row_end((size_t)n_groups + 1, 0), tail((size_t)n_groups + 1, 0);
    if (pieces)
        for (int o = 0; o < n_orb; ++o) {
            const int g = p->h_orb_last[o] + 1;
            if (g < 1 || g > n_groups) continue;
            row_end[g] = 1;
            if (o >= n_orb - 3 * kOrbBlock) tail[g] = 1;
        }
    int g0 = 0, o_fin = 0;
    while (g0 < n_groups) {
        int g1 = g0 + 1;
        while (g1 < n_groups && first[g1 + 1] - first[g0] <= chunk) {
            if (pieces) {
                // the first two pieces each end a chunk (their successors are still
                // copying); later pieces have arrived by the time they are needed.
                // A chunk ends where a row block becomes final once it holds
                // row_chunk pairs (at every one of the last three), so that
                // finished rows are copied back while the rest computes
                const int pg0 = piece_of(maxorb[g0]);
                if (pg0 < 2 && piece_of(maxorb[g1]) > pg0) break;
                if (row_end[g1] && (first[g1] - first[g0] >= row_chunk || tail[g1])) break;
            }
            ++g1;
        }
        if (pieces) {
            int o_need = 0;
            for (int g = g0; g < g1; ++g) o_need = std::max(o_need, maxorb[g] + 1);
            if ((rc = need(o_need))) return rc;
        }
        const long c0 = first[g0];
        const long R = first[g1] - c0;
        if (g0 > 0) KX_CUDA_TRY(cudaMemsetAsync(L.mx, 0, sizeof(float) * 4 * chunk, s));
        int e_count = 0;
        PassArgs a{};
        a.pairs = pairs + c0;
        a.psi32 = L.psi32;
        a.orb_max = L.orb_max;
        a.occ = occ;
        a.f32 = p->d_f32;
        a.mid_bound = mid_bound;
        if (p->precision == KX_FFT32)
            rc = fft_passes(p, R, pairs + c0, L.psi32, 0, occ, reinterpret_cast<float2 *>(L.T1), L.T0, nullptr, ex,
                            L.partial, energy_only, s);
        else
            rc = run_passes(p, a, R, L.T0, L.T1, L.mx, chunk, ex, L.partial, energy_only, nullptr, s, &e_count);
        if (rc) return rc;
        if (!energy_only) {
            AccArgs ac{};
            ac.phi = L.T0;
            ac.groups = reinterpret_cast<const Group *>(p->d_groups);
            ac.g0 = g0;
            ac.g1 = g1;
            ac.item0 = (int)c0;
            ac.n_orb = n_orb;
            ac.item_slot = reinterpret_cast<const int2 *>(p->d_item_slot);
            ac.orb_span = reinterpret_cast<const int2 *>(p->d_orb_span);
            ac.psi32 = L.psi32;
            ac.occ = occ;
            ac.acc = L.acc;
            ac.vx = vx;
            ac.vx_vec = (reinterpret_cast<uintptr_t>(vx) & 15) == 0;
            ac.acc_init = acc_init ? 1 : 0;
            ac.N = N;
            ac.e_partial = L.partial;
            ac.e_count = ex ? e_count : 0;
            ac.e_factor = -0.5 * p->dV;
            ac.ex = ex;
            if ((rc = prof_begin(p, PK_ACC, s))) return rc;
            if (N % 4 == 0) {  // rows of whole 16-byte pieces
                if ((rc = raise_smem(p, reinterpret_cast<const void *>(acc_kernel<4>), acc_smem<4>()))) return rc;
                acc_kernel<4><<<(unsigned)((N / 4 + kAccThreads - 1) / kAccThreads), kAccThreads, acc_smem<4>(), s>>>(ac);
            } else {
                acc_kernel<1><<<(unsigned)((N + kAccThreads - 1) / kAccThreads), kAccThreads, acc_smem<1>(), s>>>(ac);
            }
            KX_LAUNCH_CHECK("acc_kernel launch");
            if ((rc = prof_end(p, s))) return rc;
        }
        if (!energy_only) {
            // rows whose last group is done are final
            int o_done = o_fin;
            while (o_done < n_orb && p->h_orb_last[o_done] < g1) ++o_done;
            if ((rc = finish_rows(o_fin, o_done))) return rc;
            o_fin = o_done;
        }
        g0 = g1;
    }
    if (pieces && (rc = need(n_orb))) return rc;  // every piece is on the device when the call's work ends
    if (!energy_only) return finish_rows(o_fin, n_orb);
    return KX_OK;
}

int selftest_wait(kx_plan *p, long long max_cycles, cudaStream_t s) {
    selftest_wait_kernel<<<1, 32, 0, s>>>(max_cycles, p->d_status);
    KX_LAUNCH_CHECK("selftest_wait_kernel launch");
    return KX_OK;
}

int tc_apply_fL(kx_plan *p, int n_rhs, const double *b, double *x, cudaStream_t s) {
    const long chunk = std::min<long>(tc_default_chunk(p, 1), n_rhs);
    int rc = ensure_workspace(p, tc_workspace_bytes(p, (int)chunk, chunk));
    if (rc) return rc;
    TcLayout L = carve(p, (int)chunk, chunk, false);
    const long long N = (long long)p->N;
    const float mid_bound = fmax_sqrt(p);
    for (long c0 = 0; c0 < n_rhs; c0 += chunk) {
        const long R = std::min<long>(chunk, n_rhs - c0);
        KX_CUDA_TRY(cudaMemsetAsync(L.orb_max, 0, sizeof(float) * R, s));
        KX_CUDA_TRY(cudaMemsetAsync(L.mx, 0, sizeof(float) * 4 * chunk, s));
        dim3 g((unsigned)std::min<long long>((N + 255) / 256, 64), (unsigned)R);
        if ((rc = prof_begin(p, PK_PREP, s))) return rc;
        prep_kernel<<<g, 256, 0, s>>>(b + c0 * N, L.psi32, L.orb_max, (int)R, N, nullptr);
        KX_LAUNCH_CHECK("prep_kernel launch");
        if ((rc = prof_end(p, s))) return rc;
        PassArgs a{};
        a.rhs_mode = 1;
        a.f32 = p->d_f32;
        a.mid_bound = mid_bound;
        a.src_max = L.orb_max;
        a.in = L.psi32;
        if (p->precision == KX_FFT32)
            rc = fft_passes(p, R, nullptr, L.psi32, 1, nullptr, reinterpret_cast<float2 *>(L.T1), nullptr, x + c0 * N,
                            nullptr, nullptr, false, s);
        else
            rc = run_passes(p, a, R, L.T0, L.T1, L.mx, chunk, nullptr, nullptr, false, x + c0 * N, s);
        if (rc) return rc;
    }
    return KX_OK;
}

// ---------------------------------------------------------------------------
// f(L) B without device allocation (kx_apply_fL_noalloc).
//
// Callers that cannot allocate device memory at the point of the call (their
// device memory was reserved up front by a pool allocator, or they run inside
// a solver loop that must not pay the device-wide synchronisation of
// cudaMalloc / cudaFree) get this variant: its scratch is the file-scope
// array below, so the call itself allocates nothing.  The array is part of
// this module's image: every GPU that loads it holds kNoAllocBytes until the
// process exits.  All calls share it and it keeps the previous call's
// contents; the per-vector maxima that must start at zero are cleared at every
// call.  Calls whose GPU work overlaps (two streams, or two host threads on one
// device) race on the array.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t kNoAllocMaxElems = (size_t)5 << 19;  // n_rhs * N limit per call (2,621,440 grid values)
constexpr size_t kNoAllocMaxVec = 8192;               // >= kNoAllocMaxElems / 512 (smallest N with n % 8 == 0)
constexpr size_t kNoAllocBytes = 3 * kNoAllocMaxElems * sizeof(float) + 5 * kNoAllocMaxVec * sizeof(float);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// The host-side name of the array is only a stand-in, so the kernels get the
// address the runtime reports for the current device.  It is looked up on
// every call (the lookup allocates nothing): a cached address would outlive a
// cudaDeviceReset, after which the module and its array are loaded anew.  On
// the first call on a device the lookup may load this module's device code,
// and the array with it, like any first launch from the module.
int noalloc_scratch(void **out) {
    void *ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_error(e, "kx_apply_fL_noalloc: cudaGetSymbolAddress of the static scratch");
    *out = ptr;
    return KX_OK;
}

}  // namespace

size_t noalloc_max_elems() { return kNoAllocMaxElems; }

#ifdef KX_ROLE_CLOCKS
}  // namespace kx
// managed buffer written by the last launch of each pass (experiment builds only)
extern "C" long long *kx_debug_role_clocks() { return kx::g_clkbuf; }
namespace kx {
#endif

int tc_apply_fL_noalloc(kx_plan *p, int n_rhs, const double *b, double *x, cudaStream_t s) {
    if (p->precision != KX_F16X3)
        return set_error(KX_ERR_UNSUPPORTED, "kx_apply_fL_noalloc: needs a KX_F16X3 plan");
    const long long N = (long long)p->N;
    if ((size_t)n_rhs * (size_t)N > kNoAllocMaxElems)
        return set_error(KX_ERR_ARG, "kx_apply_fL_noalloc: n_rhs * N = " + std::to_string((size_t)n_rhs * N) +
                                         " exceeds the static scratch limit of " +
                                         std::to_string(kNoAllocMaxElems) + " grid values; split the call");
    int dev = -1;
    KX_CUDA_TRY(cudaGetDevice(&dev));
    if (dev != p->device) return set_error(KX_ERR_ARG, "kx_apply_fL_noalloc: call on the plan's device");
    void *base = nullptr;
    if (int rc = noalloc_scratch(&base)) return rc;
    const size_t elems = (size_t)n_rhs * (size_t)N;
    float *b32 = reinterpret_cast<float *>(base);
    float *T0 = b32 + elems;
    float *T1 = T0 + elems;
    float *src_max = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(base) +
                                               3 * kNoAllocMaxElems * sizeof(float));
    float *mx = src_max + kNoAllocMaxVec;  // four per-item maxima rows of kNoAllocMaxVec
    KX_CUDA_TRY(cudaMemsetAsync(src_max, 0, 5 * kNoAllocMaxVec * sizeof(float), s));
    dim3 g((unsigned)std::min<long long>((N + 255) / 256, 64), (unsigned)n_rhs);
    prep_kernel<<<g, 256, 0, s>>>(b, b32, src_max, n_rhs, N, nullptr);
    KX_LAUNCH_CHECK("prep_kernel launch");
    PassArgs a{};
    a.rhs_mode = 1;
    a.f32 = p->d_f32;
    a.mid_bound = fmax_sqrt(p);
    a.src_max = src_max;
    a.in = b32;
    return run_passes(p, a, n_rhs, T0, T1, mx, (long)kNoAllocMaxVec, nullptr, nullptr, false, x, s);
}

}  // namespace kx
