// Complex mode products of the k-point exchange, two per kernel (split-fp16 plans whose
// planes are 64 x 64 points and whose third axis has 32 or 64): three kernels per chunk
// in place of the six single products of kx_bloch.cu, in the same order,
//   F_FWD12  pair densities, axis 1 forward, axis 2 forward  (planes at fixed x3)
//   F_MID3   axis 3 forward, times f(Lambda), axis 3 inverse (pencils along axis 3)
//   F_INV21  axis 2 inverse, axis 1 inverse                  (planes at fixed x3)
// The value between the two products is rounded to float32 as the single product stores
// it and split again with the same power of two, so the results are bit-identical.  That
// power comes from the maximum over the whole pair density or potential (a split of a
// value far below it keeps fewer bits, and f(Lambda) spans many octaves: with the scale
// of a row or a tile instead the results differ by 1.6e-8), so in F_MID3 and F_INV21 the
// CTAs that share an item wait for its maximum between the two products: a cooperative
// launch, bounded waits, and the store of the tile before in the meantime.  Where the CTAs
// cannot all be resident (bloch_fused_fits) the single products run.
//
// What bounds it: six single products move 11 times a chunk's values (537 MB at 64^3 and
// 256 pairs), these move 5.  Per chunk, forward 523 -> 238 us, middle 459 -> 310 us,
// inverse 446 -> 324 us (floors at the copy rate 79, 158 and 158 us): neither memory
// nor the tensor cores (38 %) but the SM's load / store path, half of whose cycles go to
// the TMEM reads (256 KB per tile), the split operands' stores (128 KB) and the tile's
// own loads and stores, and, where CTAs wait for each other, the slowest of an item's 32
// tiles (2,500 and 5,000 of 11,000 cycles per tile; with a maximum and a counter per item
// updated by atomics instead of a word per tile 360 and 419 us).
#include "kx_internal.h"
#include "kx_conv.cuh"
#include "kx_tc_ptx.cuh"

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace kx {
namespace {

// A tile is 128 rows of the product: a pair of 64 x 64 planes (rows (plane, x2) or
// (plane, x1)) or 128 neighbouring pencils along axis 3.  Each product is the real
// GEMM [A_r | A_i] (128 x 2n) times [[M_r, M_i], [-M_i, M_r]] in three fp16 products
// (hi lo and lo hi into Da, hi hi into Db), as in kx_bloch.cu.
//
// Warps: 16 epilogue warps (TMEM lane quadrant w % 4, a quarter of the columns each), 8
// producer warps, one MMA warp.  A slot is one A buffer and 256 TMEM columns; a tile
// runs through it as
//   producers fill A -> product 1 -> the epilogue splits D into A, in place -> product 2
//   -> the epilogue stores D,
// with two slots, so that the tensor core has one tile while the epilogue has the
// other.  All epilogue warps share a tile (8 per slot: the same time per tile, but
// slots that waited for their own chain of latencies: 253 and 269 us).
//
// Shared memory (224 KB at n = 64) holds both operands and both A buffers only because
//   - an operand is stored as the strip [-M_i | M_r | M_i] of n rows: the K rows of A_r
//     multiply its columns [n, 3n) and those of A_i its columns [0, 2n);
//   - A is stored in the 128-byte swizzle, whose 8 x 128-byte atoms need no padding: a
//     warp's 32 lanes (two neighbouring values each) write one 128-byte row of an atom,
//     and a thread of the epilogue 16 bytes at its own row, both without bank conflicts.
// A with K values along the rows (kk in [0, 2n), 64 per atom column):
//   (m, kk): (kk / 64) 16384 + m 128 + (((kk / 8) % 8) ^ (m % 8)) 16 + (kk % 8) 2 bytes,
// A with the tile's rows along the rows (64 per half h):
//   (m, kk): h 256 n + kk 128 + (((m % 64) / 8) ^ (kk % 8)) 16 + (m % 8) 2 bytes.
enum { F_FWD12, F_MID3, F_INV21 };

constexpr int kFuEpiWarps = 16, kFuProdWarps = 8;
constexpr int kFuMmaWarp = kFuEpiWarps + kFuProdWarps;
constexpr int kFuThreads = 32 * (kFuMmaWarp + 1);
constexpr int kFuPlane = 64 * 64;           // values of a plane
constexpr uint32_t kFuAtomCol = 128 * 128;  // bytes of 128 rows of one 64-value atom column

__host__ __device__ constexpr int fu_strip_bytes(int n) { return 6 * n * n; }  // hi or lo of one operand
__host__ __device__ constexpr int fu_a_bytes(int n) { return 512 * n; }        // hi or lo of one A buffer
__host__ __device__ constexpr int fu_smem_bytes(int n) { return 1024 + 4 * fu_a_bytes(n) + 4 * fu_strip_bytes(n); }

struct FuArgs {
    const float2 *in;         // F_MID3, F_INV21
    const float2 *P, *F;      // F_FWD12: orbitals, vectors
    float2 *out;
    const __half *B1, *B2;    // split operands of the two products (bloch_tc_bsplit_kernel)
    const float *f;           // F_MID3
    const float *in_max;      // per item (F_MID3, F_INV21)
    int *mid;                 // F_MID3, F_INV21: per item and tile (32), the maximum between the products; zeroed
    const float *pmax, *fmax; // F_FWD12: bounds from the vectors' maxima
    float bound1, bound2;     // F_FWD12: factors of max|psi_m| max|phi_v| for the two products
    long long r0, N;
    int n_orb;
    float *out_max;           // per item, zeroed (F_FWD12, F_MID3)
    int n_tiles, tiles_per_item;
    int *status;
    long long timeout_cycles;
};

// split exponent of a maximum, capped at 100 as in the single products
__device__ __forceinline__ int fu_exp(float mx) { return min(scale_exp(mx), 100); }

// max|psi_m| max|phi_v| of item r0 + item = v n_orb + m
__device__ __forceinline__ void fu_pair(const FuArgs &a, int item, int &v, int &m) {
    const int r = (int)a.r0 + item;  // pair indices stay below 2^24 (checked at entry)
    v = r / a.n_orb;
    m = r - v * a.n_orb;
}

// Products of one tile: Da = A_hi B_lo + A_lo B_hi (the lo hi term first when LO_FIRST),
// Db = A_hi B_hi.  a_hi, a_lo: A buffers; b_hi, b_lo: operand strips.
template <int NK, bool K_MAJOR, bool LO_FIRST>
__device__ __forceinline__ void fu_issue(uint32_t da, uint32_t a_hi, uint32_t a_lo, uint32_t b_hi, uint32_t b_lo) {
    constexpr uint32_t idesc = ptx::idesc_f16(128, 2 * NK, K_MAJOR ? 0 : 1, 1);
    constexpr uint32_t gb = 48u * NK;  // strip: bytes between 8-row groups
    const uint64_t a0 = K_MAJOR ? ptx::sdesc_sw128(a_hi, 16, 1024) : ptx::sdesc_sw128(a_hi, 256u * NK, 1024);
    const uint64_t b0 = ptx::sdesc(b_hi, gb, 128);
    const uint32_t ah0 = (uint32_t)a0, ahi32 = (uint32_t)(a0 >> 32), bh0 = (uint32_t)b0, bhi32 = (uint32_t)(b0 >> 32);
    const uint32_t al0 = ah0 + ((a_lo - a_hi) >> 4), bl0 = bh0 + ((b_lo - b_hi) >> 4);
    const uint32_t db = da + 2 * NK;
#pragma unroll
    for (int ks = 0; ks < NK / 8; ++ks) {
        const uint32_t ao = (K_MAJOR ? (ks >> 2) * kFuAtomCol + (ks & 3) * 32u : ks * 2048u) >> 4;
        const uint32_t bo = (16 * ks < NK ? 16u * NK + 2u * gb * ks : 2u * gb * (ks - NK / 16)) >> 4;
        const uint32_t first = ks > 0 ? 1u : 0u;
        if (LO_FIRST) {
            ptx::mma_f16_lo(da, al0 + ao, ahi32, bh0 + bo, bhi32, idesc, first);
            ptx::mma_f16_lo(da, ah0 + ao, ahi32, bl0 + bo, bhi32, idesc, 1u);
        } else {
            ptx::mma_f16_lo(da, ah0 + ao, ahi32, bl0 + bo, bhi32, idesc, first);
            ptx::mma_f16_lo(da, al0 + ao, ahi32, bh0 + bo, bhi32, idesc, 1u);
        }
        ptx::mma_f16_lo(db, ah0 + ao, ahi32, bh0 + bo, bhi32, idesc, first);
    }
}

// fp16 hi and lo of two values, 4 bytes each
__device__ __forceinline__ void fu_store2(uint8_t *hi, uint8_t *lo, float x, float y) {
    const __half2 h = __floats2half2_rn(x, y);
    const float2 hf = __half22float2(h);
    *reinterpret_cast<__half2 *>(hi) = h;
    *reinterpret_cast<__half2 *>(lo) = __floats2half2_rn(x - hf.x, y - hf.y);
}
__device__ __forceinline__ void fu_store8(uint8_t *hi, uint8_t *lo, uint32_t off, const float2 *w) {
    uint4 h, l;
    split8(w, h, l);
    *reinterpret_cast<uint4 *>(hi + off) = h;
    *reinterpret_cast<uint4 *>(lo + off) = l;
}

__device__ __forceinline__ void fu_arrive(uint64_t *bar) {  // one arrival per warp
    __syncwarp();
    if ((threadIdx.x & 31) == 0) ptx::mbar_arrive(bar);
}

// KIND as above; NK: contraction length of both products (the axis' points).
template <int KIND, int NK>
__global__ void __launch_bounds__(kFuThreads, 1) bloch_fused_kernel(const FuArgs a) {
    extern __shared__ uint8_t fu_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(fu_raw) + 1023) & ~uintptr_t(1023));
    constexpr uint32_t ab = fu_a_bytes(NK), sb = fu_strip_bytes(NK);
    uint8_t *const strips = smem + 4 * ab;  // B1 hi, B1 lo, B2 hi, B2 lo
    __shared__ uint64_t full[2], aempty[2], tfull[2], a2full[2], tempty[2], drain;
    __shared__ uint32_t tslot;
    __shared__ volatile int s_abort;
    __shared__ int s_max[2], s_cnt[2];  // of a tile, by its parity
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == kFuMmaWarp) {
        ptx::tmem_alloc(&tslot, 512);
        ptx::tmem_relinquish();
    }
    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(&full[s], kFuProdWarps);
            ptx::mbar_init(&aempty[s], 1);
            ptx::mbar_init(&tfull[s], 1);
            ptx::mbar_init(&a2full[s], kFuEpiWarps);
            ptx::mbar_init(&tempty[s], kFuEpiWarps);
        }
        ptx::mbar_init(&drain, 1);
        ptx::fence_mbar_init();
        s_abort = 0;
        s_max[0] = s_max[1] = s_cnt[0] = s_cnt[1] = 0;
    }
    {  // operand strips: row kk of [-M_i | M_r | M_i], from the stored [[M_r, M_i], [-M_i, M_r]]
        constexpr int chunks = 3 * NK * NK / 8;  // of 16 bytes, per strip
        for (int e = tid; e < 4 * chunks; e += kFuThreads) {
            const int b = e / chunks, r = e - b * chunks;  // b: B1 hi, B1 lo, B2 hi, B2 lo
            const int kk = r / (3 * NK / 8), j8 = r - kk * (3 * NK / 8);
            const int sk = j8 < NK / 8 ? kk + NK : kk, c8 = j8 < NK / 8 ? j8 : j8 - NK / 8;
            const uint4 *src = reinterpret_cast<const uint4 *>(b < 2 ? a.B1 : a.B2) + (b & 1) * (4 * NK * NK / 8);
            reinterpret_cast<uint4 *>(strips + b * sb)[j8 * 8 + (kk >> 3) * (3 * NK) + (kk & 7)] =
                __ldg(src + c8 * 8 + (sk >> 3) * (2 * NK) + (sk & 7));
        }
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = tslot;
    const int n_my = (a.n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    auto tile_of = [&](int it) { return (int)blockIdx.x + it * (int)gridDim.x; };
    // first value of a tile (in its chunk buffer)
    auto tile_base = [&](int t) {
        if (KIND != F_MID3) return (long long)t * (2 * kFuPlane);
        return (long long)(t >> 5) * a.N + (t & 31) * 128;
    };
    auto wait = [&](uint64_t *bar, uint32_t parity) {
        const long long t0 = clock64();
        while (!ptx::mbar_try_wait(bar, parity)) {
            if (s_abort) return false;
            if (clock64() - t0 > a.timeout_cycles) {
                s_abort = 1;
                atomicExch(a.status, KX_ERR_TIMEOUT);
                return false;
            }
        }
        return true;
    };

    if (warp == kFuMmaWarp) {
        // ---------------------------------------------------------------- MMA issue
        // whichever product is ready: the second one of the older tile, else the first
        // one of the next tile
        const uint32_t sA = ptx::smem_u32(smem), sB = ptx::smem_u32(strips);
        int n1 = 0, n2 = 0;
        long long t0 = clock64();
        bool ok = true;
        while (n2 < n_my) {
            bool did = false;
            if (n2 < n1) {
                const int s = n2 & 1;
                if (__any_sync(0xffffffffu, ptx::mbar_test_wait(&a2full[s], (uint32_t)((n2 >> 1) & 1)))) {
                    ptx::tc_fence_after();
                    if (ptx::elect_one()) {
                        fu_issue<NK, KIND == F_MID3, KIND == F_INV21>(tmem + 256u * s, sA + 2 * s * ab,
                                                                      sA + (2 * s + 1) * ab, sB + 2 * sb, sB + 3 * sb);
                        ptx::mma_commit(&tfull[s]);
                        ptx::mma_commit(&aempty[s]);
                    }
                    __syncwarp();
                    ++n2;
                    did = true;
                }
            }
            if (!did && n1 < n_my && n1 < n2 + 2) {
                const int s = n1 & 1;
                const bool rdy = ptx::mbar_test_wait(&full[s], (uint32_t)((n1 >> 1) & 1)) &&
                                 (n1 < 2 || ptx::mbar_test_wait(&tempty[s], (uint32_t)(((n1 >> 1) - 1) & 1)));
                if (__any_sync(0xffffffffu, rdy)) {
                    ptx::tc_fence_after();
                    if (ptx::elect_one()) {
                        fu_issue<NK, KIND == F_FWD12, KIND == F_FWD12>(tmem + 256u * s, sA + 2 * s * ab,
                                                                       sA + (2 * s + 1) * ab, sB, sB + sb);
                        ptx::mma_commit(&tfull[s]);
                    }
                    __syncwarp();
                    ++n1;
                    did = true;
                }
            }
            if (did) {
                t0 = clock64();
            } else if (__any_sync(0xffffffffu, s_abort || clock64() - t0 > a.timeout_cycles)) {
                ok = false;
                break;
            }
        }
        if (!ok) {
            // gave up: the products already issued finish before TMEM is released
            if (lane == 0 && !s_abort) {
                s_abort = 1;
                atomicExch(a.status, KX_ERR_TIMEOUT);
            }
            __syncwarp();
            if (ptx::elect_one()) {
                ptx::mma_commit(&drain);
                ptx::mbar_wait_bounded(&drain, 0, a.timeout_cycles);
            }
            __syncwarp();
        }
    } else if (warp >= kFuEpiWarps) {
        // ---------------------------------------------------------------- producers
        // Task i of a thread is 16 bytes: the values 2 lane, 2 lane + 1 of a run of 64 (a
        // pencil along axis 1, or 64 rows of the tile at one kk); pw: the thread's warp.
        const int pw = warp - kFuEpiWarps;
        constexpr int kTasks = NK / 4;  // 8 warps x kTasks runs of 64 values per tile
        // byte offset of task 0 in an A buffer; tasks advance by whole atoms, pw is the row in one
        uint8_t *const A0 = smem + pw * 128 + (((lane >> 2) ^ pw) << 4) + (lane & 3) * 4;
        auto a_off = [](int i) {
            return KIND == F_FWD12 ? (uint32_t)i * 1024u
                                   : (uint32_t)(i % (NK / 8)) * 1024u + (uint32_t)(i / (NK / 8)) * (256u * NK);
        };
        constexpr uint32_t im_off = KIND == F_FWD12 ? kFuAtomCol : 128u * NK;
        auto put = [&](uint8_t *hi, int i, float2 x, float2 y, float sc) {
            x = mul2(x, make_float2(sc, sc));
            y = mul2(y, make_float2(sc, sc));
            uint8_t *h = hi + a_off(i);
            fu_store2(h, h + ab, x.x, y.x);
            fu_store2(h + im_off, h + im_off + ab, x.y, y.y);
        };
        auto wait_empty = [&](int it) {
            return __all_sync(0xffffffffu, it < 2 || wait(&aempty[it & 1], (uint32_t)(((it >> 1) - 1) & 1)));
        };
        if constexpr (KIND == F_FWD12) {
            constexpr int D = 4;  // tasks per batch: all loads of a batch, then all its values
            float4 x[D], y[D];
            const float4 *xp, *yp;
            float bound;
            auto aim = [&](int it) {
                const int t = tile_of(it), item = t / a.tiles_per_item;
                int v, m;
                fu_pair(a, item, v, m);
                const long long o = (long long)(t - item * a.tiles_per_item) * (2 * kFuPlane) + 64 * pw + 2 * lane;
                xp = reinterpret_cast<const float4 *>(a.P + m * a.N + o);
                yp = reinterpret_cast<const float4 *>(a.F + v * a.N + o);
                bound = a.bound1 * a.pmax[m] * a.fmax[v];
            };
            auto load = [&](int i0) {  // runs pw + 8 i: 512 values apart
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    x[d] = __ldg(xp + 256 * (i0 + d));
                    y[d] = __ldg(yp + 256 * (i0 + d));
                }
            };
            if (n_my > 0) {
                aim(0);
                load(0);
            }
            for (int it = 0; it < n_my; ++it) {
                const float sc = pow2f(fu_exp(bound));
                if (!wait_empty(it)) break;
                uint8_t *hi = A0 + 2 * (it & 1) * ab;
#pragma unroll
                for (int i0 = 0; i0 < kTasks; i0 += D) {
#pragma unroll
                    for (int d = 0; d < D; ++d) {  // conj(psi_m) phi_v
                        const float4 p = x[d], f = y[d];
                        put(hi, i0 + d, make_float2(p.x * f.x + p.y * f.y, p.x * f.y - p.y * f.x),
                            make_float2(p.z * f.z + p.w * f.w, p.z * f.w - p.w * f.z), sc);
                    }
                    if (i0 + D < kTasks) load(i0 + D);
                }
                ptx::fence_proxy_async_smem();
                fu_arrive(&full[it & 1]);
                if (it + 1 < n_my) {
                    aim(it + 1);
                    load(0);
                    if ((lane & 7) == 0) {  // the rest of the tile into L2, a 128-byte line per 8 lanes
#pragma unroll
                        for (int i = D; i < kTasks; ++i) {
                            ptx::prefetch_l2(xp + 256 * i);
                            ptx::prefetch_l2(yp + 256 * i);
                        }
                    }
                }
            }
        } else {
            // runs (kk, h) = (pw + 8 (i mod n / 8), i / (n / 8)): F_MID3 pencils 64 h.. of the tile at
            // x3 = kk, F_INV21 plane h at k2 = kk.  Batches of D: all loads, then all values (loads
            // issued between would make the values of older ones wait for them).
            constexpr int ks = KIND == F_MID3 ? kFuPlane : 64, hs = KIND == F_MID3 ? 64 : kFuPlane;
            constexpr int D = 8;
            float4 v[D];
            const float4 *src;
            float mx = 0.f;
            auto aim = [&](int it) {
                const int t = tile_of(it);
                src = reinterpret_cast<const float4 *>(a.in + tile_base(t) + pw * ks + 2 * lane);
                mx = a.in_max[t / a.tiles_per_item];
            };
            auto off = [](int i) { return (i % (NK / 8)) * (8 * ks / 2) + (i / (NK / 8)) * (hs / 2); };
            auto load = [&](int i0) {
#pragma unroll
                for (int d = 0; d < D; ++d) v[d] = __ldg(src + off(i0 + d));
            };
            if (n_my > 0) {
                aim(0);
                load(0);
            }
            for (int it = 0; it < n_my; ++it) {
                const float sc = pow2f(fu_exp(mx));
                if (it + 1 < n_my && (lane & 7) == 0) {  // the next tile into L2, a 128-byte line per 8 lanes
                    const float4 *nx =
                        reinterpret_cast<const float4 *>(a.in + tile_base(tile_of(it + 1)) + pw * ks + 2 * lane);
#pragma unroll
                    for (int i = 0; i < kTasks; ++i) ptx::prefetch_l2(nx + off(i));
                }
                if (!wait_empty(it)) break;
                uint8_t *hi = A0 + 2 * (it & 1) * ab;
#pragma unroll
                for (int i0 = 0; i0 < kTasks; i0 += D) {
                    if (i0 > 0) load(i0);
#pragma unroll
                    for (int d = 0; d < D; ++d)
                        put(hi, i0 + d, make_float2(v[d].x, v[d].y), make_float2(v[d].z, v[d].w), sc);
                }
                ptx::fence_proxy_async_smem();
                fu_arrive(&full[it & 1]);
                if (it + 1 < n_my) {
                    aim(it + 1);
                    load(0);
                }
            }
        }
    } else {
        // ---------------------------------------------------------------- epilogue
        // product 1 of tile it, then product 2 of tile it - 1: the tensor core has the other one
        const int qd = warp & 3, cq = warp >> 2;  // lane quadrant, quarter of the columns
        constexpr int G = NK / 32;                // groups of 8 columns per quarter
        const int r = 32 * qd + lane;             // row of the tile
        const uint32_t tl = tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(8 * G * cq);
        // this thread's place in the second A: with K along the rows (F_MID3) its own row, 16
        // bytes per 8 columns; else the row kk = r % 64 of half r / 64, 16 bytes per 8 rows
        const int rr = r & 63;
        uint8_t *const a2 = smem + (KIND == F_MID3 ? r * 128 : (r >> 6) * (256 * NK) + rr * 128);
        auto a2_off = [&](int g, int im) {  // columns 8 (G cq + g).., real or imaginary part
            const int c8 = G * cq + g;
            if (KIND == F_MID3) {
                const int k8 = c8 + im * (NK / 8);
                return (uint32_t)(k8 >> 3) * kFuAtomCol + (uint32_t)(((k8 & 7) ^ (r & 7)) << 4);
            }
            return (uint32_t)im * (128u * NK) + (uint32_t)((c8 ^ (rr & 7)) << 4);
        };
        auto sum2 = [](const float *x, const float *y, int k, float u) {  // (Da + Db) u, two columns
            return mul2(add2(pair(x, k), pair(y, k)), make_float2(u, u));
        };
        // maxima of a tile's item, loaded a tile ahead
        float mx0 = 0.f, mx1 = 0.f;
        auto maxima = [&](int it) {
            const int item = tile_of(it) / a.tiles_per_item;
            if constexpr (KIND == F_FWD12) {
                int v, m;
                fu_pair(a, item, v, m);
                mx0 = a.pmax[m];
                mx1 = a.fmax[v];
            } else {
                mx0 = a.in_max[item];
            }
        };
        if (n_my > 0) maxima(0);
        int e_new = 0, e_old = 0;  // split exponents of the second A of this tile and the one before
        // D of the first product: into the second A (F_FWD12), or back to TMEM as the values
        // between the products, with the item's maximum on its way
        auto first = [&](int it) {
            const int s = it & 1, t = tile_of(it);
            const int e_in = fu_exp(KIND == F_FWD12 ? a.bound1 * mx0 * mx1 : mx0);
            const int em = fu_exp(KIND == F_FWD12 ? a.bound2 * mx0 * mx1 : 0.f);
            if (it + 1 < n_my) maxima(it + 1);
            float fv[KIND == F_MID3 ? 8 * G : 1];
            if constexpr (KIND == F_MID3) {
                const float *fp = a.f + (t & 31) * 128 + r + 8 * G * cq * kFuPlane;
#pragma unroll
                for (int c = 0; c < 8 * G; ++c) fv[c] = __ldg(fp + c * kFuPlane);
            }
            if (!__all_sync(0xffffffffu, wait(&tfull[s], 0u))) return false;
            ptx::tc_fence_after();
            const uint32_t ta = tl + 256u * (uint32_t)s;
            uint8_t *const Ahi = a2 + 2 * s * ab;
            // F_FWD12: unscaled and scaled for the second product at once (powers of two: exact)
            const float us = pow2f(KIND == F_FWD12 ? em - e_in - kVScaleExp : -e_in - kVScaleExp);
            float mx = 0.f;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                float ra[8], rb[8], ia[8], ib[8];
                const uint32_t c = ta + 8u * g;
                ptx::tmem_ld8x4(c, c + 2 * NK, c + NK, c + 3 * NK, ra, rb, ia, ib);
                float2 w[4], u[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    w[k] = sum2(ra, rb, k, us);
                    u[k] = sum2(ia, ib, k, us);
                    if constexpr (KIND == F_MID3) {
                        w[k] = mul2(w[k], pair(fv + 8 * g, k));
                        u[k] = mul2(u[k], pair(fv + 8 * g, k));
                    }
                    if constexpr (KIND != F_FWD12)
                        mx = fmaxf(mx, fmaxf(fmaxf(fabsf(w[k].x), fabsf(w[k].y)), fmaxf(fabsf(u[k].x), fabsf(u[k].y))));
                }
                if constexpr (KIND == F_FWD12) {
                    fu_store8(Ahi, Ahi + ab, a2_off(g, 0), w);
                    fu_store8(Ahi, Ahi + ab, a2_off(g, 1), u);
                } else {
                    ptx::tmem_st8x2(c, c + NK, &w[0].x, &u[0].x);
                }
            }
            if constexpr (KIND == F_FWD12) {
                e_new = em;
                ptx::fence_proxy_async_smem();
                ptx::tc_fence_before();
                fu_arrive(&a2full[s]);
            } else {
                ptx::tmem_wait_st();
                for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                if (lane == 0) {
                    // the tile's last warp passes its maximum on, the sign bit marking it as there
                    atomicMax(&s_max[s], __float_as_int(mx));
                    __threadfence_block();
                    if (atomicAdd(&s_cnt[s], 1) == kFuEpiWarps - 1) {
                        __threadfence_block();
                        const int m = atomicExch(&s_max[s], 0);
                        atomicExch(&s_cnt[s], 0);
                        const int item = t / a.tiles_per_item;
                        ptx::st_relaxed(a.mid + 32 * item + t - item * a.tiles_per_item, m | (int)0x80000000);
                    }
                }
                __syncwarp();
            }
            return true;
        };
        // F_MID3, F_INV21: the values between the products into the second A, with the
        // scale of their item's maximum once all its tiles (of this and other CTAs) are in.
        // Tiles go to the CTAs in order and no CTA has two of an item (bloch_fused_fits), so a
        // wait is for another CTA's tile whose first product depends on earlier items only.
        auto between = [&](int it) {
            const int s = it & 1, t = tile_of(it);
            // a tile's word is its maximum and the mark that it is there: a lane per tile
            const int *mid = a.mid + 32 * (t / a.tiles_per_item) + lane;
            int m = 0;
            const long long t0 = clock64();
            for (;;) {
                if (lane < a.tiles_per_item) m = ptx::ld_relaxed(mid);
                if (__all_sync(0xffffffffu, m < 0 || lane >= a.tiles_per_item)) break;
                const bool late = clock64() - t0 > a.timeout_cycles;
                if (__any_sync(0xffffffffu, late || s_abort)) {
                    if (late && lane == 0) {
                        s_abort = 1;
                        atomicExch(a.status, KX_ERR_TIMEOUT);
                    }
                    return false;
                }
            }
            m = __reduce_max_sync(0xffffffffu, m & 0x7fffffff);  // not negative: ordered as the floats are
            const int em = fu_exp(__int_as_float(m));
            const float sc = pow2f(em);
            const uint32_t ta = tl + 256u * (uint32_t)s;
            uint8_t *const Ahi = a2 + 2 * s * ab;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                float re[8], im[8];
                ptx::tmem_ld8x2(ta + 8u * g, ta + 8u * g + NK, re, im);
                float2 w[4], u[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    w[k] = mul2(pair(re, k), make_float2(sc, sc));
                    u[k] = mul2(pair(im, k), make_float2(sc, sc));
                }
                fu_store8(Ahi, Ahi + ab, a2_off(g, 0), w);
                fu_store8(Ahi, Ahi + ab, a2_off(g, 1), u);
            }
            e_new = em;
            ptx::fence_proxy_async_smem();
            ptx::tc_fence_before();
            fu_arrive(&a2full[s]);
            return true;
        };
        // D of the second product to memory
        auto second = [&](int it) {
            const int s = it & 1, t = tile_of(it);
            if (!__all_sync(0xffffffffu, wait(&tfull[s], 1u))) return false;
            ptx::tc_fence_after();
            const uint32_t ta = tl + 256u * (uint32_t)s;
            const float us = pow2f(-e_old - kVScaleExp);
            float mx = 0.f;
            constexpr int cs = KIND == F_MID3 ? kFuPlane : KIND == F_FWD12 ? 64 : 1;  // column stride
            float2 *dst = a.out + tile_base(t) + 8 * G * cq * cs +
                          (KIND == F_MID3 ? r : KIND == F_FWD12 ? (r >> 6) * kFuPlane + rr : 64 * r);
            float2 w[G][4], u[G][4];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                float ra[8], rb[8], ia[8], ib[8];
                const uint32_t c = ta + 8u * g;
                ptx::tmem_ld8x4(c, c + 2 * NK, c + NK, c + 3 * NK, ra, rb, ia, ib);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    w[g][k] = sum2(ra, rb, k, us);
                    u[g][k] = sum2(ia, ib, k, us);
                }
            }
            ptx::tc_fence_before();
            fu_arrive(&tempty[s]);
#pragma unroll
            for (int g = 0; g < G; ++g) {
                float o[16];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float2 x = w[g][k], y = u[g][k];
                    if (KIND == F_INV21) {
                        o[4 * k] = x.x;
                        o[4 * k + 1] = y.x;
                        o[4 * k + 2] = x.y;
                        o[4 * k + 3] = y.y;
                    } else {
                        dst[(8 * g + 2 * k) * cs] = make_float2(x.x, y.x);
                        dst[(8 * g + 2 * k + 1) * cs] = make_float2(x.y, y.y);
                        mx = fmaxf(mx, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(y.x), fabsf(y.y))));
                    }
                }
                if (KIND == F_INV21) {
                    ptx::st_global_32(dst + 8 * g, o);
                    ptx::st_global_32(dst + 8 * g + 4, o + 8);
                }
            }
            if constexpr (KIND != F_INV21) {
                for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                if (lane == 0 && mx > 0.f)
                    atomicMax(reinterpret_cast<int *>(a.out_max + t / a.tiles_per_item), __float_as_int(mx));
            }
            return true;
        };
        for (int it = 0; it <= n_my; ++it) {
            if (it < n_my && !first(it)) break;
            if (it > 0 && !second(it - 1)) break;
            if (KIND != F_FWD12 && it < n_my && !between(it)) break;
            e_old = e_new;
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kFuMmaWarp) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, 512);
    }
}

constexpr int kFuItemTiles = 32;  // most tiles of an item (F_MID3: 4096 / 128, F_INV21: n3 / 2)

template <int KIND, int NK>
int fused_resident(kx_plan *p, int *ctas) {
    const void *kernel = reinterpret_cast<const void *>(bloch_fused_kernel<KIND, NK>);
    int per_sm = 0;
    if (int rc = raise_smem(p, kernel, fu_smem_bytes(NK))) return rc;
    if (int rc = resident_ctas(p, kernel, kFuThreads, fu_smem_bytes(NK), &per_sm)) return rc;
    *ctas = std::min(*ctas, per_sm * p->num_sms);
    return KX_OK;
}

template <int KIND, int NK>
int launch_fused(kx_plan *p, FuArgs a, long long R, cudaStream_t s) {
    a.N = (long long)p->N;
    if (R * a.N >= (1LL << 31)) return set_error(KX_ERR_ARG, "Bloch exchange: chunk too large for one launch");
    if (R == 0) return KX_OK;
    a.tiles_per_item = KIND == F_MID3 ? kFuPlane / 128 : p->n[2] / 2;
    a.n_tiles = (int)(R * a.tiles_per_item);
    a.status = p->d_status;
    a.timeout_cycles = 2000000000LL;
    const void *kernel = reinterpret_cast<const void *>(bloch_fused_kernel<KIND, NK>);
    if (int rc = raise_smem(p, kernel, fu_smem_bytes(NK))) return rc;
    if (int rc = prof_begin(p, PK_BLOCH, s)) return rc;
    const dim3 grid((unsigned)std::min(a.n_tiles, p->num_sms));  // one CTA per SM, all resident
    if constexpr (KIND == F_FWD12) {
        bloch_fused_kernel<KIND, NK><<<grid, kFuThreads, fu_smem_bytes(NK), s>>>(a);
    } else {
        void *args[] = {&a};
        const cudaError_t e =
            cudaLaunchCooperativeKernel(kernel, grid, dim3(kFuThreads), args, (size_t)fu_smem_bytes(NK), s);
        if (e == cudaErrorCooperativeLaunchTooLarge) {
            // the stream has fewer SMs than the device
            cudaGetLastError();
            p->fused_refused = true;
            p->prof.launches[PK_BLOCH] -= 1;
            if (int rc = prof_end(p, s)) return rc;
            return kFusedRefused;
        }
        KX_CUDA_TRY(e);
    }
    KX_LAUNCH_CHECK("bloch_fused_kernel launch");
    return prof_end(p, s);
}

}  // namespace

// Whether F_MID3 and F_INV21 can run: their CTAs wait for each other, so they must all be
// resident (one per SM), and a CTA must never hold two tiles of one item, as it would wait
// for its own next tile: tiles go to the CTAs in turn and an item has up to 32 neighbouring
// ones, so 32 CTAs are enough.  *fits = 0 on a smaller share of a device, whose calls
// take the single products, and, as a refused launch would invalidate it, for a capture
// with a plan one of whose launches was refused before.
int bloch_fused_fits(kx_plan *p, cudaStream_t s, bool *fits) {
    *fits = false;
    if (p->fused_refused) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        KX_CUDA_TRY(cudaStreamIsCapturing(s, &cap));
        if (cap != cudaStreamCaptureStatusNone) return KX_OK;
    }
    int coop = 0, ctas = p->num_sms;
    KX_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, p->device));
    int rc = p->n[2] == 64 ? fused_resident<F_MID3, 64>(p, &ctas) : fused_resident<F_MID3, 32>(p, &ctas);
    if (!rc) rc = fused_resident<F_INV21, 64>(p, &ctas);
    if (rc) return rc;
    *fits = coop && ctas >= p->num_sms && ctas >= kFuItemTiles;
    return KX_OK;
}

// items [r0, r0 + R): conj(P_m) F_v, both plane axes forward, into out; per-item maxima into out_max (zeroed)
int bloch_fused_forward(kx_plan *p, long long R, const float2 *P, const float2 *F, float2 *out, const __half *B1,
                        const __half *B2, const float *pmax, const float *fmax, long long r0, int n_orb,
                        float *out_max, cudaStream_t s) {
    FuArgs a = {};
    a.P = P;
    a.F = F;
    a.out = out;
    a.B1 = B1;
    a.B2 = B2;
    a.pmax = pmax;
    a.fmax = fmax;
    a.bound1 = 1.001f;  // |rho| <= max|psi_m| max|phi_v|
    a.bound2 = 1.001f * std::sqrt((float)p->n[0]);  // the bases are unitary
    a.r0 = r0;
    a.n_orb = n_orb;
    a.out_max = out_max;
    return launch_fused<F_FWD12, 64>(p, a, R, s);
}

// axis 3 forward, times f, axis 3 inverse; mid: 32 R words, zeroed
int bloch_fused_middle(kx_plan *p, long long R, const float2 *in, float2 *out, const __half *Bf, const __half *Bi,
                       const float *f, const float *in_max, int *mid, float *out_max, cudaStream_t s) {
    FuArgs a = {};
    a.in = in;
    a.out = out;
    a.B1 = Bf;
    a.B2 = Bi;
    a.f = f;
    a.in_max = in_max;
    a.mid = mid;
    a.out_max = out_max;
    return p->n[2] == 64 ? launch_fused<F_MID3, 64>(p, a, R, s) : launch_fused<F_MID3, 32>(p, a, R, s);
}

// both plane axes back: axis 2, then axis 1; mid: 32 R words, zeroed
int bloch_fused_inverse(kx_plan *p, long long R, const float2 *in, float2 *out, const __half *B2, const __half *B1,
                        const float *in_max, int *mid, cudaStream_t s) {
    FuArgs a = {};
    a.in = in;
    a.mid = mid;
    a.out = out;
    a.B1 = B2;
    a.B2 = B1;
    a.in_max = in_max;
    return launch_fused<F_INV21, 64>(p, a, R, s);
}

}  // namespace kx
