// Plain float64 Kronecker path on the CUDA cores: the accuracy reference on the
// GPU and the denominator of the tensor-core speed-up.
//
// For a chunk of R right-hand sides (pair products rho_ij = psi_i psi_j, or
// caller vectors), Sec. 3 Eq. 19 is applied as mode products with Vk^T (forward)
// and Vk (inverse), with the Hadamard scaling by f(Lambda) between them.
// Eq. 3-5 then accumulate (Vx psi)_i -= g_j psi_j phi_ij and
// (Vx psi)_j -= g_i psi_i phi_ij in a fixed pair order per grid point.
//
// What bounds it: float64 issue.  An SM retires about two float64 FMAs per clock (a
// warp's FMA occupies its sub-core for ~64 cycles), so loads, shared memory and
// index work hide behind the FMAs and only their number and their even spread over
// the SMs count.  Every 1D matrix here is symmetric under reflection of its axis
// (x -> n-1-x, periodic axes x -> n-x), so each eigenvector is even or odd: the
// even ones act on sums b(x) + b(x'), the odd ones on differences, and a mode
// product takes half the FMAs (n^2 / 2 a pencil instead of n^2).  Tiles shrink
// with the problem so that a small one still covers every SM several times, a
// thread's outputs are counted at compile time (a predicated-off FMA costs as much
// as a live one), the pair product is formed in the first product's load, and both
// products along axis 3 with the scaling between them run in one kernel.
// 32^3, 4 orbitals (10 solves): 954 us a call with dense products, 64 pencils per CTA
// and 32 outputs per thread of which n / 4 were live; 115 us so (14 us a mode
// product, whose FMAs alone take 9.4 us at two per clock and SM).
#include "kx_internal.h"
#include "kx_fd.cuh"

#include <algorithm>

namespace kx {
namespace {

// One axis as the kernels see it.  The he even eigenvectors come first in every
// spectral index, then the ho = n - he odd ones.  Rows r < np pair the points xa(r)
// and xb(r) = n-1-r, the remaining he - np rows are points that are their own mirror
// image.  Without parity: np = 0, he = n and every row is such a point.
struct Axis64 {
    int n, he, np, periodic;
    long long inner;
    const double *fe, *fo;  // forward tables [r][k] of the even and odd vectors
    const double *ie, *io;  // the same transposed, [k][r]
    __device__ __forceinline__ int xa(int r) const {
        if (r < np) return r + periodic;
        if (np == 0 && !periodic) return r;
        return periodic ? (r == np ? 0 : n / 2) : np;
    }
    __device__ __forceinline__ int xb(int r) const { return n - 1 - r; }
};

enum Mode64 { kFwd = 0, kFwdPair, kInv, kAxis3, kAxis3Energy };

struct Args64 {
    Axis64 ax;
    const double *in;
    double *out;
    long long n_cols;       // pencils
    long long N;
    int qb, groups;         // pencils per tile, output groups (threads / qb)
    const int2 *pairs;      // pair mode and energy weights
    const double *psi, *occ;
    const double *f;        // spectral order
    double *partial;        // per-CTA energy (nullable)
};

// acc_e[u] += sum_r me[r][e] T[row_e(r)], acc_o likewise, for the outputs
// e = g + groups u (indices past the end repeat the last and are not stored).
template <int U, class RowE, class RowO>
__device__ __forceinline__ void products64(const double *T, int ld, int q, int g, int groups, const double *me, int he,
                                           const double *mo, int ho, RowE row_e, RowO row_o, double (&ae)[U],
                                           double (&ao)[U]) {
    int ce[U], co[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        ae[u] = ao[u] = 0.0;
        ce[u] = min(g + groups * u, he - 1);
        co[u] = min(g + groups * u, max(ho - 1, 0));
    }
    int r = 0;
#pragma unroll 2
    for (; r < ho; ++r) {
        const double s = T[row_e(r) * ld + q], d = T[row_o(r) * ld + q];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            ae[u] = fma(__ldg(me + r * he + ce[u]), s, ae[u]);
            ao[u] = fma(__ldg(mo + r * ho + co[u]), d, ao[u]);
        }
    }
    for (; r < he; ++r) {
        const double s = T[row_e(r) * ld + q];
#pragma unroll
        for (int u = 0; u < U; ++u) ae[u] = fma(__ldg(me + r * he + ce[u]), s, ae[u]);
    }
}

template <int U, int MODE>
__global__ void __launch_bounds__(256) mode64_kernel(const Args64 a) {
    extern __shared__ double T[];  // n x (qb + 1): T[x * ld + q]
    __shared__ double red[8];
    const Axis64 ax = a.ax;
    const int n = ax.n, he = ax.he, ho = n - he, qb = a.qb, ld = qb + 1;
    const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31, warps = nt >> 5;
    const long long q0 = (long long)blockIdx.x * qb;
    const int nq = (int)min((long long)qb, a.n_cols - q0);
    const int q = tid % qb, g = tid / qb;
    const bool on = q < nq;
    // element (pencil, x) sits at base + x * inner
    long long base = 0;
    int i_in = 0;
    double w = 0.0;
    if (MODE == kFwdPair) {  // axis 1: pencils are rows of n values, formed from the pair's orbitals
        const long long ppi = a.N / n;
        for (int r = warp; r < nq; r += warps) {
            const long long item = (q0 + r) / ppi, off = (q0 + r - item * ppi) * n;
            const int2 ij = __ldg(a.pairs + item);
            const double *pi = a.psi + (long long)ij.x * a.N + off, *pj = a.psi + (long long)ij.y * a.N + off;
            for (int x = lane; x < n; x += 32) T[x * ld + r] = pi[x] * pj[x];
        }
    } else if (ax.inner == 1) {
        const double *src = a.in + q0 * n;
        for (int r = warp; r < nq; r += warps)
            for (int x = lane; x < n; x += 32) T[x * ld + r] = src[(long long)r * n + x];
    } else if (on) {
        const unsigned qq = (unsigned)(q0 + q), in32 = (unsigned)ax.inner;  // n_cols < 2^31
        const unsigned o = qq / in32;
        i_in = (int)(qq - o * in32);
        base = (long long)o * n * ax.inner + i_in;
        for (int x = g; x < n; x += a.groups) T[x * ld + q] = a.in[base + (long long)x * ax.inner];
        if ((MODE == kAxis3 || MODE == kAxis3Energy) && a.partial != nullptr) {
            const int2 ij = __ldg(a.pairs + o);  // axis 3: one item per outer index
            w = (ij.x == ij.y) ? 1.0 : 2.0;
            if (a.occ) w *= a.occ[ij.x] * a.occ[ij.y];
        }
    }
    __syncthreads();
    double ae[U], ao[U];
    if (MODE != kInv) {
        // fold: sums into xa, differences into xb
        if (on)
            for (int r = g; r < ax.np; r += a.groups) {
                const int xa = ax.xa(r) * ld + q, xb = ax.xb(r) * ld + q;
                const double u = T[xa], v = T[xb];
                T[xa] = u + v;
                T[xb] = u - v;
            }
        __syncthreads();
        if (on)
            products64<U>(T, ld, q, g, a.groups, ax.fe, he, ax.fo, ho, [&](int r) { return ax.xa(r); },
                          [&](int r) { return ax.xb(r); }, ae, ao);
        double e = 0.0;
        if (MODE == kAxis3 || MODE == kAxis3Energy) {
            if (on) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int k = g + a.groups * u;
                    if (k < he) {
                        const double fy = __ldg(a.f + (long long)k * ax.inner + i_in) * ae[u];
                        e = fma(fy, ae[u], e);
                        ae[u] = fy;
                    }
                    if (k < ho) {
                        const double fy = __ldg(a.f + (long long)(he + k) * ax.inner + i_in) * ao[u];
                        e = fma(fy, ao[u], e);
                        ao[u] = fy;
                    }
                }
            }
            if (a.partial != nullptr) {
                e *= w;
                for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
                if (lane == 0) red[warp] = e;
                __syncthreads();
                if (tid == 0) {
                    double s = 0.0;
                    for (int k = 0; k < warps; ++k) s += red[k];
                    a.partial[blockIdx.x] = s;
                }
            }
            if (MODE == kAxis3Energy) return;
        }
        __syncthreads();
        if (on) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int k = g + a.groups * u;
                if (k < he) T[k * ld + q] = ae[u];
                if (k < ho) T[(he + k) * ld + q] = ao[u];
            }
        }
        __syncthreads();
    }
    if (MODE == kInv || MODE == kAxis3) {
        if (on)
            products64<U>(T, ld, q, g, a.groups, ax.ie, he, ax.io, ho, [&](int k) { return k; },
                          [&](int k) { return he + k; }, ae, ao);
        __syncthreads();
        if (on) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int r = g + a.groups * u;
                if (r < ax.np) {
                    T[ax.xa(r) * ld + q] = ae[u] + ao[u];
                    T[ax.xb(r) * ld + q] = ae[u] - ao[u];
                } else if (r < he) {
                    T[ax.xa(r) * ld + q] = ae[u];
                }
            }
        }
        __syncthreads();
    }
    if (ax.inner == 1) {
        double *dst = a.out + q0 * n;
        for (int r = warp; r < nq; r += warps)
            for (int x = lane; x < n; x += 32) dst[(long long)r * n + x] = T[x * ld + r];
    } else if (on) {
        for (int x = g; x < n; x += a.groups) a.out[base + (long long)x * ax.inner] = T[x * ld + q];
    }
}

// ex += factor sum partial[0 .. count): fixed strided sums and a fixed tree.
__global__ void __launch_bounds__(512) energy_sum64_kernel(const double *__restrict__ partial, int count,
                                                           double factor, double *e_x) {
    __shared__ double red[16];
    double s = 0.0;
    for (int i = threadIdx.x; i < count; i += 512) s += partial[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < 16; ++k) t += red[k];
        *e_x += factor * t;
    }
}

// (Vx psi)_i -= g_j psi_j phi_ij, (Vx psi)_j -= g_i psi_i phi_ij (i != j), one thread per
// grid point, pairs visited in chunk order (deterministic, no atomics).
__global__ void accum_f64_kernel(const double *__restrict__ phi, const int2 *__restrict__ pairs, int R,
                                 const double *__restrict__ psi, const double *__restrict__ occ, size_t N,
                                 double *__restrict__ vx) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        for (int r = 0; r < R; ++r) {
            int2 ij = pairs[r];
            double v = phi[(size_t)r * N + x];
            double gi = occ ? occ[ij.x] : 1.0, gj = occ ? occ[ij.y] : 1.0;
            vx[(size_t)ij.x * N + x] -= gj * psi[(size_t)ij.y * N + x] * v;
            if (ij.x != ij.y) vx[(size_t)ij.y * N + x] -= gi * psi[(size_t)ij.x * N + x] * v;
        }
    }
}

// Parity tables of one axis per CTA.  Periodic axes: cos(2 pi k x / n) and
// sin(2 pi k x / n) in closed form with the stencil's symbol as eigenvalues.
// Dirichlet axes: the plan's eigenvectors sorted by parity and symmetrised; *ok = 0
// (then the whole matrix goes into the even table) if one has none: what symmetrising
// drops of a unit vector is at most 2.1e-12 over every n and stencil order (the
// eigensolver's own error), results are held to 1e-11.
constexpr double kParityTol = 1e-11;
struct Tables64 {
    int n[3], periodic[3];
    double h[3];
    int order;
    const double *V[3], *lam[3];
    double *tab[3];   // 2 n^2 each: fe | fo | ie | io
    double *lam_out;  // 3 x kMaxN, spectral order
    int *ok;          // 3
};
__global__ void tables64_kernel(const Tables64 t) {
    __shared__ int par[kMaxN], slot[kMaxN];
    __shared__ int good;
    const int axis = blockIdx.x, n = t.n[axis], k = threadIdx.x;
    const bool periodic = t.periodic[axis] != 0;
    double *lam_out = t.lam_out + axis * kMaxN;
    const double *V = t.V[axis];
    int np = periodic ? (n - 1) / 2 : n / 2, he = n - np;
    if (k == 0) good = 1;
    __syncthreads();
    if (!periodic) {
        if (k < n) {
            double s = 0.0, odd = 0.0, even = 0.0;  // overlap with the mirror image, largest parts of each parity
            for (int x = 0; x < n; ++x) {
                const double a = V[x * n + k], b = V[(n - 1 - x) * n + k];
                s += a * b;
                odd = fmax(odd, 0.5 * fabs(a - b));
                even = fmax(even, 0.5 * fabs(a + b));
            }
            par[k] = s > 0.0 ? 0 : 1;
            if (!((s > 0.0 ? odd : even) < kParityTol)) good = 0;
        }
        __syncthreads();
        if (k == 0) {
            int cnt[2] = {0, 0};
            for (int i = 0; i < n; ++i) slot[i] = cnt[par[i]]++;
            if (cnt[0] != he) good = 0;
        }
        __syncthreads();
        if (!good) {
            np = 0;
            he = n;
        }
    }
    if (k == 0) t.ok[axis] = good;
    const int ho = n - he;
    double *fe = t.tab[axis], *fo = fe + (size_t)he * he, *ie = fo + (size_t)ho * ho, *io = ie + (size_t)he * he;
    if (k >= n) return;
    if (periodic) {
        // column k < he: cos(2 pi k x / n); the rest: sin(2 pi m x / n), m = k - he + 1
        const bool even = k < he;
        const int m = even ? k : k - he + 1;
        const double c = sqrt((even && (m == 0 || 2 * m == n) ? 1.0 : 2.0) / n);
        const int rows = even ? he : ho, col = even ? k : k - he;
        for (int r = 0; r < rows; ++r) {
            const int x = r < np ? r + 1 : (r == np ? 0 : n / 2);
            double sv, cv;
            sincospi(2.0 * (double)(((long long)m * x) % n) / n, &sv, &cv);
            const double v = c * (even ? cv : sv);
            (even ? fe : fo)[r * rows + col] = v;
            (even ? ie : io)[col * rows + r] = v;
        }
        const int mo = t.order / 2;
        double s = fd_weight(mo, 0);
        for (int p = 1; p <= mo; ++p) s += 2.0 * fd_weight(mo, p) * cospi(2.0 * (double)(((long long)p * m) % n) / n);
        lam_out[k] = s / (t.h[axis] * t.h[axis]);
    } else if (good) {
        const bool even = par[k] == 0;
        const int rows = even ? he : ho, col = slot[k];
        for (int r = 0; r < rows; ++r) {
            const double v = r < np ? 0.5 * (even ? V[r * n + k] + V[(n - 1 - r) * n + k]
                                                  : V[r * n + k] - V[(n - 1 - r) * n + k])
                                    : V[r * n + k];  // the middle point
            (even ? fe : fo)[r * rows + col] = v;
            (even ? ie : io)[col * rows + r] = v;
        }
        lam_out[even ? col : he + col] = t.lam[axis][k];
    } else {
        for (int x = 0; x < n; ++x) {
            fe[x * n + k] = V[x * n + k];
            ie[k * n + x] = V[x * n + k];
        }
        lam_out[k] = t.lam[axis][k];
    }
}

__global__ void ftable64_kernel(int n1, int n2, int n3, const double *lam, int kind, double omega, double *f) {
    const size_t N = (size_t)n1 * n2 * n3;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < N; e += (size_t)gridDim.x * blockDim.x) {
        const int k1 = (int)(e % n1), k2 = (int)((e / n1) % n2), k3 = (int)(e / ((size_t)n1 * n2));
        f[e] = kernel_f_value(kind, omega, lam[k1] + lam[kMaxN + k2] + lam[2 * kMaxN + k3]);
    }
}

template <int MODE, int U>
int launch_u(kx_plan *p, const Args64 &a, unsigned blocks, int threads, size_t smem, cudaStream_t s) {
    if (int rc = raise_smem(p, reinterpret_cast<const void *>(mode64_kernel<U, MODE>), sizeof(double) * kMaxN * 65))
        return rc;
    mode64_kernel<U, MODE><<<blocks, threads, smem, s>>>(a);
    KX_LAUNCH_CHECK("mode64_kernel launch");
    return KX_OK;
}

// Tile width: 64 pencils (256 threads) where that still gives every SM eight tiles,
// else 32, 16 (128 threads), never so narrow that a group has no output.
// 32^3, 10 pairs (10,240 pencils a mode): 16 pencils, 640 tiles.
void tile_shape(const kx_plan *p, int axis, long long n_cols, int *qb, int *threads) {
    const int he = p->p64_he[axis];
    *qb = 64;
    *threads = 256;
    for (int w : {32, 16}) {
        if (n_cols / *qb >= 8LL * p->num_sms || 128 / w > he) break;
        *qb = w;
        *threads = 128;
    }
}

template <int MODE>
int launch_mode(kx_plan *p, int axis, int R, Args64 a, cudaStream_t s, int *blocks_out = nullptr) {
    const int n = p->n[axis], he = p->p64_he[axis], ho = n - he;
    a.ax.n = n;
    a.ax.he = he;
    a.ax.periodic = p->bc[axis] == KX_PERIODIC ? 1 : 0;
    a.ax.np = he == n ? 0 : ho;  // without parity every row stands alone
    a.ax.inner = axis == 0 ? 1 : (axis == 1 ? p->n[0] : (long long)p->n[0] * p->n[1]);
    a.ax.fe = p->d_p64_tab[axis];
    a.ax.fo = a.ax.fe + (size_t)he * he;
    a.ax.ie = a.ax.fo + (size_t)ho * ho;
    a.ax.io = a.ax.ie + (size_t)he * he;
    a.N = (long long)p->N;
    a.n_cols = (long long)R * (long long)(p->N / n);
    int threads;
    tile_shape(p, axis, a.n_cols, &a.qb, &threads);
    a.groups = threads / a.qb;
    const size_t smem = sizeof(double) * (size_t)n * (a.qb + 1);
    const unsigned blocks = (unsigned)((a.n_cols + a.qb - 1) / a.qb);
    if (blocks_out) *blocks_out = (int)blocks;
    const int u = (he + a.groups - 1) / a.groups;
    if (int rc = prof_begin(p, PK_FP64_MODE, s)) return rc;
    int rc;
    if (u <= 1) rc = launch_u<MODE, 1>(p, a, blocks, threads, smem, s);
    else if (u <= 2) rc = launch_u<MODE, 2>(p, a, blocks, threads, smem, s);
    else if (u <= 3) rc = launch_u<MODE, 3>(p, a, blocks, threads, smem, s);
    else if (u <= 4) rc = launch_u<MODE, 4>(p, a, blocks, threads, smem, s);
    else if (u <= 5) rc = launch_u<MODE, 5>(p, a, blocks, threads, smem, s);
    else if (u <= 6) rc = launch_u<MODE, 6>(p, a, blocks, threads, smem, s);
    else if (u <= 8) rc = launch_u<MODE, 8>(p, a, blocks, threads, smem, s);
    else if (u <= 10) rc = launch_u<MODE, 10>(p, a, blocks, threads, smem, s);
    else if (u <= 12) rc = launch_u<MODE, 12>(p, a, blocks, threads, smem, s);
    else if (u <= 17) rc = launch_u<MODE, 17>(p, a, blocks, threads, smem, s);
    else rc = launch_u<MODE, 32>(p, a, blocks, threads, smem, s);  // no parity
    if (rc) return rc;
    return prof_end(p, s);
}

// f(L) on R items: forward modes 1 (of `src`, or of the pairs' products) and 2, axis 3
// both ways with the scaling (and energy), inverse modes 2 and 1 into `dst`.
int fl_chunk(kx_plan *p, const double *src, double *b0, double *b1, double *dst, int R, bool energy_only,
             const int2 *pairs, const double *psi, const double *occ, double *partial, double *e_x, cudaStream_t s) {
    int rc;
    Args64 a{};
    a.in = src;
    a.out = b0;
    a.pairs = pairs;
    a.psi = psi;
    if ((rc = src ? launch_mode<kFwd>(p, 0, R, a, s) : launch_mode<kFwdPair>(p, 0, R, a, s))) return rc;
    a.in = b0;
    a.out = b1;
    if ((rc = launch_mode<kFwd>(p, 1, R, a, s))) return rc;
    a.in = b1;
    a.out = b0;
    a.occ = occ;
    a.f = p->d_p64_f;
    a.partial = e_x != nullptr ? partial : nullptr;
    int blocks = 0;
    if ((rc = energy_only ? launch_mode<kAxis3Energy>(p, 2, R, a, s, &blocks) : launch_mode<kAxis3>(p, 2, R, a, s, &blocks)))
        return rc;
    if (e_x != nullptr) {
        p->prof.launches[PK_FP64_OTHER] += 1;
        energy_sum64_kernel<<<1, 512, 0, s>>>(partial, blocks, -0.5 * p->dV, e_x);
        KX_LAUNCH_CHECK("energy_sum64_kernel launch");
    }
    if (energy_only) return KX_OK;
    a.partial = nullptr;
    a.in = b0;
    a.out = b1;
    if ((rc = launch_mode<kInv>(p, 1, R, a, s))) return rc;
    a.in = b1;
    a.out = dst;
    return launch_mode<kInv>(p, 0, R, a, s);
}

// Energy partials of a chunk: the axis-3 tiles (at least 16 pencils each).
size_t partials64(const kx_plan *p, long chunk) { return (size_t)chunk * (p->N / p->n[2]) / 16 + 1; }

}  // namespace

// Tables of the parity form: made with the plan for KX_FP64, and by the multipole
// set-up (which solves in float64) for the others.  Synchronous.
int fp64_setup(kx_plan *p) {
    if (p->d_p64_f) return KX_OK;
    Tables64 t{};
    int *d_ok = nullptr, ok[3] = {0, 0, 0};
    double *d_lam = nullptr, *f = nullptr;
    t.order = p->fd_order;
    for (int a = 0; a < 3; ++a) {
        t.n[a] = p->n[a];
        t.periodic[a] = p->bc[a] == KX_PERIODIC ? 1 : 0;
        t.h[a] = p->h[a];
        t.V[a] = p->d_V[a];
        t.lam[a] = p->d_lam[a];
        if (!p->d_p64_tab[a]) KX_CUDA_TRY(cudaMalloc(&p->d_p64_tab[a], sizeof(double) * 2 * p->n[a] * p->n[a]));
        t.tab[a] = p->d_p64_tab[a];
    }
    KX_CUDA_TRY(cudaMalloc(&f, sizeof(double) * p->N));
    cudaError_t e = cudaMalloc(&d_lam, sizeof(double) * 3 * kMaxN + sizeof(int) * 4);
    if (e == cudaSuccess) {
        d_ok = reinterpret_cast<int *>(d_lam + 3 * kMaxN);
        t.lam_out = d_lam;
        t.ok = d_ok;
        tables64_kernel<<<3, kMaxN>>>(t);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        const int blocks = (int)std::min<size_t>((p->N + 255) / 256, (size_t)4 * p->num_sms);
        ftable64_kernel<<<blocks, 256>>>(p->n[0], p->n[1], p->n[2], d_lam, p->kind, p->omega, f);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(ok, d_ok, sizeof(ok), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    cudaFree(d_lam);
    if (e != cudaSuccess) {
        cudaFree(f);
        return cuda_error(e, "float64 tables");
    }
    for (int a = 0; a < 3; ++a) {
        const int n = p->n[a], np = p->bc[a] == KX_PERIODIC ? (n - 1) / 2 : n / 2;
        p->p64_he[a] = ok[a] ? n - np : n;
    }
    p->d_p64_f = f;
    return KX_OK;
}

long fp64_chunk(const kx_plan *p, long want) {
    const size_t budget = (size_t)2 << 30;  // scratch budget of the float64 path
    long c = (long)std::max<size_t>(1, budget / (2 * p->N * sizeof(double)));
    return std::max(1L, std::min(c, want));
}

size_t fp64_workspace_bytes(const kx_plan *p, long chunk) {
    return sizeof(double) * (2 * chunk * p->N + partials64(p, chunk));
}

int fp64_apply_fL(kx_plan *p, int n_rhs, const double *b, double *x, cudaStream_t s) {
    long chunk = fp64_chunk(p, n_rhs);
    int rc = ensure_workspace(p, fp64_workspace_bytes(p, chunk));
    if (rc) return rc;
    double *w0 = (double *)p->ws.ptr;
    double *w1 = w0 + chunk * p->N;
    for (long c0 = 0; c0 < n_rhs; c0 += chunk) {
        int R = (int)std::min<long>(chunk, n_rhs - c0);
        rc = fl_chunk(p, b + c0 * p->N, w0, w1, x + c0 * p->N, R, false, nullptr, nullptr, nullptr, nullptr, nullptr, s);
        if (rc) return rc;
    }
    return KX_OK;
}

int fp64_vx(kx_plan *p, int n_orb, const double *psi, const double *occ, double *vx, double *ex,
            bool energy_only, cudaStream_t s, long pair_begin, long pair_end) {
    int rc = ensure_pairs(p, n_orb, s, pair_begin, pair_end);
    if (rc) return rc;
    long P = p->h_group_first.back();  // items of the (range-restricted) pair list
    pair_begin = 0;
    pair_end = P;
    long chunk = fp64_chunk(p, std::max(1L, P));
    rc = ensure_workspace(p, fp64_workspace_bytes(p, chunk));
    if (rc) return rc;
    double *w0 = (double *)p->ws.ptr;
    double *w1 = w0 + chunk * p->N;
    double *partial = w1 + chunk * p->N;
    if (!energy_only) KX_CUDA_TRY(cudaMemsetAsync(vx, 0, sizeof(double) * n_orb * p->N, s));
    if (ex) KX_CUDA_TRY(cudaMemsetAsync(ex, 0, sizeof(double), s));
    const int2 *pairs = (const int2 *)p->d_pairs;
    for (long c0 = pair_begin; c0 < pair_end; c0 += chunk) {
        int R = (int)std::min<long>(chunk, pair_end - c0);
        rc = fl_chunk(p, nullptr, w0, w1, w0, R, energy_only, pairs + c0, psi, occ, partial, ex, s);
        if (rc) return rc;
        if (!energy_only) {
            p->prof.launches[PK_FP64_OTHER] += 1;
            int ab = (int)std::min<size_t>((p->N + 255) / 256, (size_t)8 * p->num_sms);
            accum_f64_kernel<<<ab, 256, 0, s>>>(w0, pairs + c0, R, psi, occ, p->N, vx);
            KX_LAUNCH_CHECK("accum_f64_kernel launch");
        }
    }
    return KX_OK;
}

}  // namespace kx
