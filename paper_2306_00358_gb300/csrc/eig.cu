// Isometry of the HOTRG step: leading eigenvectors of the environment M.
//
// The paper (Sec. 2, SVD helper of the coarse-graining listing) keeps the
// leading min(n, Dcut) left singular vectors of M; M is a Gram matrix
// (symmetric PSD), so these are its leading eigenvectors.  Here they come from
// block subspace iteration:
//   Y = M Q                                  (GEMM, the context's precision)
//   H = Q^T Y, H = W diag(theta) W^T         (Rayleigh-Ritz, FP64 Jacobi)
//   residual |Y w_i - theta_i Q w_i| <= tol * theta_1 for i < Dn  -> done
//   Q <- orth(Y W)                           (FP64 Cholesky-QR, two passes)
// Cholesky-QR works on column-normalised blocks; a column whose Cholesky
// pivot shows it is numerically dependent on the earlier ones is replaced by
// a fresh seeded random column (this happens when M's spectrum falls below
// rounding, e.g. in the ordered phase).  All blocks are column-major (n x m).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>

#include "internal.h"
#include "jacobi32.cuh"

namespace trg {

namespace {

constexpr int MAX_M = 112;   // largest block (Dcut + oversampling) held in shared memory

// The small kernels of an iteration are chained: each may be brought onto the
// SMs while the one before it still runs, waits there for that one's results
// (griddepcontrol.wait: all of its memory, and by the same wait all of the
// kernels' before it) and lets the next one do the same, which hides the launch.
// A kernel launched through launch_chained calls after_previous first.  Isometry
// n = 256 (FP64) 2.02 -> 1.82 ms, n = 1024 (split) 2.29 -> 2.17 ms.
__device__ __forceinline__ void after_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
void launch_chained_if(bool chain, Ctx& ctx, void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = chain ? 1 : 0;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ctx.stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    TRG_CUDA(cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...));
}
template <typename... P, typename... A>
void launch_chained(Ctx& ctx, void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, A&&... args) {
    launch_chained_if(true, ctx, kernel, grid, block, smem, std::forward<A>(args)...);
}
// The kernels whose blocks are the work of an SM each (Gram parts, factor and
// solve) are chained only while their blocks are short: brought in early, two
// may come to share an SM while another has none.  Both chained against neither,
// an isometry of Dcut sqrt(n): n = 1225 4.00 / 4.06 ms, 1600 4.87 / 4.89, 2025
// 7.18 / 7.57, 2704 9.71 / 9.48, 3364 14.65 / 13.04, 4096 17.5 / 15.3.
inline bool chain_wide(const Ctx& ctx, int64_t n) { return n <= 16 * ctx.sm_count; }

__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// Seeded uniform(-1, 1) entries; only columns with flags[c] != 0 when flags is given.
__global__ void k_rand_cols(double* Y, int64_t n, int m, const int* flags, uint64_t seed, uint64_t salt) {
    const int c = blockIdx.y;
    if (c >= m || (flags && !flags[c])) return;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
        uint64_t h = splitmix64(seed ^ splitmix64(salt * 0x100000001B3ull + (uint64_t)c * 0x9E3779B1ull + (uint64_t)r));
        Y[(int64_t)c * n + r] = 2.0 * ((double)(h >> 11) * (1.0 / 9007199254740992.0)) - 1.0;
    }
}

template <int NT>
__device__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < 32) {
        s = (threadIdx.x < NT / 32) ? red[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) red[0] = s;
    }
    __syncthreads();
    return red[0];
}

// Scale every column to unit 2-norm; flag columns that are zero or not finite.
__global__ void __launch_bounds__(256) k_col_normalize(double* Y, int64_t n, int* flags) {
    after_previous();
    __shared__ double red[32];
    const int c = blockIdx.x;
    if (threadIdx.x == 0) flags[c] = 0;
    double* y = Y + (int64_t)c * n;
    double mx = 0.0;
    for (int64_t r = threadIdx.x; r < n; r += 256) mx = fmax(mx, fabs(y[r]));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int i = 0; i < 8; ++i) v = fmax(v, red[i]);
        red[8] = v;
    }
    __syncthreads();
    mx = red[8];
    __syncthreads();
    if (!(mx > 0.0) || !isfinite(mx)) {
        if (threadIdx.x == 0) flags[c] = 1;
        return;
    }
    const double inv = 1.0 / mx;   // scale first so the squares cannot under/overflow
    double s = 0.0;
    for (int64_t r = threadIdx.x; r < n; r += 256) { const double v = y[r] * inv; s = fma(v, v, s); }
    s = block_sum<256>(s, red);
    const double scale = inv / sqrt(s);
    for (int64_t r = threadIdx.x; r < n; r += 256) y[r] *= scale;
}

// What the host reads of a solve while it runs: mapped host memory that the
// deciding kernels write, `seq` last.
struct EigBox {
    unsigned long long seq;
    int nbad;                 // dependent columns of the last Cholesky-QR pass
    int status;
    int sweeps[2];
    double pivmin;            // its smallest pivot ratio d_j / G_jj
    double res;
    double theta[MAX_M];
};
__device__ __forceinline__ void box_done(EigBox* box, unsigned long long seq) {
    __threadfence_system();
    *(volatile unsigned long long*)&box->seq = seq;
}

// One Cholesky-QR pass after the Gram product: G = L L^T (m x m, unit
// columns), then Y <- Y L^{-T} for the block's RB rows.  A pivot d_j <= tau *
// G_jj marks column j as dependent (flags[j] = 1, counted in box->nbad); the
// pivot is replaced by G_jj so the factorisation can continue, and Y is left
// as it is unless `always`.  Every block factors G itself (the same bits), so
// no launch and no host decision lies between the two parts; block 0 tells
// the host (box, may be null) as soon as the pivots are known, while the
// triangular solve still runs.
//
// Factorisation.  Bound by the chain of FP64 operations from pivot to pivot: a
// warp's FP64 instruction holds its quarter of the SM's pipe for 64 clocks,
// with one active lane or with 32.  So the chain is kept to warp 0, while the
// warps of the other three quarters update the trailing triangle:
//  - warp 0 takes two columns a step in registers, their pivots by shuffle,
//    and brings the next two up to date itself while the others apply the
//    current two to the rest: one barrier per two columns;
//  - pivot ratios (a division each) are taken in parallel at the end.
// The trailing elements (i, k), k <= i, are listed once by k descending, so
// those of a step are a prefix of the list and all lanes work.  Every element
// goes through the operations of the plain right-looking form in its order
// (scale by rsqrt(d_j), subtract in order of j): the bits of Q decide the
// digits of the split products that follow, so a rounding changed here moves
// split-mode vectors by far more than a rounding.
//
// Triangular solve.  Right-looking in steps of four columns: one warp solves
// a step's 4 x 4 triangle for the block's rows, then all warps subtract its
// products from the later columns (a lane per row; with RB < 32 the lanes'
// groups take different columns).  Bound by the FP64 pipe (n m^2 / 2 FMAs)
// for large n and by the chain of steps for small n, where fewer rows per
// block use more SMs (chol_trsm below).
// Measured, both parts, at 256 x 40 / 1024 x 56 / 4096 x 88: 39.9 / 58.0 / 124.7 us (as
// two kernels 42 / 61 / 129, with one column a step, two barriers and the
// division in the chain, 32 rows a block and a barrier per column 62 / 98 / 192).
constexpr int CHOL_THREADS = 512;
__host__ __device__ constexpr int chol_even(int m) { return m + (m & 1); }
__host__ __device__ constexpr int chol_table_entries(int m) { return chol_even(m) * (chol_even(m) + 1) / 2; }
template <int RB>
__global__ void __launch_bounds__(CHOL_THREADS) k_chol_trsm(const double* G, double* Y, int64_t n, int m, double tau,
                                                            int always, int* flags, EigBox* box,
                                                            unsigned long long seq) {
    after_previous();
    // me rows of ld = me + 1 (an odd stride: the rows of one column fall in
    // different banks; an odd m gets a unit row and column), tau times the
    // diagonal, the diagonal, the pivots before a replacement, two buffers of
    // a step's two columns, RB rows of Y, 2 x 4 x RB solved values, then the list
    extern __shared__ double L[];
    __shared__ int bad_s;
    const int me = chol_even(m), ld = me + 1;
    double* gd = L + me * ld;
    double* tg = gd + me;
    double* draw = tg + me;
    double* cols = draw + me;              // [2][2][me]
    double* rows = cols + 4 * me;
    double* xb = rows + RB * (m + 1);
    uint16_t* tab = (uint16_t*)(xb + 8 * RB);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t r0 = (int64_t)blockIdx.x * RB;
    if (threadIdx.x == 0) bad_s = 0;
    for (int e = threadIdx.x; e < m * RB; e += CHOL_THREADS) {
        const int j = e / RB, t = e % RB;
        rows[t * (m + 1) + j] = (r0 + t < n) ? Y[(int64_t)j * n + r0 + t] : 0.0;
    }
    for (int e = threadIdx.x; e < me * me; e += CHOL_THREADS) {
        const int i = e / me, j = e % me;
        L[i * ld + j] = (i < m && j < m) ? G[i * m + j] : (i == j ? 1.0 : 0.0);
    }
    for (int i = threadIdx.x; i < me; i += CHOL_THREADS) {
        gd[i] = i < m ? G[(int64_t)i * m + i] : 1.0;
        tg[i] = i < m ? tau * gd[i] : 0.0;
    }
    for (int e = threadIdx.x; e < chol_table_entries(m); e += CHOL_THREADS) {
        // group q = me-1-k holds the q+1 elements (k..me-1, k) from offset q(q+1)/2
        int q = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
        while (q * (q + 1) / 2 > e) --q;
        while ((q + 1) * (q + 2) / 2 <= e) ++q;
        const int k = me - 1 - q, i = k + (e - q * (q + 1) / 2);
        tab[e] = (uint16_t)((i << 7) | k);
    }
    __syncthreads();
    for (int j = 0; j < me; j += 2) {
        double* cur = cols + ((j >> 1) & 1) * 2 * me;           // this step's columns
        const double* old = cols + (((j >> 1) & 1) ^ 1) * 2 * me;   // the previous step's
        if (warp == 0) {
            // columns j, j + 1 less the previous step's part, rows i >= j
            double x0[4], x1[4];
            const double v00 = j ? old[j] : 0.0, v01 = j ? old[j + 1] : 0.0;
            const double v10 = j ? old[me + j] : 0.0, v11 = j ? old[me + j + 1] : 0.0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = j + lane + 32 * q;
                x0[q] = x1[q] = 0.0;
                if (j + 32 * q < me && i < me) {
                    x0[q] = L[i * ld + j];
                    x1[q] = L[i * ld + j + 1];
                    if (j) {
                        const double u0 = old[i], u1 = old[me + i];
                        x0[q] = fma(-u0, v00, x0[q]);
                        x1[q] = fma(-u0, v01, x1[q]);
                        x0[q] = fma(-u1, v10, x0[q]);
                        x1[q] = fma(-u1, v11, x1[q]);
                    }
                }
            }
            // pivot c of the step: flagged and replaced if dependent
            auto pivot = [&](double d, int c) {
                if (lane == 0) draw[c] = d;
                if (!(d > tg[c]) || !isfinite(d)) {
                    if (lane == 0 && c < m) {
                        ++bad_s;
                        if (blockIdx.x == 0) flags[c] = 1;
                    }
                    d = (gd[c] > 0.0 && isfinite(gd[c])) ? gd[c] : 1.0;
                }
                return d;
            };
            const double d0 = pivot(__shfl_sync(0xffffffffu, x0[0], 0), j);
            const double il0 = rsqrt(d0);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (j + 32 * q < me) x0[q] *= il0;
            const double w = __shfl_sync(0xffffffffu, x0[0], 1);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (j + 32 * q < me) x1[q] = fma(-x0[q], w, x1[q]);
            const double d1 = pivot(__shfl_sync(0xffffffffu, x1[0], 1), j + 1);
            const double il1 = rsqrt(d1);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = j + lane + 32 * q;
                if (j + 32 * q < me && i < me) {
                    x1[q] *= il1;
                    cur[i] = x0[q];
                    cur[me + i] = x1[q];
                    L[i * ld + j] = i == j ? d0 * il0 : x0[q];
                    L[i * ld + j + 1] = i == j + 1 ? d1 * il1 : x1[q];
                }
            }
        } else if (j && (warp & 3)) {
            // the previous step's part of the columns from j + 2 on
            const int n2 = me - 2 - j, cnt = n2 * (n2 + 1) / 2;
            const int t0 = ((warp >> 2) * 3 + (warp & 3) - 1) * 32 + lane;
            for (int e = t0; e < cnt; e += CHOL_THREADS / 4 * 3) {
                const unsigned t = tab[e];
                const int i = (int)(t >> 7), k = (int)(t & 127u);
                double v = L[i * ld + k];
                v = fma(-old[i], old[k], v);
                v = fma(-old[me + i], old[me + k], v);
                L[i * ld + k] = v;
            }
        }
        __syncthreads();
    }
    const int bad = bad_s;
    double* dinv = cols;                   // 1 / L_jj
    if (blockIdx.x == 0 && box && warp == CHOL_THREADS / 32 - 1) {
        double pm = 1.0;   // 1 / pivmin bounds cond(Y)^2 from below
        for (int i = lane; i < m; i += 32) pm = fmin(pm, (gd[i] > 0.0 && isfinite(draw[i])) ? draw[i] / gd[i] : 0.0);
        for (int o = 16; o > 0; o >>= 1) pm = fmin(pm, __shfl_xor_sync(0xffffffffu, pm, o));
        if (lane == 0) {
            box->nbad = bad;
            box->pivmin = pm;
            box_done(box, seq);
        }
    }
    if (bad && !always) return;
    for (int i = threadIdx.x; i < m; i += CHOL_THREADS) dinv[i] = 1.0 / L[i * ld + i];
    __syncthreads();

    constexpr int CG = 32 / RB;            // columns a warp updates at a time
    constexpr int WARPS = CHOL_THREADS / 32;
    const int row = lane % RB, cg = lane / RB;
    double* y = rows + row * (m + 1);
    for (int j = 0, s = 0; j < m; j += 4, ++s) {
        double* xs = xb + (s & 1) * 4 * RB;
        const int w = min(4, m - j);
        if (warp == (s & (WARPS - 1))) {
            // the step's triangle, every lane group redundantly
            double x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (q < w) {
                    double v = y[j + q];
#pragma unroll
                    for (int p = 0; p < q; ++p) v = fma(-L[(j + q) * ld + j + p], x[p], v);
                    x[q] = v * dinv[j + q];
                } else {
                    x[q] = 0.0;
                }
            }
            if (cg == 0) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    xs[q * RB + row] = x[q];
                    if (q < w) y[j + q] = x[q];
                }
            }
        }
        __syncthreads();
        if (j + 4 >= m) break;
        double x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = xs[q * RB + row];
        for (int k = j + 4 + warp * CG + cg; k < m; k += WARPS * CG) {
            const double* lr = L + k * ld + j;
            double v = y[k];
#pragma unroll
            for (int q = 0; q < 4; ++q) v = fma(-lr[q], x[q], v);
            y[k] = v;
        }
        __syncthreads();    // the next triangle's columns belong to several warps
    }
    for (int e = threadIdx.x; e < m * RB; e += CHOL_THREADS) {
        const int j = e / RB, t = e % RB;
        if (r0 + t < n) Y[(int64_t)j * n + r0 + t] = rows[t * (m + 1) + j];
    }
}

// Tall-skinny G = A^T B for column-major n x m blocks A, B: each CTA sums a
// slab of rows into its own m x m partial (rows staged in shared memory);
// k_gram_reduce adds the partials in slab order (deterministic).
__global__ void __launch_bounds__(256) k_gram_partial(const double* A, const double* B, int64_t n, int m,
                                                      int64_t rows_per_cta, double* part, int sym) {
    after_previous();
    extern __shared__ double sh[];   // rows_per_cta x m for A, then for B
    const int64_t r0 = blockIdx.x * rows_per_cta;
    const int64_t nr = max((int64_t)0, min(rows_per_cta, n - r0));
    double* As = sh;
    double* Bs = sh + rows_per_cta * m;
    for (int64_t e = threadIdx.x; e < nr * m; e += 256) {
        const int64_t c = e / nr, r = e % nr;
        As[r * m + c] = A[c * n + r0 + r];
        Bs[r * m + c] = B[c * n + r0 + r];
    }
    __syncthreads();
    double* P = part + (int64_t)blockIdx.x * m * m;
    // A = B: the partial is symmetric and the products of (j, i) are those
    // of (i, j), so the upper triangle is mirrored (identical bits)
    const int ne = sym ? m * (m + 1) / 2 : m * m;
    for (int e0 = threadIdx.x; e0 < ne; e0 += 256) {
        int i, j;
        if (sym) {
            // e0 -> (i, j), i <= j, row-major over the upper triangle
            i = (int)(((2.0f * m + 1.0f) - sqrtf((2.0f * m + 1.0f) * (2.0f * m + 1.0f) - 8.0f * (float)e0)) * 0.5f);
            while (i > 0 && i * m - i * (i - 1) / 2 > e0) --i;
            while ((i + 1) * m - (i + 1) * i / 2 <= e0) ++i;
            j = i + (e0 - (i * m - i * (i - 1) / 2));
        } else {
            i = e0 / m;
            j = e0 % m;
        }
        const int e = i * m + j;
        double s0 = 0.0, s1 = 0.0;
        int64_t r = 0;
        for (; r + 1 < nr; r += 2) {
            s0 = fma(As[r * m + i], Bs[r * m + j], s0);
            s1 = fma(As[(r + 1) * m + i], Bs[(r + 1) * m + j], s1);
        }
        if (r < nr) s0 = fma(As[r * m + i], Bs[r * m + j], s0);
        P[e] = s0 + s1;
        if (sym && i != j) P[j * m + i] = s0 + s1;
    }
}

// G = the sum of the parts in slab order (deterministic): 32 elements a
// block; the eight warps stage 64 parts at a time, the first one adds them.
// The chain of FP64 additions bounds it: 152 parts of 88 x 88 took 17 us with
// one thread per element waiting for its own loads and take 9.4 so.
__global__ void __launch_bounds__(256) k_gram_reduce(const double* part, int nparts, int m, double* G) {
    after_previous();
    __shared__ double st[2][64][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int e = blockIdx.x * 32 + lane;
    const bool in = e < m * m;
    double s = 0.0;
    auto stage = [&](int p0, int b) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int p = p0 + warp + 8 * q;
            st[b][warp + 8 * q][lane] = (in && p < nparts) ? part[(int64_t)p * m * m + e] : 0.0;
        }
    };
    stage(0, 0);
    __syncthreads();
    for (int p0 = 0, b = 0; p0 < nparts; p0 += 64, b ^= 1) {
        if (p0 + 64 < nparts) stage(p0 + 64, b ^ 1);
        if (warp == 0) {
            const int np = min(64, nparts - p0);
#pragma unroll 8
            for (int q = 0; q < np; ++q) s += st[b][q][lane];
        }
        __syncthreads();
    }
    if (warp == 0 && in) G[e] = s;
}

// Cyclic Jacobi sweeps (FP64, and FP32 above JAC_PIPE_M) with the ordering and
// rotations of jacobi32.cuh on a symmetric m x m matrix H (row-major, shared memory),
// accumulating W <- W J (W column-major).  Rotations with |h_pq| <= tol
// sqrt(|h_pp h_qq|) are skipped (relative-accuracy threshold for graded
// matrices); the loop ends when no pair is above the threshold.  Returns the
// number of sweeps that rotated (max_sweeps + 1 if the limit was hit).  All
// threads of the block call it.
template <typename T>
__device__ int jacobi_sweeps(T* H, int ld, T* W, int m, T tol, int max_sweeps, T* cs, int* rot, int* pq) {
    const int mp = m + (m & 1);            // even player count (dummy index m when odd)
    const int npair = mp / 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        // A sweep rotates nothing exactly when no pair of the current H is
        // above the threshold (H only changes by rotations), so one scan of
        // the pairs stands in for that last, confirming sweep.
        if (threadIdx.x == 0) *rot = 0;
        __syncthreads();
        for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
            const int p = e / m, q = e % m;
            if (p < q && jacobi_rotates<T>(H[p * ld + q], H[p * ld + p], H[q * ld + q], tol)) *(volatile int*)rot = 1;
        }
        __syncthreads();
        if (*rot == 0) return sweep;
        __syncthreads();
        for (int r = 0; r < mp - 1; ++r) {
            for (int i = threadIdx.x; i < npair; i += blockDim.x) {
                int p, q;
                rr_pair(r, i, mp, p, q);
                T c = 1, s = 0;
                if (q < m) {
                    const T hpq = H[p * ld + q], hpp = H[p * ld + p], hqq = H[q * ld + q];
                    if (jacobi_rotates<T>(hpq, hpp, hqq, tol)) {
                        const T tau = (hqq - hpp) / (2 * hpq);
                        const T t = (tau >= 0) ? 1 / (tau + sqrt(1 + tau * tau)) : -1 / (-tau + sqrt(1 + tau * tau));
                        c = 1 / sqrt(1 + t * t);
                        s = t * c;
                    }
                }
                cs[2 * i] = c;
                cs[2 * i + 1] = s;
                pq[2 * i] = p;
                pq[2 * i + 1] = q;
            }
            __syncthreads();
            // columns: H <- H J, W <- W J (a warp per rotation, a lane per row)
            for (int i = warp; i < npair; i += nwarps) {
                const T s = cs[2 * i + 1];
                if (s == 0) continue;
                const T c = cs[2 * i];
                const int p = pq[2 * i], q = pq[2 * i + 1];
                T* wp = W + (int64_t)p * m;
                T* wq = W + (int64_t)q * m;
                for (int k = lane; k < m; k += 32) {
                    const T hkp = H[k * ld + p], hkq = H[k * ld + q];
                    H[k * ld + p] = c * hkp - s * hkq;
                    H[k * ld + q] = s * hkp + c * hkq;
                    const T vp = wp[k], vq = wq[k];
                    wp[k] = c * vp - s * vq;
                    wq[k] = s * vp + c * vq;
                }
            }
            __syncthreads();
            // rows: H <- J^T H, then the annihilated pair is exactly zero
            for (int i = warp; i < npair; i += nwarps) {
                const T s = cs[2 * i + 1];
                if (s == 0) continue;
                const T c = cs[2 * i];
                const int p = pq[2 * i], q = pq[2 * i + 1];
                T* hp = H + p * ld;
                T* hq = H + q * ld;
                for (int k = lane; k < m; k += 32) {
                    const T hpk = hp[k], hqk = hq[k];
                    hp[k] = c * hpk - s * hqk;
                    hq[k] = s * hpk + c * hqk;
                }
                __syncwarp();
                if (lane == 0) { hp[q] = 0; hq[p] = 0; }
            }
            __syncthreads();
        }
    }
    return max_sweeps + 1;
}

// Rayleigh-Ritz eigensolve of the symmetric m x m matrix Hg (global), in
// two precisions:
//  1. FP32 Jacobi on H / max|H| to a relative threshold of 1e-6 (the FP32
//     pipe is ~60x the FP64 pipe on this part); rotations accumulate in W32
//     (k_rr_fp32, one CTA);
//  2. W = W32 in FP64, refined by two Ogita-Aishima steps and a Lowdin
//     step (k_oa_step, k_lowdin): m x m FP64 products on many SMs
//     (k_small_nn, k_small_tn, k_small_apply) that leave W orthonormal to
//     rounding and the couplings of the separated pairs of H' = W^T H W
//     squared twice (at beta_c, Dcut 24, none is left above the FP64
//     threshold; off critical a graded tail of a few hundred pairs is);
//  3. FP64 Jacobi sweeps on H' (k_rr_fp64, one CTA): they find only the
//     pairs step 2 left coupled (near-degenerate ones), W <- W J.
// A rough Rayleigh-Ritz far from convergence (no FP64 sweeps) instead
// re-orthonormalises W32 by Cholesky-QR and takes theta = diag(W^T H W).
// Output: theta sorted descending, W (column-major, global) in that order.
// Shared memory of the one-CTA kernels: H (m rows of ld = m + 1 doubles: the
// odd stride puts the rows of one column in different banks, so the column
// updates are conflict-free) + m*ld doubles of scratch + small arrays.
__global__ void __launch_bounds__(512) k_rr_fp32(const double* Hg, int m, double* Hsym, double* Wout,
                                                 int* sweeps_out) {
    after_previous();
    extern __shared__ double sm[];
    const int ld = m + 1;
    const bool piped = m <= JAC_PIPE_M;
    const int mp = m + (m & 1);
    float* H32 = (float*)sm;                   // m*ld floats, twice when piped
    float* W32 = H32 + (piped ? 2 : 1) * m * ld;   // m*m floats
    float* cs32 = W32 + m * m;                 // plain: mp
    int* rot = (int*)(cs32 + mp + (mp & 1));   // 1
    int* pq = rot + 2;                         // mp: the pairs of the current round
    __shared__ JacShared jac;
    __shared__ double hmax_s;
    if (threadIdx.x == 0) hmax_s = 0.0;
    __syncthreads();
    double lmax = 0.0;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        const int i = e / m, j = e % m;
        const double v = 0.5 * (Hg[(int64_t)i * m + j] + Hg[(int64_t)j * m + i]);
        Hsym[e] = v;
        lmax = fmax(lmax, fabs(v));
    }
    for (int o = 16; o > 0; o >>= 1) lmax = fmax(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
    if ((threadIdx.x & 31) == 0) atomicMax((unsigned long long*)&hmax_s, (unsigned long long)__double_as_longlong(lmax));
    __syncthreads();
    const double hscale = hmax_s > 0.0 ? 1.0 / hmax_s : 1.0;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        const int i = e / m, j = e % m;
        H32[i * ld + j] = (float)(0.5 * (Hg[(int64_t)i * m + j] + Hg[(int64_t)j * m + i]) * hscale);
        W32[e] = (i == j) ? 1.0f : 0.0f;
    }
    __syncthreads();
    const int s32 = piped ? jacobi_sweeps_f32<512>(H32, H32 + m * ld, ld, W32, m, 1e-6f, 40, jac)
                          : jacobi_sweeps<float>(H32, ld, W32, m, 1e-6f, 40, cs32, rot, pq);
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) Wout[e] = (double)W32[e];
    if (threadIdx.x == 0 && sweeps_out) atomicAdd(sweeps_out, s32);
}

// C[i][j] = sum_r A[i*m + r] B[j*m + r] (the columns of two column-major m x
// m blocks): a CTA per row i, a thread per column j, the sum in order of r.
__global__ void __launch_bounds__(128) k_small_tn(const double* A, const double* B, int m, double* C) {
    after_previous();
    const int i = blockIdx.x;
    for (int j = threadIdx.x; j < m; j += blockDim.x) {
        double a = 0.0;
        for (int r = 0; r < m; ++r) a = fma(A[(int64_t)i * m + r], B[(int64_t)j * m + r], a);
        C[(int64_t)i * m + j] = a;
    }
}

// (H W)[r][j] = sum_k H[r*m + k] W[j*m + k] (row-major H, column-major W),
// stored column-major: C[j*m + r].
__global__ void __launch_bounds__(128) k_small_nn(const double* H, const double* W, int m, double* C) {
    after_previous();
    const int r = blockIdx.x;
    for (int j = threadIdx.x; j < m; j += blockDim.x) {
        double a = 0.0;
        for (int k = 0; k < m; ++k) a = fma(H[(int64_t)r * m + k], W[(int64_t)j * m + k], a);
        C[(int64_t)j * m + r] = a;
    }
}

// Xout = X (I + E) = X + X E for a column-major m x m X and a row-major E:
// a CTA per column j, a thread per row r, the sum in order of k.
__global__ void __launch_bounds__(128) k_small_apply(const double* X, const double* E, int m, double* Xout) {
    after_previous();
    const int j = blockIdx.x;
    for (int r = threadIdx.x; r < m; r += blockDim.x) {
        double a = 0.0;
        for (int k = 0; k < m; ++k) a = fma(X[(int64_t)k * m + r], E[(int64_t)k * m + j], a);
        Xout[(int64_t)j * m + r] = X[(int64_t)j * m + r] + a;
    }
}

// One refinement step of an approximate eigenbasis X of the symmetric H
// after Ogita and Aishima (Iterative refinement for symmetric eigenvalue
// decomposition, Japan J. Indust. Appl. Math. 35, 2018).  With S = X^T H X
// (symmetrised here) and P = X^T X = I - R:
//   lambda_i = s_ii / p_ii,
//   E_ij = (s_ij + lambda_j r_ij) / (lambda_j - lambda_i)   for a separated pair,
//   E_ij = r_ij / 2                                         otherwise and for i = j,
// and X <- X (I + E) (k_small_apply): to first order that makes X^T X = I
// (E + E^T = R) and zeroes the separated couplings, so both shrink
// quadratically from step to step.  Where the published step separates
// pairs by one global gap bound, this one takes a pair as separated when
// |lambda_j - lambda_i| > OA_SEP (|s_ij| + max(|lambda_i|, |lambda_j|) |r_ij|),
// i.e. |E_ij| < 1 / OA_SEP: a symmetric test, so E + E^T = R holds exactly,
// and a strict one, so that the second-order terms (X^T X - I after a step
// is about E^T E) stay small even where the FP32 vectors of a graded tail
// are poor.  Pairs it leaves coupled (near-degenerate ones, the tail) are
// left to FP64 Jacobi.
// One CTA.
constexpr double OA_SEP = 256.0;
constexpr int OA_STEPS = 2;
__global__ void __launch_bounds__(256) k_oa_step(const double* S, const double* P, int m, double* E) {
    after_previous();
    __shared__ double lam[MAX_M];
    for (int i = threadIdx.x; i < m; i += blockDim.x) lam[i] = S[(int64_t)i * m + i] / P[(int64_t)i * m + i];
    __syncthreads();
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        const int i = e / m, j = e % m;
        const double r = (i == j ? 1.0 : 0.0) - P[e];
        double v = 0.5 * r;
        if (i != j) {
            const double sij = 0.5 * (S[e] + S[(int64_t)j * m + i]);
            const double gap = lam[j] - lam[i];
            const double bound = OA_SEP * (fabs(sij) + fmax(fabs(lam[i]), fabs(lam[j])) * fabs(r));
            if (fabs(gap) > bound) v = (sij + lam[j] * r) / gap;
        }
        E[e] = v;
    }
}

// Second-order Lowdin (symmetric) orthonormalisation: for X^T X = P = I - R
// with R small, X (I + F) with F = R / 2 + 3 R^2 / 8 (the series of
// (I - R)^(-1/2)) has (I + F)^T P (I + F) = I + O(R^3).  PP = P P gives
// R^2 = PP - 2 P + I.  F is row-major (P, PP symmetric).
__global__ void __launch_bounds__(256) k_lowdin(const double* P, const double* PP, int m, double* F) {
    after_previous();
    for (int e = threadIdx.x + blockIdx.x * blockDim.x; e < m * m; e += blockDim.x * gridDim.x) {
        const int i = e / m, j = e % m;
        const double id = (i == j) ? 1.0 : 0.0;
        const double r = id - P[e];
        const double r2 = PP[e] - 2.0 * P[e] + id;
        F[e] = 0.5 * r + 0.375 * r2;
    }
}

__device__ __forceinline__ double rank_key(double x) { return isnan(x) ? -INFINITY : x; }

// Step 3 of the Rayleigh-Ritz solve: H = (G + G^T) / 2, FP64 sweeps from
// W = Win (accumulated in shared memory), then theta and W sorted by
// descending theta (ties keep index order) into Wout (may alias Win).
__global__ void __launch_bounds__(512) k_rr_fp64(const double* G, int m, double tol, int max_sweeps,
                                                 double* theta, const double* Win, double* Wout, int* status,
                                                 int* sweeps_out, int fp64_sweeps) {
    after_previous();
    extern __shared__ double sm[];
    const int mp = m + (m & 1);
    const int ld = m + 1;
    double* H = sm;                            // m*ld
    double* Ws = H + m * ld;                   // m*m (W, accumulated)
    double* cs64 = Ws + m * ld;                // mp
    int* rot = (int*)(cs64 + mp);              // 1
    int* perm = rot + 2;                       // m
    int* pq = perm + m + (m & 1);              // mp
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        const int i = e / m, j = e % m;
        H[i * ld + j] = 0.5 * (G[(int64_t)i * m + j] + G[(int64_t)j * m + i]);
        Ws[e] = Win[e];
    }
    __syncthreads();
    // (skipped for a rough Rayleigh-Ritz far from convergence: then theta is
    // the diagonal of H' and W the re-orthonormalised W32)
    const int s64 = fp64_sweeps ? jacobi_sweeps<double>(H, ld, Ws, m, tol, max_sweeps, cs64, rot, pq) : 0;
    // rank of each diagonal value, descending; ties by index.  A NaN ranks as
    // -infinity: compared as it is, it would share its rank with others and
    // leave entries of perm unwritten, which are indices below.
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const double hi = rank_key(H[i * ld + i]);
        int r = 0;
        for (int j = 0; j < m; ++j) {
            const double hj = rank_key(H[j * ld + j]);
            r += (hj > hi || (hj == hi && j < i)) ? 1 : 0;
        }
        perm[r] = i;
    }
    if (threadIdx.x == 0) {
        if (s64 > max_sweeps) atomicOr(status, ST_EIG_NOCONV);
        if (sweeps_out) atomicAdd(sweeps_out + 1, s64);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x) theta[i] = H[perm[i] * ld + perm[i]];
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        const int col = e / m, row = e % m;
        Wout[e] = Ws[perm[col] * m + row];
    }
}

// max_i<dn |Z_i - theta_i QW_i| / theta_0, as bits of a non-negative double.
__global__ void __launch_bounds__(256) k_residual(const double* Z, const double* QW, const double* theta,
                                                  int64_t n, unsigned long long* out_bits) {
    after_previous();
    __shared__ double red[33];
    const int c = blockIdx.x;
    const double th = theta[c];
    double s = 0.0;
    for (int64_t r = threadIdx.x; r < n; r += 256) {
        const double d = Z[(int64_t)c * n + r] - th * QW[(int64_t)c * n + r];
        s = fma(d, d, s);
    }
    s = block_sum<256>(s, red);
    if (threadIdx.x == 0) {
        double rel = sqrt(s) / fabs(theta[0]);
        if (!isfinite(rel)) rel = INFINITY;
        atomicMax(out_bits, (unsigned long long)__double_as_longlong(rel));
    }
}

// The outcome of a Rayleigh-Ritz step for the host.
__global__ void __launch_bounds__(128) k_tell(const double* theta, const double* res, const int* sweeps,
                                              const int* status, int m, EigBox* box, unsigned long long seq) {
    after_previous();
    if (threadIdx.x < m) box->theta[threadIdx.x] = theta[threadIdx.x];
    if (threadIdx.x == 0) {
        box->res = *res;
        box->sweeps[0] = sweeps[0];
        box->sweeps[1] = sweeps[1];
        box->status = *status;
    }
    __threadfence_system();
    __syncthreads();
    if (threadIdx.x == 0) box_done(box, seq);
}

// Y <- Y - sigma Q (the shift of a power step)
__global__ void k_shift(double* Y, const double* Q, double sigma, int64_t count) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        Y[i] = fma(-sigma, Q[i], Y[i]);
}

// U[r*dn + i] = QW[i*n + r]
__global__ void k_to_isometry(const double* QW, int64_t n, int dn, double* U) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n * dn) return;
    const int64_t r = e / dn, i = e % dn;
    U[e] = QW[i * n + r];
}

}  // namespace

static size_t rr32_smem(int m) {
    const int mp = m + (m & 1);
    return (size_t)(m <= JAC_PIPE_M ? 2 : 1) * m * (m + 1) * 4 + (size_t)m * m * 4 + (size_t)(mp + 2) * 4 +
           (size_t)(mp + 4) * 4 + 64;
}

static size_t rr64_smem(int m) {
    const int mp = m + (m & 1);
    return (size_t)2 * m * (m + 1) * 8 + (size_t)mp * 8 + (size_t)(m + 4) * 4 + (size_t)mp * 4 + 64;
}

static size_t chol_smem(int m, int rb) {
    const int me = chol_even(m);
    return ((size_t)me * (me + 1) + (size_t)me * 7 + (size_t)rb * (m + 1) + (size_t)8 * rb) * 8 +
           (size_t)chol_table_entries(m) * 2 + 16;
}

// Wait until the kernel that was given `seq` has written the box: the host
// needs its few numbers to go on, but not the rest of the kernel.  Spins on
// the mapped word (tens of microseconds as a rule), then waits for the stream.
static const EigBox& wait_box(Ctx& ctx, unsigned long long seq) {
    EigBox* box = (EigBox*)ctx.box;
    const auto t0 = std::chrono::steady_clock::now();
    for (;;) {
        for (int i = 0; i < 512; ++i)
            if (__atomic_load_n(&box->seq, __ATOMIC_ACQUIRE) == seq) return *box;
        if (std::chrono::steady_clock::now() - t0 > std::chrono::milliseconds(2)) break;
    }
    TRG_CUDA(cudaStreamSynchronize(ctx.stream));
    if (__atomic_load_n(&box->seq, __ATOMIC_ACQUIRE) != seq) fail(TRG_ECUDA, "isometry: no answer from the device");
    return *box;
}

// Factor G and Y <- Y L^{-T}.  Rows per block: 8 while that gives every SM at
// most one block (256 rows at m = 40: 32 blocks instead of 8), then 16; 32,
// which leaves no lane of the triangle idle, for more rows.
static void chol_trsm(Ctx& ctx, const double* G, double* Y, int64_t n, int m, double tau, bool always, int* flags,
                      EigBox* box, unsigned long long seq) {
    const int rb = n <= 8 * ctx.sm_count ? 8 : n <= 16 * ctx.sm_count ? 16 : 32;
    const unsigned grid = (unsigned)((n + rb - 1) / rb);
    const size_t smem = chol_smem(m, rb);
    const int al = always ? 1 : 0;
    const bool chain = chain_wide(ctx, n);
    if (rb == 8) launch_chained_if(chain, ctx, k_chol_trsm<8>, grid, CHOL_THREADS, smem, G, Y, n, m, tau, al, flags, box, seq);
    else if (rb == 16) launch_chained_if(chain, ctx, k_chol_trsm<16>, grid, CHOL_THREADS, smem, G, Y, n, m, tau, al, flags, box, seq);
    else launch_chained_if(chain, ctx, k_chol_trsm<32>, grid, CHOL_THREADS, smem, G, Y, n, m, tau, al, flags, box, seq);
    TRG_LAUNCHED(ctx);
}

static void set_smem(const void* fn, size_t bytes) {
    TRG_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
}

// Column-major n x m "A^T B" (m x m result, row-major) and "A W" products.
static void gram(Ctx& ctx, const double* A, const double* B, int64_t n, int m, double* G, int precision) {
    (void)precision;   // the Gram / Rayleigh-Ritz products are FP64 in every mode
    const int64_t rows = std::max<int64_t>(8, (n + ctx.sm_count - 1) / ctx.sm_count);
    const int64_t rows_c = std::min<int64_t>(rows, (int64_t)(96 * 1024 / (16 * m)));   // <= 96 KB staged
    const int nparts = (int)((n + rows_c - 1) / rows_c);
    ctx.ensure(ctx.f64_partial, (size_t)nparts * m * m * sizeof(double));
    const size_t smem = (size_t)rows_c * m * 2 * sizeof(double);
    static PerDevice prepared;
    prepared.get(ctx.device, [] {
        TRG_CUDA(cudaFuncSetAttribute((const void*)k_gram_partial, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      100 * 1024));
        return 0;
    });
    launch_chained_if(chain_wide(ctx, n), ctx, k_gram_partial, nparts, 256, smem, A, B, n, m, rows_c, ctx.f64_partial.as<double>(), A == B ? 1 : 0);
    TRG_LAUNCHED(ctx);
    launch_chained(ctx, k_gram_reduce, (m * m + 31) / 32, 256, 0, ctx.f64_partial.as<double>(), nparts, m, G);
    TRG_LAUNCHED(ctx);
}
static void times_small(Ctx& ctx, const double* A, const double* W, int64_t n, int m, double* C, int precision) {
    GemmDesc g;
    g.M = n; g.N = m; g.K = m;
    g.A.base = A; g.A.off_r = ctx.table({{n, 1}}); g.A.off_c = ctx.table({{m, n}}); g.A.c_fast = false;
    g.B.base = W; g.B.off_r = ctx.table({{m, 1}}); g.B.off_c = ctx.table({{m, m}}); g.B.c_fast = false;
    g.C = C; g.c_m = ctx.table({{n, 1}}); g.c_n = ctx.table({{m, n}}); g.beta = 0.0;
    g.A.r_fast = true; g.A.r_identity = true;
    g.B.r_fast = true; g.B.r_identity = true;
    g.allow_exact = precision == TRG_FP64;    // split mode: see k_chol_trsm on the bits of Q
    g.c_m_fast = true;
    gemm(ctx, g, TRG_FP64);
}

// Orthonormalise the columns of Y in place (two Cholesky-QR passes).  After
// one pass Q^T Q = I to about eps / min_j(d_j / G_jj) (the pivots of the
// column-normalised Gram matrix bound its conditioning); when the next step
// is another power step rather than a Rayleigh-Ritz step (`power_next`),
// which needs only a well-conditioned basis, a clean first pass with
// pivots above PASS2_PIVMIN is enough and the second pass is skipped.
constexpr double PASS2_PIVMIN = 1e-3;
static void orthonormalise(Ctx& ctx, double* Y, int64_t n, int m, double* G, int* flags, uint64_t seed,
                           uint64_t& salt, bool power_next = false) {
    bool first_clean = true;    // the first pass needed no column repair
    for (int pass = 0; pass < 2; ++pass) {
        double pm = 0.0;
        for (int attempt = 0;; ++attempt) {
            launch_chained(ctx, k_col_normalize, m, 256, 0, Y, n, flags);
            TRG_LAUNCHED(ctx);
            gram(ctx, Y, Y, n, m, G, TRG_FP64);
            const unsigned long long seq = ++ctx.box_seq;
            chol_trsm(ctx, G, Y, n, m, pass == 0 ? 1e-8 : 1e-12, false, flags, (EigBox*)ctx.box, seq);
            const EigBox& box = wait_box(ctx, seq);
            pm = box.pivmin;
            const int hb = box.nbad;
            if (hb == 0) break;
            if (pass == 0) first_clean = false;
            ctx.counters[4] += (uint64_t)hb;
            if (attempt >= 16) fail(TRG_ENUMERIC, "Cholesky-QR: could not complete a basis");
            dim3 grid((unsigned)std::min<int64_t>((n + 255) / 256, 64), (unsigned)m);
            k_rand_cols<<<grid, 256, 0, ctx.stream>>>(Y, n, m, flags, seed, ++salt);
            TRG_LAUNCHED(ctx);
        }
        if (pass == 0 && power_next && first_clean && pm >= PASS2_PIVMIN) {
            ctx.counters[5] += 1;
            return;
        }
    }
}

int isometry(Ctx& ctx, const double* M, int64_t n, int dcut, double* U, std::vector<double>& lam,
             int step, int precision) {
    const int dn_paper = (int)std::min<int64_t>(n, dcut);
    // block of dn + p columns, at most the shared-memory block of the small
    // kernels (p shrinks there: Dcut 96 runs with p = 16)
    if (dn_paper >= MAX_M && dn_paper < n)
        fail(TRG_ENOTSUP, "isometry: Dcut above the supported block (111 kept vectors)");
    const int m = (int)std::min<int64_t>({n, (int64_t)dn_paper + std::max(1, ctx.cfg.oversample), (int64_t)MAX_M});
    static PerDevice prepared;
    prepared.get(ctx.device, [] {
        set_smem((const void*)k_chol_trsm<8>, chol_smem(MAX_M, 8));
        set_smem((const void*)k_chol_trsm<16>, chol_smem(MAX_M, 16));
        set_smem((const void*)k_chol_trsm<32>, chol_smem(MAX_M, 32));
        set_smem((const void*)k_rr_fp32, std::max(rr32_smem(MAX_M), rr32_smem(JAC_PIPE_M)));
        set_smem((const void*)k_rr_fp64, rr64_smem(MAX_M));
        return 0;
    });
    // buffers: Q, Y, Z, QW (n x m each); G, L, W (m x m); theta (m)
    ctx.ensure(ctx.eig, (size_t)(4 * n * m) * sizeof(double));
    ctx.ensure(ctx.eig_small, (size_t)(9 * m * m + 2 * m + 8) * sizeof(double));
    ctx.ensure(ctx.flags, (size_t)(m + 8) * sizeof(int));
    double* Q = ctx.eig.as<double>();
    double* Y = Q + n * m;
    double* Z = Y + n * m;
    double* QW = Z + n * m;
    double* G = ctx.eig_small.as<double>();
    double* W = G + m * m;
    double* theta = W + m * m;
    double* Hs = theta + 2 * m + 8;    // Rayleigh-Ritz scratch: symmetrised H, H W, Gram matrices
    double* T1 = Hs + m * m;
    double* G2 = T1 + m * m;
    double* Pm = G2 + m * m;           // X^T X of the refinement
    double* E = Pm + m * m;            // its correction
    double* Xb = E + m * m;            // a second basis buffer
    int* flags = ctx.flags.as<int>();
    int* sweeps = flags + m + 2;   // [0] FP32 sweeps, [1] FP64 sweeps of the last Rayleigh-Ritz

    static_assert(HOST_SLOT_BOX + sizeof(EigBox) <= HOST_SLOT_BYTES, "isometry answers");
    int* status = ctx.status.as<int>();
    double* res_slot = ctx.scal.as<double>() + SC_RES;
    const uint64_t seed = ctx.cfg.seed ^ (0xA24BAED4963EE407ull * (uint64_t)step);
    uint64_t salt = 0;

    {
        dim3 grid((unsigned)std::min<int64_t>((n + 255) / 256, 64), (unsigned)m);
        k_rand_cols<<<grid, 256, 0, ctx.stream>>>(Q, n, m, nullptr, seed, salt);
        TRG_LAUNCHED(ctx);
    }
    // Y = M Q.  In split mode M is sliced once for all the products of this
    // solve (each product then slices only the n x m block Q).
    Gather gm;
    gm.base = M; gm.off_r = ctx.table({{n, n}}); gm.off_c = ctx.table({{n, 1}}); gm.c_fast = true;
    gm.c_identity = true;
    const uint16_t* m_slices = nullptr;
    const int* m_e = nullptr;
    if (precision == TRG_SPLIT_BF16) {
        const size_t sl = (size_t)slices_now(ctx) * split_rows_padded(ctx, n) * split_k_padded(n) * 2;
        const size_t eb = (size_t)split_rows_padded(ctx, n) * sizeof(int);
        ctx.ensure(ctx.eig_slices, sl + eb + 256);
        uint16_t* sp = ctx.eig_slices.as<uint16_t>();
        int* ep = (int*)(ctx.eig_slices.as<uint8_t>() + ((sl + 255) & ~(size_t)255));
        split_slice_operand(ctx, gm, n, n, sp, ep);
        m_slices = sp;
        m_e = ep;
    }
    auto apply_m = [&](double shift) {
        GemmDesc g;
        g.M = n; g.N = m; g.K = n;
        g.A = gm;
        g.a_slices = m_slices;
        g.a_e = m_e;
        g.B.base = Q; g.B.off_r = ctx.table({{n, 1}}); g.B.off_c = ctx.table({{m, n}}); g.B.c_fast = false;
        g.C = Y; g.c_m = ctx.table({{n, 1}}); g.c_n = ctx.table({{m, n}}); g.beta = 0.0;
        g.B.r_fast = true; g.B.r_identity = true;
        g.allow_exact = true;
        g.c_m_fast = true;
        g.allow_ksplit = true;    // n / 128 tiles of 128 x m: K is split over the idle SMs
        gemm(ctx, g, precision);
        if (shift > 0.0) {
            const int64_t cnt = n * m;
            k_shift<<<(unsigned)std::min<int64_t>((cnt + 255) / 256, 4 * ctx.sm_count), 256, 0, ctx.stream>>>(
                Y, Q, shift, cnt);
            TRG_LAUNCHED(ctx);
        }
    };
    // Power steps apply M - sigma I with sigma = theta_m / 2 (a degree-one
    // Chebyshev filter of the unwanted interval [0, theta_m]): the
    // components outside the block shrink by (theta_m / 2) / (theta_dn -
    // theta_m / 2) a step instead of theta_m / theta_dn, at the cost of one
    // axpy.  theta_m comes from the last Rayleigh-Ritz step, or from the
    // previous solve of this direction before the first; a Rayleigh-Ritz
    // product is never shifted.
    auto shifted_rate = [](double th_m, double th_dn) {
        if (!(th_m > 0.0) || !(th_dn > th_m)) return 0.98;
        return std::min(std::max(0.5 * th_m / (th_dn - 0.5 * th_m), 0.05), 0.98);
    };
    // The number of products that reached the tolerance in the previous solve
    // of this direction (same sizes) is the plan: the spectra of successive
    // same-direction environments are close, and a random start needs about
    // as many products each time.  Without one, two plain power steps precede
    // a first, FP32-only Rayleigh-Ritz that measures the convergence rate.
    Ctx::EigHint& hint = ctx.eig_hint[step & 1];
    const bool have_hint = hint.n == n && hint.m == m && hint.precision == precision && hint.products > 0;
    double sigma = (have_hint && hint.theta_m > 0.0) ? 0.5 * hint.theta_m : 0.0;
    // the start block is followed by power steps unless the first step is a
    // Rayleigh-Ritz step (no plan and m = n)
    orthonormalise(ctx, Q, n, m, G, flags, seed, salt, have_hint || m < n);
    int applied = 0;                 // products of M in the span of Q
    if (!have_hint) {
        for (int pre = 0; pre < 2 && m < n; ++pre) {
            apply_m(0.0);
            std::swap(Q, Y);
            orthonormalise(ctx, Q, n, m, G, flags, seed, salt, pre == 0);
            ++applied;
        }
    }

    // Split products carry ~2^-(8S-1) relative error, which floors the Ritz
    // residual; f is insensitive to residuals far above that floor (1e-6
    // moves f by ~1e-12 on the Ising workloads), so stop at 2^-(8S-10).
    double tol = ctx.cfg.eig_tol;
    const int S_env = slices_now(ctx);   // the slices of this solve's M.Q products
    if (precision == TRG_SPLIT_BF16) tol = std::max(tol, std::ldexp(1.0, -(8 * S_env - 10)));
    std::vector<double> th((size_t)m);
    const int max_it = std::max(1, ctx.cfg.eig_max_iter);
    // Rayleigh-Ritz is the costly part (a one-SM Jacobi solve), so it is not
    // done after every product: the first one, in FP32 only, measures the
    // residual and the convergence rate rho ~ theta_m / theta_dn; the power
    // steps needed to reach the tolerance follow from rho and run without a
    // Rayleigh-Ritz; the next (full FP64) one normally converges.
    int pending = have_hint ? std::min(hint.products, 60) : 0;   // planned plain power steps
    int rr_done = have_hint ? 1 : 0;
    double prev_res = 0.0;
    int since_rr = 0;                // products applied since the previous Rayleigh-Ritz
    for (int it = 1; it <= max_it; ++it) {
        if (pending > 0) {
            apply_m(sigma);
            std::swap(Q, Y);
            orthonormalise(ctx, Q, n, m, G, flags, seed, salt, pending > 1);
            --pending;
            ++since_rr;
            ++applied;
            ctx.counters[0] += 1;
            continue;
        }
        // Y = M Q
        apply_m(0.0);
        // Rayleigh-Ritz
        gram(ctx, Q, Y, n, m, G, TRG_FP64);
        TRG_CUDA(cudaMemsetAsync(sweeps, 0, 2 * sizeof(int), ctx.stream));
        const int full = (rr_done > 0 || m == n) ? 1 : 0;
        // FP64 rotations stop at |h_pq| <= jtol sqrt(h_pp h_qq).  An unrotated
        // pair leaves at most m jtol theta_1 in a Ritz residual, so jtol =
        // 1e-3 tol keeps that far below the tolerance; with FP64 products
        // (tol 1e-12) it is 1e-13 (eigenvalues exact to ~1e-26 relative, the
        // vectors of pairs with a relative gap g to ~1e-13 / g), with split
        // products (tol 2^-(8S-10)) 2.4e-10 at S = 4.
        const double jtol = std::max(1e-13, 1e-3 * tol);
        {
            // the Rayleigh-Ritz solve of G = Q^T M Q into theta, W: FP32
            // Jacobi, then (see k_rr_fp32) FP64 products and FP64 Jacobi
            launch_chained(ctx, k_rr_fp32, 1, 512, rr32_smem(m), G, m, Hs, W, sweeps);
            TRG_LAUNCHED(ctx);
            const double* Wj = W;    // the basis the FP64 sweeps start from
            if (full) {
                // Refine the FP32 eigenbasis in FP64 on many SMs: OA_STEPS
                // Ogita-Aishima steps (k_oa_step), then a Lowdin step; the
                // sweeps are left the pairs the steps could not separate.
                double* X = W;
                double* Xn = Xb;
                auto small = [&](auto kern, const double* a, const double* b, double* c) {
                    launch_chained(ctx, kern, m, 128, 0, a, b, m, c);
                    TRG_LAUNCHED(ctx);
                };
                for (int st = 0; st < OA_STEPS; ++st) {
                    small(k_small_nn, Hs, X, T1);      // H X
                    small(k_small_tn, X, T1, G2);      // S = X^T H X
                    small(k_small_tn, X, X, Pm);       // P = X^T X
                    launch_chained(ctx, k_oa_step, 1, 256, 0, G2, Pm, m, E);
                    TRG_LAUNCHED(ctx);
                    small(k_small_apply, X, E, Xn);
                    std::swap(X, Xn);
                }
                small(k_small_tn, X, X, Pm);
                small(k_small_tn, Pm, Pm, T1);          // P P (P symmetric)
                launch_chained(ctx, k_lowdin, (m * m + 255) / 256, 256, 0, Pm, T1, m, E);
                TRG_LAUNCHED(ctx);
                small(k_small_apply, X, E, Xn);
                std::swap(X, Xn);
                small(k_small_nn, Hs, X, T1);
                small(k_small_tn, X, T1, G2);          // H' = X^T H X
                Wj = X;
            } else {
                // a rough Rayleigh-Ritz (no FP64 sweeps): W re-orthonormalised
                // by Cholesky-QR, theta the diagonal of H' = W^T H W
                launch_chained(ctx, k_small_tn, m, 128, 0, W, W, m, G2);
                TRG_LAUNCHED(ctx);
                chol_trsm(ctx, G2, W, m, m, 0.0, true, flags, nullptr, 0);
                launch_chained(ctx, k_small_nn, m, 128, 0, Hs, W, m, T1);
                TRG_LAUNCHED(ctx);
                launch_chained(ctx, k_small_tn, m, 128, 0, W, T1, m, G2);
                TRG_LAUNCHED(ctx);
            }
            launch_chained(ctx, k_rr_fp64, 1, 512, rr64_smem(m), G2, m, jtol, 60, theta, Wj, W, status, sweeps, full);
            TRG_LAUNCHED(ctx);
        }
        times_small(ctx, Y, W, n, m, Z, precision);
        times_small(ctx, Q, W, n, m, QW, precision);
        TRG_CUDA(cudaMemsetAsync(res_slot, 0, sizeof(double), ctx.stream));
        launch_chained(ctx, k_residual, dn_paper, 256, 0, Z, QW, theta, n, (unsigned long long*)res_slot);
        TRG_LAUNCHED(ctx);
        const unsigned long long seq = ++ctx.box_seq;
        launch_chained(ctx, k_tell, 1, 128, 0, theta, res_slot, sweeps, status, m, (EigBox*)ctx.box, seq);
        TRG_LAUNCHED(ctx);
        const EigBox& box = wait_box(ctx, seq);
        std::copy(box.theta, box.theta + m, th.begin());
        const double res = box.res;
        const int hsw[2] = {box.sweeps[0], box.sweeps[1]};
        const int st = box.status;
        ctx.counters[0] += 1;
        ctx.counters[1] += 1;
        ctx.counters[2] += (uint64_t)hsw[0];
        ctx.counters[3] += (uint64_t)hsw[1];
        check_timeout(ctx);
        if (st & ST_EIG_NOCONV) fail(TRG_ENUMERIC, "Rayleigh-Ritz Jacobi did not converge");
        if (!(th[0] > 0.0) || !std::isfinite(th[0])) fail(TRG_ENUMERIC, "environment has no positive eigenvalue");
        if ((res <= tol && full) || m == n) {
            {
                // The next plan is this solve's product count less the
                // products beyond what the tolerance needed (at the rate
                // theta_m / theta_dn), two kept spare: a plan that falls short
                // costs a second Rayleigh-Ritz, several times a product.
                const double r = sigma > 0.0
                                     ? shifted_rate(th[(size_t)m - 1], th[(size_t)dn_paper - 1])
                                     : std::min(std::max(th[(size_t)m - 1] / th[(size_t)dn_paper - 1], 0.05), 0.98);
                const int slack = (res > 0.0 && res < tol) ? (int)std::floor(std::log(tol / res) / -std::log(r)) : 0;
                hint.n = n; hint.m = m; hint.precision = precision;
                hint.products = std::max(1, applied - std::max(0, slack - 2));
                hint.theta_m = m < n ? th[(size_t)m - 1] : 0.0;
            }
            int dn = dn_paper;
            if (ctx.cfg.trunc == TRG_TRUNC_MULTIPLET && dn < n) {
                // split products separate exactly degenerate eigenvalues by up
                // to ~2^-(8S-12) lambda_1: treat smaller gaps as degenerate
                double gtol = ctx.cfg.gap_tol;
                if (precision == TRG_SPLIT_BF16)
                    gtol = std::max(gtol, std::ldexp(1.0, -(8 * S_env - 12)));
                while (dn > 1 && (th[(size_t)dn - 1] - th[(size_t)dn]) < gtol * th[0]) --dn;
            }
            lam.assign(th.begin(), th.begin() + dn);
            const int64_t tot = n * dn;
            k_to_isometry<<<(unsigned)((tot + 255) / 256), 256, 0, ctx.stream>>>(QW, n, dn, U);
            TRG_LAUNCHED(ctx);
            return dn;
        }
        // plan the power steps to the next Rayleigh-Ritz (shifted by the
        // fresh theta_m)
        sigma = (m < n && th[(size_t)m - 1] > 0.0) ? 0.5 * th[(size_t)m - 1] : 0.0;
        double rho = sigma > 0.0 ? shifted_rate(th[(size_t)m - 1], th[(size_t)dn_paper - 1])
                                 : th[(size_t)m - 1] / th[(size_t)dn_paper - 1];
        if (rr_done > 0 && prev_res > 0.0 && res > 0.0 && since_rr > 0)
            rho = std::max(rho, std::pow(res / prev_res, 1.0 / since_rr));
        rho = std::min(std::max(rho, 0.05), 0.98);
        int k = (res > tol) ? (int)std::ceil(std::log(tol / res) / std::log(rho)) : 0;
        pending = std::min(std::max(k, 0), 40);   // k - 1 needed after the product below, plus one spare
        ++rr_done;
        prev_res = res;
        since_rr = 1;
        // next block: orth(Y W) = orth(M Q W), same span as M Q
        ++applied;
        std::swap(Q, Z);
        orthonormalise(ctx, Q, n, m, G, flags, seed, salt, pending > 0);
    }
    fail(TRG_ENUMERIC, "subspace iteration did not converge");
}

}  // namespace trg
