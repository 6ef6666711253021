// Plain FP64 gathered GEMM on the CUDA cores (the TRG_FP64 precision mode).
//
// Every contraction of the HOTRG step (environment, U.T.T.U, M.Q products of
// the subspace iteration) is a matrix product once its multi-indices are
// flattened; offset tables do the flattening, so permuted and rotated views
// (the y half-step) cost nothing extra.
//
// What bounds it: the FP64 pipe, 1.9 FMA a clock and SM on this part.  One
// warp-wide FMA occupies an SM's pipe for 16 clocks, so shared-memory and L2
// operand traffic are free even at one output per thread, and the only thing
// that counts is that every SM has the same share of the FMAs.  The output
// tile T is therefore chosen by size (choose_shape): 64 x 64 for large
// products, down to 8 x 8 for the m-column blocks of the isometry, where
// 64 x 64 tiles left four SMs with all the work: 256 x 40 x 256 took 210 us
// on 64 x 64 tiles and takes 14 us on 8 x 8 ones, the three products of a
// (24, 22) environment 1623 us on 64 (81 tiles, both halves of the Gram
// products) and 651 us on 16.
// Operands of the next K stage are loaded to registers while the current one
// is multiplied; every output sums its products in order of k whatever the
// tile, so the tile changes no bit (split K does).
#include <algorithm>
#include <cmath>

#include "internal.h"

namespace trg {

namespace {

struct GemmArgs {
    int64_t M, N, K;
    int64_t kper;          // split-K: K range of blockIdx.z is [z*kper, min(K, (z+1)*kper))
    double* partial;       // split-K: dense M x N partial sums per z (else nullptr)
    const double* A; const int64_t* a_m; const int64_t* a_k; int a_kfast;
    const double* B; const int64_t* b_k; const int64_t* b_n; int b_nfast;
    double* C; const int64_t* c_m; const int64_t* c_n;
    double beta;
    int64_t tiles_n, tiles;
    int sym;               // C = A A^T: tiles below the diagonal are mirrors of those above
};

// T x T outputs per block, R x R per thread (stride T / R), BK deep stages.
template <int T, int R, int BK, int NT>
__global__ void __launch_bounds__(NT) k_gemm_f64(const GemmArgs g) {
    constexpr int W = T / R;                  // threads along a tile side
    constexpr int E = T * BK / NT;            // elements a thread stages per operand
    static_assert(W * W == NT && E * NT == T * BK, "tile shape");
    __shared__ double As[BK][T + 1];
    __shared__ double Bs[BK][T + 1];
    const int tid = threadIdx.x;
    const int tx = tid % W, ty = tid / W;

    const int64_t kbeg = (int64_t)blockIdx.z * g.kper;
    const int64_t kend = min(g.K, kbeg + g.kper);
    for (int64_t tile = blockIdx.x; tile < g.tiles; tile += gridDim.x) {
        const int64_t tm = tile / g.tiles_n, tn = tile - tm * g.tiles_n;
        if (g.sym && tn < tm) continue;
        const int64_t m0 = tm * T, n0 = tn * T;

        double acc[R][R];
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < R; ++j) acc[i][j] = 0.0;

        double ra[E], rb[E];
        auto load = [&](int64_t k0) {
#pragma unroll
            for (int q = 0; q < E; ++q) {
                const int e = tid + q * NT;
                int r, kk;
                if (g.a_kfast) { kk = e % BK; r = e / BK; } else { r = e % T; kk = e / T; }
                const int64_t m = m0 + r, k = k0 + kk;
                ra[q] = (m < g.M && k < kend) ? g.A[g.a_m[m] + g.a_k[k]] : 0.0;
            }
#pragma unroll
            for (int q = 0; q < E; ++q) {
                const int e = tid + q * NT;
                int c, kk;
                if (g.b_nfast) { c = e % T; kk = e / T; } else { kk = e % BK; c = e / BK; }
                const int64_t n = n0 + c, k = k0 + kk;
                rb[q] = (n < g.N && k < kend) ? g.B[g.b_k[k] + g.b_n[n]] : 0.0;
            }
        };
        load(kbeg);
        for (int64_t k0 = kbeg; k0 < kend; k0 += BK) {
            __syncthreads();                  // the previous stage has been read
#pragma unroll
            for (int q = 0; q < E; ++q) {
                const int e = tid + q * NT;
                if (g.a_kfast) As[e % BK][e / BK] = ra[q]; else As[e / T][e % T] = ra[q];
                if (g.b_nfast) Bs[e / T][e % T] = rb[q]; else Bs[e % BK][e / BK] = rb[q];
            }
            __syncthreads();
            if (k0 + BK < kend) load(k0 + BK);
#pragma unroll 8
            for (int kk = 0; kk < BK; ++kk) {
                double a[R], b[R];
#pragma unroll
                for (int i = 0; i < R; ++i) a[i] = As[kk][ty + W * i];
#pragma unroll
                for (int j = 0; j < R; ++j) b[j] = Bs[kk][tx + W * j];
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int j = 0; j < R; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
            }
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int64_t m = m0 + ty + W * i;
            if (m >= g.M) continue;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const int64_t n = n0 + tx + W * j;
                if (n >= g.N) continue;
                const double v = acc[i][j];
                if (g.partial) {
                    double* P = g.partial + (int64_t)blockIdx.z * g.M * g.N;
                    P[m * g.N + n] = v;
                    if (g.sym && tn > tm) P[n * g.N + m] = v;
                } else {
                    double* dst = g.C + g.c_m[m] + g.c_n[n];
                    *dst = (g.beta != 0.0) ? fma(g.beta, *dst, v) : v;
                    if (g.sym && tn > tm) g.C[g.c_m[n] + g.c_n[m]] = v;
                }
            }
        }
    }
}

// C = beta C + sum_z P[z], summed in z order (deterministic).
__global__ void k_reduce_partials(const double* __restrict__ P, int nz, int64_t M, int64_t N, double* C,
                                  const int64_t* c_m, const int64_t* c_n, double beta) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= M * N) return;
    double s = 0.0;
    for (int z = 0; z < nz; ++z) s += P[(int64_t)z * M * N + e];
    const int64_t m = e / N, n = e % N;
    double* dst = C + c_m[m] + c_n[n];
    *dst = (beta != 0.0) ? fma(beta, *dst, s) : s;
}

// Tile side and K parts of a product: the pair with the least modelled time,
// in clocks.  A block's time is its FMAs at the pipe's rate, the blocks are
// dealt evenly over the SMs, each K stage costs the latency of its loads
// unless several blocks share the SM, and split K adds a second launch.
struct Shape { int T; int64_t nz; double clocks; };
Shape choose_shape(int64_t M, int64_t N, int64_t K, int sms, bool sym, int64_t max_nz = 64) {
    Shape best{64, 1, 0.0};
    double best_t = 1e300;
    for (int T : {64, 32, 16, 8}) {
        const int bk = T == 64 ? 16 : T == 8 ? 64 : 32;
        const int64_t gx = (N + T - 1) / T, gy = (M + T - 1) / T;
        const double tiles = sym ? 0.5 * (double)gx * (double)(gx + 1) : (double)gx * (double)gy;
        for (int64_t nz = 1; nz <= max_nz; nz *= 2) {
            if (nz > 1 && (K / nz < 128 || (double)nz * M * N * 8 > (double)(4 << 20))) break;
            const double kper = std::ceil((double)K / nz / bk) * bk;
            const double per_sm = std::ceil(tiles * nz / sms);
            const double t = per_sm * T * T * kper / 1.9 + std::ceil(kper / bk) * (1200.0 / std::min(per_sm, 4.0)) * per_sm +
                             (nz > 1 ? 7000.0 : 0.0);
            if (t < best_t) { best_t = t; best = {T, nz, t}; }
        }
    }
    return best;
}

template <int T, int R, int BK, int NT>
void launch(Ctx& ctx, GemmArgs g, int64_t nz) {
    g.tiles_n = (g.N + T - 1) / T;
    g.tiles = g.tiles_n * ((g.M + T - 1) / T);
    if (nz > 1) g.kper = ((g.K + nz - 1) / nz + BK - 1) / BK * BK;
    const int64_t parts = nz > 1 ? (g.K + g.kper - 1) / g.kper : 1;
    if (parts > 1) {
        ctx.ensure(ctx.f64_partial, (size_t)(parts * g.M * g.N) * sizeof(double));
        g.partial = ctx.f64_partial.as<double>();
    }
    dim3 grid((unsigned)std::min<int64_t>(g.tiles, 1 << 30), 1, (unsigned)parts);
    k_gemm_f64<T, R, BK, NT><<<grid, NT, 0, ctx.stream>>>(g);
    TRG_LAUNCHED(ctx);
    if (parts > 1) {
        const int64_t tot = g.M * g.N;
        k_reduce_partials<<<(unsigned)((tot + 255) / 256), 256, 0, ctx.stream>>>(g.partial, (int)parts, g.M, g.N, g.C,
                                                                              g.c_m, g.c_n, g.beta);
        TRG_LAUNCHED(ctx);
    }
}

}  // namespace

double f64_us(const Ctx& ctx, int64_t M, int64_t N, int64_t K, bool sym) {
    return choose_shape(M, N, std::max<int64_t>(K, 1), ctx.sm_count, sym).clocks / 1900.0 + 3.0;
}

void gemm_f64(Ctx& ctx, const GemmDesc& d) {
    if (d.M <= 0 || d.N <= 0) return;
    GemmArgs g;
    g.M = d.M; g.N = d.N; g.K = d.K;
    g.kper = std::max<int64_t>(d.K, 1);
    g.partial = nullptr;
    g.A = d.A.base; g.a_m = d.A.off_r; g.a_k = d.A.off_c; g.a_kfast = d.A.c_fast ? 1 : 0;
    g.B = d.B.base; g.b_k = d.B.off_r; g.b_n = d.B.off_c; g.b_nfast = d.B.c_fast ? 1 : 0;
    g.C = d.C; g.c_m = d.c_m; g.c_n = d.c_n; g.beta = d.beta;
    // a Gram product's C(n, m) sums the products of C(m, n) in the same order
    g.sym = (d.gram && d.M == d.N && d.beta == 0.0) ? 1 : 0;
    if ((d.M + 63) / 64 > 65535) fail(TRG_EINVAL, "gemm_f64: too many row tiles");
    // The K parts (whose length follows the tile) change bits, the tile alone
    // does not: a slab takes the parts of its whole product, and without any the
    // tile of its own size.
    const int64_t k = std::max<int64_t>(d.K, 1);
    Shape s = choose_shape(d.choice_m(), d.choice_n(), k, ctx.sm_count, g.sym != 0);
    if (s.nz == 1) s = choose_shape(d.M, d.N, k, ctx.sm_count, g.sym != 0, 1);
    switch (s.T) {
        case 64: launch<64, 4, 16, 256>(ctx, g, s.nz); break;
        case 32: launch<32, 2, 32, 256>(ctx, g, s.nz); break;
        case 16: launch<16, 1, 32, 256>(ctx, g, s.nz); break;
        default: launch<8, 1, 64, 64>(ctx, g, s.nz); break;
    }
}

}  // namespace trg
