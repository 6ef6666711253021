// FP64 products on the tcgen05 tensor cores (TRG_FP64, large products).
//
// The FP64 pipe of this part does 1.9 FMA a clock and SM, 1/2000 of the BF16
// tensor rate, so an FP64 product that is large enough is computed from BF16
// digit products instead, to more than FP64 accuracy.  Each operand row (A) /
// column (B) gets a power-of-two scale 2^e with |x| < 2^e, and
//     X = rint(x 2^(119 - e)) = sum_p d_p 2^(8 (14 - p)),   p = 0..14,
// d_0 in [-128, 128], d_p in [-128, 127] (an error-free splitting as in
// split_gemm.cu, with every sum exact: Ozaki, Ogita, Oishi, Rump, Numer.
// Algorithms 59 (2012) 95).  With D_d = sum_{p + q = d} A_p B_q,
//     C = 2^(ea + eb - 126) sum_{d < 15} D_d 2^(8 (14 - d)):
// digit products are integers up to 2^14, a run of 64 K sums the at most 15
// products of a D_d exactly in FP32 (15 x 64 x 2^14 < 2^24), the epilogue
// moves each run into int64 sums and the wide total is turned into FP64.
//
// Why 15 digits: what is left out is below 16 K 2^-120 2^(ea + eb), so every
// element of C is as accurate as an FP64 sum, relative to its own sum |a||b|,
// down to sums 2^-60 of the largest possible one.  Eight digits are enough for
// an error far below FP64's relative to the largest elements, and cost a
// third, but the method needs the small elements too: the couplings between
// nearly decoupled sectors of a tensor decide how near-degenerate vectors mix.
// (Critical Ising with a field, Dcut 16, 20 half-steps: <s> varies with the
// start vectors by 8e-10 with the FP64 pipe, by 9e-8 with eight digits.)
//
// Rows or columns whose largest entry lies outside 2^-400 .. 2^400, or that
// hold an infinity or a NaN, raise a device flag: the tensor kernel then
// returns at once and the FP64 pipe kernel that is queued behind it, idle
// otherwise, computes the product.
//
// What bounds it: the tensor pipe, 120 digit products of 2 M N K each.
// 128 x 32 output tile, one persistent CTA per SM: the 15 D_d of 32 columns
// take 480 TMEM columns.  A stage is 16 K of both operands (60 KB of A digits,
// 15 KB of B digits, one TMA box each), two stages.  The products of one A
// digit with adjacent B digits land in adjacent accumulators, so 22
// instructions of up to N = 256 cover the 120 products of a step.  They are
// issued in two groups, the one that lands in D_7..D_14 (92 products) before
// the one that lands in D_0..D_6: a run's drain of D_7..D_14 runs under the
// other group's products, and the drain of D_0..D_6 under the next run's first
// group.  Measured, contraction at Dx = Dy = Dn = 48 (three products, 1.22e12
// FP64 FLOPs): 993 ms on the
// FP64 pipe, 113 here, 110 of them in this kernel (1.5e14 digit FLOPs, 1340
// TFLOP/s); environment at (24, 22): 0.65 -> 0.28 ms.
#include <algorithm>
#include <cmath>

#include "internal.h"
#include "slicing.cuh"
#include "tcgen05.cuh"

namespace trg {

namespace {

constexpr int XS = 15;                           // digits
constexpr int XM = 128, XN = 32, XK = 16;        // tile rows, columns, K per stage
constexpr int XL = 7;                            // D_0 .. D_(XL-1) are group 0, the rest group 1
constexpr int XA_TILE = XM * XK * 2;             // bytes of one digit's A tile
constexpr int XB_TILE = XN * XK * 2;
constexpr int XSTAGE = XS * (XA_TILE + XB_TILE); // 75 KB
constexpr int XSTAGES = 2;
constexpr int XRUN = 64 / XK;                    // stages of an exact run
constexpr int XEPI = 16;                         // epilogue warps
constexpr int XTHREADS = 64 + 32 * XEPI;
constexpr int XCPT = XN / 4;                     // columns per epilogue thread
constexpr int XSTAGING = XEPI * 32 * 8 * 8;      // store staging, 32 KB
constexpr int XBAR = 256;
constexpr int XSMEM = XSTAGES * XSTAGE + XSTAGING + XBAR + 1024;
static_assert(XSMEM <= 232448, "exact product shared memory");

// The digit products of one 16-deep step: A digit a times the n <= 8 B digits
// from b on, into the accumulators D_(a+b) .. D_(a+b+n-1).  Group 1 lands in
// D_7..D_14, group 0 in D_0..D_6; the first entry of a group covers all of its
// accumulators and resets them at the start of a run.
struct XIns { int a, b, n, group; };
__host__ __device__ constexpr int xins_count() { return XS + XL; }
__host__ __device__ constexpr XIns xins(int t) {
    return t < XS ? XIns{t, t < XL ? XL - t : 0, t < XL ? XS - XL : XS - t, 1} : XIns{t - XS, 0, XL - (t - XS), 0};
}
__host__ __device__ constexpr bool xins_ok() {
    int seen[XS][XS] = {};
    for (int t = 0; t < xins_count(); ++t) {
        const XIns in = xins(t);
        if (in.n < 1 || in.n * XN > 256) return false;
        for (int q = in.b; q < in.b + in.n; ++q) {
            const int d = in.a + q;
            if (d >= XS || (d >= XL) != (in.group == 1)) return false;
            seen[in.a][q] += 1;
        }
    }
    for (int p = 0; p < XS; ++p)
        for (int q = 0; q < XS; ++q)
            if (seen[p][q] != (p + q < XS ? 1 : 0)) return false;
    return xins(0).n == XS - XL && xins(XS).n == XL;
}
static_assert(xins_ok(), "digit product table");
static_assert(XS * XN <= 512 && (double)XS * 64 * (1 << 14) <= (1 << 24), "accumulators");

// Shared-memory matrix descriptor: K-major BF16 tile, 32-byte rows, 32-byte
// swizzle; 8-row groups 256 bytes apart.
__device__ __forceinline__ uint64_t xsmem_desc(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);          // start address
    d |= (uint64_t)1 << 16;                         // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(256 >> 4) << 32;                // stride byte offset
    d |= (uint64_t)1 << 46;                         // descriptor version
    d |= (uint64_t)6 << 61;                         // swizzle: 32 bytes
    return d;
}

struct XArgs {
    int M, N, Kp;
    const int* fa;                 // largest exponent field of each A row
    const int* fb;                 // ... of each B column
    double* C;
    const int64_t* c_m;
    const int64_t* c_n;
    int rows_fast;                 // consecutive rows are (mostly) adjacent in C: store row-wise
    int sym;                       // C symmetric: the tile list holds the tiles that reach the diagonal
    const long long* tile_list;    // mb << 32 | nb, or nullptr for all
    int n_list;
    int group_n;                   // tile order: column blocks per group
    const int* bad;                // the operands are outside the digits' range: do nothing
    int* status;
};

// The int64 sums of an element: D_0..D_3, D_4..D_7, D_8..D_11, D_12..D_14, each
// in units of its last D: V = w0 2^88 + w1 2^56 + w2 2^24 + w3.
// V 2^e2 in FP64, within 2 units in the last place.
__device__ __forceinline__ double wide_to_double(const long long (&w)[4], int e2) {
    long long w2 = w[2] + (w[3] >> 24);
    long long w1 = w[1] + (w2 >> 32);
    const long long w0 = w[0] + (w1 >> 32);
    double r = fma((double)w0, 4294967296.0, (double)(unsigned)(w1 & 0xffffffffll));
    r = fma(r, 4294967296.0, (double)(unsigned)(w2 & 0xffffffffll));
    r = fma(r, 16777216.0, (double)(int)(w[3] & 0xffffffll));
    if (r == 0.0) return 0.0;
    // (nonzero rows and columns have -928 <= e2 <= 676 and |r| < 2^150: the field stays in range)
    return __longlong_as_double(__double_as_longlong(r) + ((long long)e2 << 52));
}

__global__ void __launch_bounds__(XTHREADS, 1)
k_exact_mma(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const XArgs g) {
    if (*g.bad) return;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + XSTAGES * XSTAGE + XSTAGING);
    uint64_t* empty = full + XSTAGES;
    uint64_t* acc_full = empty + XSTAGES;        // [group]
    uint64_t* acc_empty = acc_full + 2;          // [group]
    uint64_t* mma_done = acc_empty + 2;
    uint32_t* tmem_slot = (uint32_t*)(mma_done + 1);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    double* staging = (double*)(smem + XSTAGES * XSTAGE);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles_m = (g.M + XM - 1) / XM, tiles_n = (g.N + XN - 1) / XN;
    const int num_tiles = g.tile_list ? g.n_list : tiles_m * tiles_n;
    const int num_kb = g.Kp / XK;
    auto coords = [&](int tile, int& mb, int& nb) {
        if (g.tile_list) {
            const long long v = g.tile_list[tile];
            mb = (int)(v >> 32);
            nb = (int)(v & 0xffffffffll);
        } else {
            const int per_group = tiles_m * g.group_n;
            const int group = tile / per_group, first = group * g.group_n;
            const int width = min(g.group_n, tiles_n - first), local = tile - group * per_group;
            mb = local / width;
            nb = first + local % width;
        }
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < XSTAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int q = 0; q < 2; ++q) { mbar_init(&acc_full[q], 1); mbar_init(&acc_empty[q], XEPI); }
        mbar_init(mma_done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(512u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            int issued[XSTAGES];
#pragma unroll
            for (int s = 0; s < XSTAGES; ++s) issued[s] = -1;
            bool ok = true;
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
                int mb, nb;
                coords(tile, mb, nb);
                for (int kb = 0; kb < num_kb; ++kb) {
                    ok = mbar_wait(&empty[stage], phase ^ 1, abort_flag, g.status);
                    if (!ok) break;
                    uint8_t* st = smem + stage * XSTAGE;
                    mbar_expect_tx(&full[stage], XSTAGE);
                    tma_load_3d(st, &tmA, kb * XK, mb * XM, 0, &full[stage]);
                    tma_load_3d(st + XS * XA_TILE, &tmB, kb * XK, nb * XN, 0, &full[stage]);
#pragma unroll
                    for (int s = 0; s < XSTAGES; ++s)
                        if (s == stage) issued[s] = (int)phase;
                    if (++stage == XSTAGES) { stage = 0; phase ^= 1; }
                }
            }
            // every load issued has landed before the CTA may exit (bounded, also after an abort)
            volatile int never = 0;
#pragma unroll
            for (int s = 0; s < XSTAGES; ++s)
                if (issued[s] >= 0) mbar_wait(&full[s], (uint32_t)issued[s], &never, g.status);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t run_no = 0;        // runs begun so far (all tiles)
            bool ok = true;
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
                for (int kb = 0; kb < num_kb; ++kb) {
                    const bool run_start = kb % XRUN == 0;
                    const bool run_end = (kb + 1) % XRUN == 0 || kb + 1 == num_kb;
                    ok = mbar_wait(&full[stage], phase, abort_flag, g.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t dbase = xsmem_desc(smem_u32(smem + stage * XSTAGE));
                    auto issue = [&](int group) {
#pragma unroll
                        for (int t = 0; t < xins_count(); ++t) {
                            const XIns in = xins(t);
                            if (in.group != group) continue;
                            const uint32_t acc = ((t == 0 || t == XS) && run_start) ? 0u : 1u;
                            const uint64_t da = dbase + (uint64_t)((in.a * XA_TILE) >> 4);
                            const uint64_t db = dbase + (uint64_t)((XS * XA_TILE + in.b * XB_TILE) >> 4);
                            mma_bf16<1>(tmem + (uint32_t)((in.a + in.b) * XN), da, db, idesc_bf16(XM, in.n * XN), acc);
                        }
                    };
                    if (run_start && run_no > 0) {
                        ok = mbar_wait(&acc_empty[1], (run_no - 1) & 1, abort_flag, g.status);
                        if (!ok) break;
                        tc_fence_after();
                    }
                    issue(1);
                    if (run_end) mma_commit<1>(&acc_full[1]);
                    if (run_start && run_no > 0) {
                        ok = mbar_wait(&acc_empty[0], (run_no - 1) & 1, abort_flag, g.status);
                        if (!ok) break;
                        tc_fence_after();
                    }
                    issue(0);
                    mma_commit<1>(&empty[stage]);
                    if (run_end) {
                        mma_commit<1>(&acc_full[0]);
                        ++run_no;
                    }
                    if (++stage == XSTAGES) { stage = 0; phase ^= 1; }
                }
            }
            // every MMA issued has completed (also after an abort)
            mma_commit<1>(mma_done);
            volatile int never = 0;
            mbar_wait(mma_done, 0, &never, g.status);
        }
    } else {
        const int ew = warp - 2, quad = warp & 3, colq = ew >> 2;
        const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
        uint32_t run_no = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
            int mb, nb;
            coords(tile, mb, nb);
            const int nruns = (num_kb + XRUN - 1) / XRUN;
            long long w[XCPT][4];
#pragma unroll
            for (int j = 0; j < XCPT; ++j) w[j][0] = w[j][1] = w[j][2] = w[j][3] = 0;
            for (int c = 0; c < nruns && ok; ++c, ++run_no) {
#pragma unroll
                for (int grp = 1; grp >= 0; --grp) {
                    int w_ok = 1;
                    if (lane == 0) w_ok = mbar_wait(&acc_full[grp], run_no & 1, abort_flag, g.status) ? 1 : 0;
                    ok = __shfl_sync(0xffffffffu, w_ok, 0) != 0;
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll
                    for (int d = grp ? XL : 0; d < (grp ? XS : XL); ++d) {
                        uint32_t r[XCPT];
                        tmem_ld8(tmem + lane_base + (uint32_t)(d * XN + colq * XCPT), r);
                        tmem_wait_ld();
                        constexpr int last[4] = {3, 7, 11, 14};
                        const long long unit = 1ll << (8 * (last[d >> 2] - d));
#pragma unroll
                        for (int j = 0; j < XCPT; ++j) w[j][d >> 2] += (long long)__float2int_rn(__uint_as_float(r[j])) * unit;
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[grp]);
                }
            }
            if (!ok) break;
            const int m = mb * XM + quad * 32 + lane;
            const bool row_ok = m < g.M;
            const int nt = nb * XN + colq * XCPT;
            // the warp's eight columns are the same for every lane: lane j loads
            // column j's exponent and offset, the loop takes them by shuffle
            const bool col_in = lane < XCPT && nt + lane < g.N;
            const int fb = col_in ? g.fb[nt + lane] : 0;
            const long long cn_l = col_in ? (long long)g.c_n[nt + lane] : 0;
            const int ea = row_ok ? max(g.fa[m], 1) - 1022 : 0;
            const int eb_l = max(fb, 1) - 1022 - 126;
            if (g.rows_fast) {
                // lanes are adjacent rows, adjacent in C
                double* cp = g.C + (row_ok ? g.c_m[m] : 0);
#pragma unroll
                for (int j = 0; j < XCPT; ++j) {
                    const int e2 = ea + __shfl_sync(0xffffffffu, eb_l, j);
                    const long long cn = __shfl_sync(0xffffffffu, cn_l, j);
                    if (row_ok && nt + j < g.N) cp[cn] = wide_to_double(w[j], e2);
                }
                continue;
            }
            double v[XCPT];
#pragma unroll
            for (int j = 0; j < XCPT; ++j) {
                const int e2 = ea + __shfl_sync(0xffffffffu, eb_l, j);
                v[j] = (row_ok && nt + j < g.N) ? wide_to_double(w[j], e2) : 0.0;
            }
            if (g.sym && row_ok) {
                // the mirror (n, m) of each element above the diagonal
                const int64_t cm_mirror = g.c_n[m];
#pragma unroll
                for (int j = 0; j < XCPT; ++j) {
                    const int n = nt + j;
                    if (n < g.N && n > m) g.C[g.c_m[n] + cm_mirror] = v[j];
                }
            }
            // columns adjacent in C: through the warp's 32 x 8 staging tile, so
            // that a quarter-warp writes 8 adjacent columns of one row
            double* stg = staging + ew * (32 * 8);
            const int quarter = lane >> 3, cl = lane & 7;
#pragma unroll
            for (int pass = 0; pass < XCPT / 8; ++pass) {
#pragma unroll
                for (int jj = 0; jj < 8; ++jj) stg[lane * 8 + (jj ^ ((lane >> 1) & 7))] = v[pass * 8 + jj];
                const int64_t cn = __shfl_sync(0xffffffffu, cn_l, pass * 8 + cl);
                __syncwarp();
                const int n = nt + pass * 8 + cl;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int rr = 4 * q + quarter;
                    const int mr = mb * XM + quad * 32 + rr;
                    if (mr < g.M && n < g.N && (!g.sym || n >= mr))
                        g.C[g.c_m[mr] + cn] = stg[rr * 8 + (cl ^ ((rr >> 1) & 7))];
                }
                __syncwarp();
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
    }
}

// ------------------------------------------------------------- host side ---
// Digit planes [XS][rows][kp] as a 3D map, boxes of box_rows x XK of every digit.
CUtensorMap digit_map(const void* base, int rows, int kp, int box_rows) {
    CUtensorMap m;
    std::memset(&m, 0, sizeof(m));
    const cuuint64_t dims[3] = {(cuuint64_t)kp, (cuuint64_t)rows, (cuuint64_t)XS};
    const cuuint64_t strides[2] = {(cuuint64_t)kp * 2, (cuuint64_t)kp * 2 * (cuuint64_t)rows};
    const cuuint32_t box[3] = {(cuuint32_t)XK, (cuuint32_t)box_rows, (cuuint32_t)XS};
    const cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
                             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) fail(TRG_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
    return m;
}

int64_t up(int64_t v, int64_t q) { return (v + q - 1) / q * q; }

// Exponent fields and digits of rows [0, R) of an operand.
void digits(Ctx& ctx, const Gather& g, int R, int K, int Rp, int Kp, int* ef, uint16_t* out, int* bad) {
    if (g.c_identity && Kp <= CUT_ROWS_MAX_K) {
        launch_cut_rows<XS, true>(ctx.stream, g.base, g.off_r, R, K, Rp, Kp, ef, nullptr, out, bad);
        TRG_LAUNCHED(ctx);
        return;
    }
    TRG_CUDA(cudaMemsetAsync(ef, 0, (size_t)R * sizeof(int), ctx.stream));
    launch_row_field<true>(ctx.stream, g, R, K, ef);
    TRG_LAUNCHED(ctx);
    launch_cut<XS>(ctx.stream, g, R, K, Rp, Kp, ef, nullptr, out, bad);
    TRG_LAUNCHED(ctx);
}

const long long* diagonal_tiles(Ctx& ctx, int tiles_m, int tiles_n, int& n) {
    const std::string key = "xsym:" + std::to_string(tiles_m) + ":" + std::to_string(tiles_n);
    auto it = ctx.lists.find(key);
    if (it == ctx.lists.end()) {
        std::vector<long long> h;
        for (int mb = 0; mb < tiles_m; ++mb)
            for (int nb = 0; nb < tiles_n; ++nb)
                if ((int64_t)nb * XN + XN - 1 >= (int64_t)mb * XM) h.push_back(((long long)mb << 32) | nb);
        Buf buf;
        ctx.ensure(buf, h.size() * sizeof(long long));
        TRG_CUDA(cudaMemcpyAsync(buf.p, h.data(), h.size() * sizeof(long long), cudaMemcpyHostToDevice, ctx.stream));
        TRG_CUDA(cudaStreamSynchronize(ctx.stream));   // h dies here
        it = ctx.lists.emplace(key, buf).first;
        ctx.list_len[key] = (int)h.size();
    }
    n = ctx.list_len[key];
    return it->second.as<long long>();
}

// Rows of an operand whose digits are held at a time: at most XCAP bytes of
// them (a multiple of the tile).
constexpr int64_t XCAP = (int64_t)1 << 30;
int64_t block_rows(int64_t rows, int64_t kp, int64_t tile) {
    const int64_t most = std::max<int64_t>(tile, XCAP / (2 * XS * kp) / tile * tile);
    return std::min(up(rows, tile), most);
}

}  // namespace

int64_t exact_scratch_bytes(int64_t M, int64_t N, int64_t K) {
    const int64_t kp = up(std::max<int64_t>(K, 1), XK);
    const int64_t ra = block_rows(M, kp, XM), rb = block_rows(N, kp, XN);
    return 2 * XS * kp * (ra + rb) + 4 * (ra + rb) + 2048;
}

double exact_us(const Ctx& ctx, int64_t M, int64_t N, int64_t K, bool sym) {
    if (M > (1ll << 30) || N > (1ll << 30) || K > (1 << 17)) return 1e300;
    const double tm = (double)up(M, XM) / XM, tn = (double)up(N, XN) / XN;
    const double tiles = sym ? 0.5 * tm * (tn + 4) : tm * tn;
    const double runs = std::ceil((double)K / 64.0);
    const double mma = std::ceil(tiles / ctx.sm_count) * (runs * 4.4 + 3.0);
    const double moved = (46.0 * (double)K * ((double)M + (sym ? 0.0 : (double)N)) + 8.0 * (double)M * (double)N) / 4.0e6;
    return 25.0 + mma + moved;
}

bool gemm_exact(Ctx& ctx, const GemmDesc& d) {
    const int K = (int)std::max<int64_t>(d.K, 1), Kp = (int)up(K, XK);
    const int64_t ra = block_rows(d.M, Kp, XM), rb = block_rows(d.N, Kp, XN);
    const bool sym = d.gram && d.M == d.N && ra >= d.M;
    try {
        ctx.ensure(ctx.split_ws, (size_t)exact_scratch_bytes(d.M, sym ? 1 : d.N, K));
    } catch (const Error& e) {
        if (e.status == TRG_ENOMEM) return false;    // no room for the digits: the FP64 pipe needs none
        throw;
    }
    uint8_t* p = ctx.split_ws.as<uint8_t>();
    auto take = [&](size_t bytes) { uint8_t* q = p; p += (bytes + 255) & ~(size_t)255; return q; };
    int* bad = (int*)take(4);
    int* fa = (int*)take((size_t)ra * 4);
    int* fb = sym ? fa : (int*)take((size_t)rb * 4);
    uint16_t* sa = (uint16_t*)take((size_t)(2 * XS) * ra * Kp);
    uint16_t* sb = sym ? sa : (uint16_t*)take((size_t)(2 * XS) * rb * Kp);
    TRG_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), ctx.stream));
    static std::once_flag once;
    std::call_once(once, [] {
        TRG_CUDA(cudaFuncSetAttribute(k_exact_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, XSMEM));
    });

    // B as rows n, columns k
    const Gather bt = transposed(d.B);
    for (int64_t m0 = 0; m0 < d.M; m0 += ra) {
        const int mr = (int)std::min(ra, d.M - m0), mp = (int)up(mr, XM);
        Gather ga = d.A;
        ga.off_r += m0;
        digits(ctx, ga, mr, K, mp, Kp, fa, sa, bad);
        const CUtensorMap ta = digit_map(sa, mp, Kp, XM);
        for (int64_t n0 = 0; n0 < d.N; n0 += rb) {
            const int nr = (int)std::min(rb, d.N - n0), np = sym ? mp : (int)up(nr, XN);
            if (!sym && (m0 == 0 || rb < d.N)) {
                Gather gb = bt;
                gb.off_r += n0;
                digits(ctx, gb, nr, K, np, Kp, fb, sb, bad);
            }
            const CUtensorMap tb = digit_map(sb, np, Kp, XN);
            XArgs a;
            a.M = mr; a.N = sym ? mr : nr; a.Kp = Kp;
            a.fa = fa; a.fb = fb;
            a.C = d.C; a.c_m = d.c_m + m0; a.c_n = d.c_n + n0;
            a.rows_fast = d.c_m_fast && !sym ? 1 : 0;
            a.sym = sym ? 1 : 0;
            a.tile_list = nullptr; a.n_list = 0;
            a.bad = bad; a.status = ctx.status.as<int>();
            const int tiles_m = mp / XM, tiles_n = (a.N + XN - 1) / XN;
            int tiles = tiles_m * tiles_n;
            if (sym) {
                a.tile_list = diagonal_tiles(ctx, tiles_m, tiles_n, a.n_list);
                tiles = a.n_list;
            }
            // column blocks whose digits share L2 (about 40 MB of them)
            a.group_n = (int)std::max<int64_t>(1, std::min<int64_t>(tiles_n, (40ll << 20) / ((int64_t)XN * Kp * 2 * XS)));
            const int grid = std::min(tiles, ctx.sm_count);
            const int tok = ctx.region_begin(TRG_PHASE_MMA);
            k_exact_mma<<<grid, XTHREADS, XSMEM, ctx.stream>>>(ta, tb, a);
            TRG_LAUNCHED(ctx);
            ctx.region_end(tok, 2.0 * (double)mr * nr * K, 120.0 * 2.0 * (double)mr * nr * Kp);
            if (sym) break;
        }
    }
    gemm_f64(ctx, d, bad);    // computes the product if an operand was out of range, else returns at once
    return true;
}

}  // namespace trg
