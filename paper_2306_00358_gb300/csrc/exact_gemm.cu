// FP64 products on the tcgen05 tensor cores (TRG_FP64, large products).
//
// The FP64 pipe of this part does 1.9 FMA a clock and SM, 1/2000 of the BF16
// tensor rate, so an FP64 product that is large enough is computed from BF16
// digit products instead, to more than FP64 accuracy.  Each operand row (A) /
// column (B) gets a power-of-two scale 2^e with |x| < 2^e, and
//     X = rint(x 2^(119 - e)) = sum_p d_p 2^(8 (14 - p)),   p = 0..14,
// d_0 in [-128, 128], d_p in [-128, 127] (an error-free splitting as in
// split_gemm.cu, with every sum exact: Ozaki, Ogita, Oishi, Rump, Numer.
// Algorithms 59 (2012) 95).  With D_d = sum_{p + q = d} A_p B_q and S digits,
//     C = 2^(ea + eb - 14) sum_{d < S} D_d 2^(-8 d):
// digit products are integers up to 2^14, a short run of K (64 for 15 digits,
// 96 for 9) sums the at most S products of a D_d exactly in FP32, the
// epilogue moves each run into int64 sums and the wide total is turned into
// FP64.
//
// How many digits: S leave out less than (S + 2) K 2^(-8 S) 2^(ea + eb).  The
// result has to be as accurate as an FP64 sum element by element, relative to
// its own sum |a||b| (the method feeds the couplings between nearly decoupled
// sectors of a tensor back, so small elements count).  So every form comes with
// that sum, taken from one more BF16 plane of each operand, |x| cut off:
//  - 15 digits (120 digit products) do it down to sums |a||b| of 2^-60 2^(ea +
//    eb): they leave out less than K 2^-55 |a||b|, where an FP64 sum's roundings
//    amount to up to K 2^-53 |a||b|; products too small for a choice always take
//    them.  The sum is one more accumulator of the same kernel, which marks the
//    elements below 2^-60, and those of rows or columns whose largest entry lies
//    outside 2^-400 .. 2^400 or that hold an infinity or a NaN.  A kernel queued
//    behind it computes the marked elements on the FP64 pipe (k_weak_f64; it
//    returns at once if there is none).  In FP64 solves at the critical point no
//    sum lies below 2^-54; far from it, once the tensor has flowed to a fixed
//    point, 2 to 40 % of them do;
//  - 9 digits (45 digit products) do it if the sum |a||b| does not lie between 0
//    and 2^-8 2^(ea + eb): they leave out less than K 2^-60 |a||b| then, which is
//    also below what the roundings of an FP64 sum amount to when their signs are
//    random.  A kernel takes all of |A||B| first and marks the rows with a sum
//    for which 9 do not suffice (the columns, where the product is a slab of
//    columns; the whole of a Gram product).  The nine-digit kernel stores the
//    others, the fifteen-digit kernel these, and each leaves out the tiles that
//    hold none of its own.  A row's decision is its own, so an element has the
//    same bits whatever slab or block of the product it is computed in.  (By
//    tiles there would be less to compute twice, but tiles begin where a slab
//    does.)
//
// What bounds it: the tensor pipe (9 digits in a long product: active 62 % of
// the time, with MMA instructions of N = 48 .. 240; a tenth goes to drains that
// nothing covers).  128 x 32 output tile with 15 digits, 128 x 48 with 9, one
// persistent CTA per SM: the S accumulators D_d of the tile's columns (and with 15
// digits the sums) fill tensor memory.  A stage is 16 (32) K of both operands, one
// TMA box each, two stages; the cut stores the digits in the order of a stage, so
// that a box is made of 4 KB pieces (as [p][r][k] planes its rows are pieces of 32
// or 64 bytes, and the TMA unit's requests hold the products up: 72 -> 68.6 us a
// product of an environment at (24, 22), both without the sums).  The products of
// one A digit with adjacent B digits land in adjacent accumulators, so 24 (13)
// instructions of up to N = 256 cover the products of a 16-deep step, the sums
// among them (one instruction more with 15; the launches of a contraction at (6,
// 37, 36) 149 -> 153 us with the marks).  They are issued in two
// groups, the one that lands in the higher D_d (84 of 120, 35 of 45 products)
// before the other: a run's drain of the higher D_d runs under the other group's
// products, and the drain of the lower ones under the next run's first group.
// Measured, contraction at Dx = Dy = Dn = 48 (1.22e12 FP64 FLOPs): 993 ms on
// the FP64 pipe, 110.7 ms where every row needs 15 digits, 44.8 ms where 9 suffice
// (39 ms of it in this kernel, 1.6 ms in the |A||B| sums, 3.8 ms in the cut), 619
// ms where half of the elements are left to the pipe.
#include <algorithm>
#include <cmath>

#include "internal.h"
#include "slicing.cuh"
#include "tcgen05.cuh"

namespace trg {

namespace {

constexpr int XM = 128;                          // tile rows
constexpr int XKP = 32;                          // K is padded to this
constexpr int XPLANES = planes(15);
constexpr int XBAR = 256;

// Shape of the kernel for S digits; S = 1 is the sum of |a||b|.
template <int S>
struct XT {
    static constexpr int N = S == 15 ? 32 : S == 9 ? 48 : 256;     // tile columns
    static constexpr int K = S == 15 ? 16 : 32;                    // K per stage
    static constexpr int L = S == 15 ? 8 : S == 9 ? 4 : 0;         // D_0 .. D_(L-1) are group 0, the rest group 1
    static constexpr int EPI = S == 9 ? 12 : 16;                   // epilogue warps: 16 columns each with 9 digits
    static constexpr int THREADS = 64 + 32 * EPI;
    static constexpr int KB = K / 16;
    static constexpr int A_TILE = XM * 32, B_TILE = N * 32;        // bytes of 16 K of one digit's tiles
    // 15 digits come with the |x| plane: its product, the sum of |a||b|, has
    // accumulators of its own (SUM) and runs over the whole K
    static constexpr bool SUM = S == 15;
    static constexpr int P = S + (SUM ? 1 : 0);                    // planes staged
    static constexpr int STAGE = KB * P * (A_TILE + B_TILE);       // 80, 99 and 24 KB
    static constexpr int STAGES = S == 1 ? 4 : 2;
    static constexpr int RUN = S == 1 ? 1 << 30 : S == 9 ? 3 : 4;  // stages of an exact run
    static constexpr int CPT = N / (EPI / 4);                      // columns per epilogue thread
    static constexpr int LIMBS = S == 15 ? 4 : 2;
    static constexpr int STAGING = S == 1 ? 0 : EPI * 32 * 8 * 8;  // store staging
    // at least 120 KB, so that a second CTA (and its tensor memory) never shares the SM
    static constexpr int BYTES = STAGES * STAGE + STAGING + XBAR + 1024;
    static constexpr int SMEM = BYTES > 120 * 1024 ? BYTES : 120 * 1024;
    static_assert(SMEM <= 232448, "exact product shared memory");
    static_assert(P * N <= 512 && (S == 1 || (double)S * RUN * K * (1 << 14) <= (1 << 24)), "accumulators");
};

// The digit products of one 16-deep step: A digit a times the n B digits from
// b on, into the accumulators D_(a+b) .. D_(a+b+n-1).  The first entry of a
// group covers all of its accumulators and resets them at the start of a run.
struct XIns { int a, b, n, group; };
template <int S>
__host__ __device__ constexpr int xins_count() { return S + XT<S>::L; }
template <int S>
__host__ __device__ constexpr XIns xins(int t) {
    constexpr int L = XT<S>::L;
    return t < S ? XIns{t, t < L ? L - t : 0, t < L ? S - L : S - t, 1} : XIns{t - S, 0, L - (t - S), 0};
}
template <int S>
__host__ __device__ constexpr bool xins_ok() {
    constexpr int L = XT<S>::L;
    int seen[S][S] = {};
    for (int t = 0; t < xins_count<S>(); ++t) {
        const XIns in = xins<S>(t);
        if (in.n < 1 || in.n * XT<S>::N > 256) return false;
        for (int q = in.b; q < in.b + in.n; ++q) {
            const int d = in.a + q;
            if (d >= S || (d >= L) != (in.group == 1)) return false;
            seen[in.a][q] += 1;
        }
    }
    for (int p = 0; p < S; ++p)
        for (int q = 0; q < S; ++q)
            if (seen[p][q] != (p + q < S ? 1 : 0)) return false;
    return xins<S>(0).n == S - L && (L == 0 || xins<S>(S).n == L);
}
static_assert(xins_ok<15>() && xins_ok<9>() && xins_ok<1>(), "digit product table");

// Shared-memory matrix descriptor: K-major BF16 tile, 32-byte rows, 32-byte
// swizzle; 8-row groups 256 bytes apart.
__device__ __forceinline__ uint64_t smem_desc32(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);          // start address
    d |= (uint64_t)1 << 16;                         // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(256 >> 4) << 32;                // stride byte offset
    d |= (uint64_t)1 << 46;                         // descriptor version
    d |= (uint64_t)6 << 61;                         // swizzle: 32 bytes
    return d;
}

enum Scope { NONE = 0, ROWS = 1, COLUMNS = 2, WHOLE = 3 };
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
    int* flags;                    // [0] some element is left to the FP64 pipe, [1] / [2] some need / do not need 15 digits
    // Which elements need 15 digits, if nine are tried: those of the rows (ROWS),
    // of the columns (COLUMNS) or of the product (WHOLE) with need[] set; state[]
    // says it for the tiles, 1: some do, 2: some do not.
    int scope;
    int* need;
    const int* state;
    uint32_t* weak;                // the elements left to it: bit n % 32 of weak[(n / 32) weak_rows + m]
    int* weak_tile;                // ... does the 128 x 32 tile (m / 128) words + n / 32 hold one
    int weak_rows, words;
    // a second Gram product of the same size: its rows are those from half on
    // (0: none), its tiles are in tile_list too
    int half;
    double* C1;
    const int64_t* c_m1;
    const int64_t* c_n1;
    int* status;
    unsigned long long acc_wait_ns;   // limit of the epilogue's waits (trg_set_wait_limit)
    double* flops;                 // profiling: the digit products of the tiles computed are added here
    double tile_flops;
};

// The int64 sums of an element, each in units of its last D, as FP64 times
// 2^e2, within 2 units in the last place.  15 digits: D_0..D_3, D_4..D_7,
// D_8..D_11, D_12..D_14, V = w0 2^88 + w1 2^56 + w2 2^24 + w3; 9 digits:
// D_0..D_3, D_4..D_8, V = w0 2^40 + w1.
__device__ __forceinline__ double wide_to_double(const long long (&w)[4], int e2) {
    long long w2 = w[2] + (w[3] >> 24);
    long long w1 = w[1] + (w2 >> 32);
    const long long w0 = w[0] + (w1 >> 32);
    double r = fma((double)w0, 4294967296.0, (double)(unsigned)(w1 & 0xffffffffll));
    r = fma(r, 4294967296.0, (double)(unsigned)(w2 & 0xffffffffll));
    r = fma(r, 16777216.0, (double)(int)(w[3] & 0xffffffll));
    if (r == 0.0) return 0.0;
    // (nonzero rows and columns have -928 <= e2 <= 732 and |r| < 2^150: the field stays in range)
    return __longlong_as_double(__double_as_longlong(r) + ((long long)e2 << 52));
}
__device__ __forceinline__ double wide_to_double(const long long (&w)[2], int e2) {
    const long long w0 = w[0] + (w[1] >> 40);
    const double r = fma((double)w0, 1099511627776.0, (double)(w[1] & 0xffffffffffll));
    if (r == 0.0) return 0.0;
    return __longlong_as_double(__double_as_longlong(r) + ((long long)e2 << 52));
}

__device__ __forceinline__ void tmem_ldn(uint32_t taddr, uint32_t (&r)[8]) { tmem_ld8(taddr, r); }
__device__ __forceinline__ void tmem_ldn(uint32_t taddr, uint32_t (&r)[16]) { tmem_ld16(taddr, r); }
// Keeps the use of loaded registers behind the wait for them.
template <int N>
__device__ __forceinline__ void tmem_arrived(uint32_t (&r)[N]) {
#pragma unroll
    for (int j = 0; j < N; ++j) asm volatile("" : "+r"(r[j]));
}

constexpr int XNINE_K = 16384;                    // the nine-digit sums fit in int64 up to this K
static_assert(5.0 * XNINE_K * (1 << 14) * 4294967296.0 * 1.01 < 9.2e18, "nine-digit sums");
// Sums |a||b| as the |x| planes give them, at which 9 and 15 digits suffice: 2^-8
// and 2^-60 of 2^(ea + eb).
constexpr float two_to(int e) { return e == 0 ? 1.0f : e > 0 ? 2.0f * two_to(e - 1) : 0.5f * two_to(e + 1); }
constexpr float SUM9_MIN = two_to(2 * SIZE_SHIFT - 8), SUM15_MIN = two_to(2 * SIZE_SHIFT - 60);
__device__ __forceinline__ bool sum_below(uint32_t bits, float least) {
    const float s = __uint_as_float(bits);
    return s > 0.0f && s < least;
}
// Largest exponent field of a row that the digits do not reach (2^-400 .. 2^400,
// infinities and NaN).
__device__ __forceinline__ bool field_outside(int f) { return f && (f < 1023 - 400 || f > 1023 + 400); }

template <int S>
__global__ void __launch_bounds__(XT<S>::THREADS, 1)
k_exact_mma(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const XArgs g) {
    constexpr int XN = XT<S>::N, XK = XT<S>::K, XL = XT<S>::L, XSTAGES = XT<S>::STAGES, XSTAGE = XT<S>::STAGE;
    constexpr int XA_TILE = XT<S>::A_TILE, XKB = XT<S>::KB, XB_TILE = XT<S>::B_TILE, XRUN = XT<S>::RUN, XCPT = XT<S>::CPT;
    if ((S == 9 && !g.flags[2]) || (S == 15 && g.scope && !g.flags[1])) return;
    constexpr int XP = XT<S>::P;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + XSTAGES * XSTAGE + XT<S>::STAGING);
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

    // What the tile holds (state[]): this kernel computes those with the bit MINE.
    // Its roles ask for the next tile while they work on the present one.
    constexpr int MINE = S == 9 ? 2 : 1;
    const bool mixed = S != 1 && g.scope && g.flags[1] && g.flags[2];     // (else every tile is this kernel's)
    auto state_of = [&](int tile) {
        if (!mixed || tile >= num_tiles) return MINE;
        int mb, nb;
        coords(tile, mb, nb);
        return g.state[g.scope == ROWS ? mb : g.scope == COLUMNS ? nb : 0];
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < XSTAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int q = 0; q < 2; ++q) { mbar_init(&acc_full[q], 1); mbar_init(&acc_empty[q], XT<S>::EPI); }
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
            int ahead = state_of(blockIdx.x);
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
                const int now = ahead;
                ahead = state_of(tile + gridDim.x);
                if (!(now & MINE)) continue;
                int mb, nb;
                coords(tile, mb, nb);
                for (int kb = 0; kb < num_kb; ++kb) {
                    ok = mbar_wait(&empty[stage], phase ^ 1, abort_flag, g.status);
                    if (!ok) break;
                    uint8_t* st = smem + stage * XSTAGE;
                    mbar_expect_tx(&full[stage], XSTAGE);
                    tma_load_4d(st, &tmA, 0, mb * (XM / 4), 0, kb * XKB, &full[stage]);
                    tma_load_4d(st + XKB * XP * XA_TILE, &tmB, 0, nb * (XN / 4), 0, kb * XKB, &full[stage]);
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
            int done = 0;               // tiles
            bool ok = true;
            int ahead = state_of(blockIdx.x);
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
                const int now = ahead;
                ahead = state_of(tile + gridDim.x);
                if (!(now & MINE)) continue;
                ++done;
                for (int kb = 0; kb < num_kb; ++kb) {
                    const bool run_start = kb % XRUN == 0;
                    const bool run_end = (kb + 1) % XRUN == 0 || kb + 1 == num_kb;
                    ok = mbar_wait(&full[stage], phase, abort_flag, g.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t dbase = smem_desc32(smem_u32(smem + stage * XSTAGE));
                    auto issue = [&](int group) {
#pragma unroll
                        for (int kk = 0; kk < XKB; ++kk) {
#pragma unroll
                            for (int t = 0; t < xins_count<S>(); ++t) {
                                const XIns in = xins<S>(t);
                                if (in.group != group) continue;
                                const uint32_t acc = ((t == 0 || t == S) && run_start && kk == 0) ? 0u : 1u;
                                const uint64_t da = dbase + (uint64_t)(((kk * XP + in.a) * XA_TILE) >> 4);
                                const uint64_t db =
                                    dbase + (uint64_t)((XKB * XP * XA_TILE + (kk * XP + in.b) * XB_TILE) >> 4);
                                mma_bf16<1>(tmem + (uint32_t)((in.a + in.b) * XN), da, db, idesc_bf16(XM, in.n * XN),
                                            acc);
                            }
                            if (XT<S>::SUM && group == 1)
                                mma_bf16<1>(tmem + (uint32_t)(S * XN), dbase + (uint64_t)(((kk * XP + S) * XA_TILE) >> 4),
                                            dbase + (uint64_t)((XKB * XP * XA_TILE + (kk * XP + S) * XB_TILE) >> 4),
                                            idesc_bf16(XM, XN), (kb == 0 && kk == 0) ? 0u : 1u);
                        }
                    };
                    if (run_start && run_no > 0) {
                        ok = mbar_wait(&acc_empty[1], (run_no - 1) & 1, abort_flag, g.status);
                        if (!ok) break;
                        tc_fence_after();
                    }
                    issue(1);
                    if (run_end) mma_commit<1>(&acc_full[1]);
                    if constexpr (XL > 0) {
                        if (run_start && run_no > 0) {
                            ok = mbar_wait(&acc_empty[0], (run_no - 1) & 1, abort_flag, g.status);
                            if (!ok) break;
                            tc_fence_after();
                        }
                        issue(0);
                        if (run_end) mma_commit<1>(&acc_full[0]);
                    }
                    mma_commit<1>(&empty[stage]);
                    if (run_end) ++run_no;
                    if (++stage == XSTAGES) { stage = 0; phase ^= 1; }
                }
            }
            if (S != 1 && g.flops && done) atomicAdd(g.flops, done * g.tile_flops);
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
            // (read under the tile's first run of products)
            const int now = state_of(tile);
            if (!(now & MINE)) continue;
            int mb, nb;
            coords(tile, mb, nb);
            if constexpr (S == 1) {
                // the sums of |a||b|: which are small, or outside the digits' range?
                const int row = mb * XM + quad * 32 + lane, col0 = nb * XN + colq * XCPT;
                const bool row_out = row < g.M && field_outside(g.fa[row]);
                unsigned col_out = 0;        // bit h: column col0 + 32 h + lane
#pragma unroll
                for (int h = 0; h < XCPT / 32; ++h)
                    if (col0 + h * 32 + lane < g.N && field_outside(g.fb[col0 + h * 32 + lane])) col_out |= 1u << h;
                int w_ok = 1;
                if (lane == 0) w_ok = mbar_wait(&acc_full[1], run_no & 1, abort_flag, g.status, g.acc_wait_ns) ? 1 : 0;
                ok = __shfl_sync(0xffffffffu, w_ok, 0) != 0;
                if (!ok) break;
                tc_fence_after();
                bool small = row_out;
#pragma unroll
                for (int h = 0; h < XCPT / 8; ++h) {
                    uint32_t r[8];
                    tmem_ld8(tmem + lane_base + (uint32_t)(colq * XCPT + h * 8), r);
                    tmem_wait_ld();
                    tmem_arrived(r);
                    if (g.scope == COLUMNS) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (__any_sync(0xffffffffu, row_out || sum_below(r[j], SUM9_MIN)) && lane == j &&
                                col0 + h * 8 + j < g.N)
                                g.need[col0 + h * 8 + j] = 1;
                    } else {
#pragma unroll
                        for (int j = 0; j < 8; ++j) small |= sum_below(r[j], SUM9_MIN);
                    }
                }
                tc_fence_before();
                if (g.scope == COLUMNS) {
#pragma unroll
                    for (int h = 0; h < XCPT / 32; ++h)
                        if (col_out >> h & 1u) g.need[col0 + h * 32 + lane] = 1;
                } else {
                    small |= __any_sync(0xffffffffu, col_out != 0);    // (every row meets that column)
                }
                if (g.scope == ROWS && small && row < g.M) g.need[row] = 1;
                if (g.scope == WHOLE && small) g.need[0] = 1;
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[1]);
                ++run_no;
            } else {
            const int nruns = (num_kb + XRUN - 1) / XRUN;
            long long w[XCPT][XT<S>::LIMBS];
#pragma unroll
            for (int j = 0; j < XCPT; ++j)
#pragma unroll
                for (int q = 0; q < XT<S>::LIMBS; ++q) w[j][q] = 0;
            // The columns of this thread's row that this kernel stores, kept in the
            // store staging until they are needed: the sums take the registers.
            uint32_t* const keep_slot = (uint32_t*)(staging + ew * (32 * 8)) + lane;
            if (mixed) {
                unsigned k = ~0u;
                const int i = g.scope == ROWS ? mb * XM + quad * 32 + lane : nb * XN + colq * XCPT + lane;
                const bool in = g.scope == ROWS ? i < g.M : lane < XCPT && i < g.N;
                if (now != MINE && g.scope != WHOLE) {
                    const bool mine = in && (g.need[i] != 0) == (S == 15);
                    k = g.scope == ROWS ? (mine ? ~0u : 0u) : __ballot_sync(0xffffffffu, mine);
                }
                *keep_slot = k;
            }
            unsigned weak = 0;      // columns of this thread's row that 15 digits do not suffice for
            for (int c = 0; c < nruns && ok; ++c, ++run_no) {
#pragma unroll
                for (int grp = 1; grp >= 0; --grp) {
                    int w_ok = 1;
                    if (lane == 0) w_ok = mbar_wait(&acc_full[grp], run_no & 1, abort_flag, g.status, g.acc_wait_ns) ? 1 : 0;
                    ok = __shfl_sync(0xffffffffu, w_ok, 0) != 0;
                    if (!ok) break;
                    tc_fence_after();
                    // two D's at a time
#pragma unroll
                    for (int d = grp ? XL : 0; d < (grp ? S : XL); d += 2) {
                        uint32_t r[2][XCPT];
                        const uint32_t src = tmem + lane_base + (uint32_t)(d * XN + colq * XCPT);
                        tmem_ldn(src, r[0]);
                        if (d + 1 < S) tmem_ldn(src + XN, r[1]);
                        tmem_wait_ld();
                        tmem_arrived(r[0]);
                        if (d + 1 < S) tmem_arrived(r[1]);
                        constexpr long long TERM = (long long)XRUN * XK << 14;       // |D_d| <= (d + 1) TERM
                        const int q = S == 9 && d == 8 ? 1 : d >> 2;
                        const int last = S == 9 && d >= 4 ? 8 : d >= 12 ? 14 : (d | 3);
#pragma unroll
                        for (int j = 0; j < XCPT; ++j) {
                            const int x = __float2int_rn(__uint_as_float(r[0][j]));
                            const int y = d + 1 < S ? __float2int_rn(__uint_as_float(r[1][j])) : 0;
                            if (d + 1 == S) w[j][q] += x;
                            else if ((d + 1) * TERM * 256 + (d + 2) * TERM < (1ll << 31))
                                w[j][q] += (long long)(x * 256 + y) * (1ll << (8 * (last - d - 1)));
                            else
                                w[j][q] += (long long)x * (1ll << (8 * (last - d))) + (long long)y * (1ll << (8 * (last - d - 1)));
                        }
                    }
                    if constexpr (XT<S>::SUM) {
                        if (grp == 1 && c == nruns - 1) {
                            uint32_t r[XCPT];
                            tmem_ldn(tmem + lane_base + (uint32_t)(S * XN + colq * XCPT), r);
                            tmem_wait_ld();
                            tmem_arrived(r);
#pragma unroll
                            for (int j = 0; j < XCPT; ++j) weak |= sum_below(r[j], SUM15_MIN) ? 1u << j : 0u;
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[grp]);
                }
            }
            if (!ok) break;
            const bool second = g.half && mb * XM >= g.half;
            const int r0 = second ? g.half : 0;
            double* const C = second ? g.C1 : g.C;
            const int64_t* const c_m = second ? g.c_m1 : g.c_m;
            const int64_t* const c_n = second ? g.c_n1 : g.c_n;
            const int m = mb * XM + quad * 32 + lane - r0;
            const bool row_ok = m < g.M;
            const int nt = nb * XN + colq * XCPT - r0;
            // the warp's columns are the same for every lane: lane j loads
            // column j's exponent and offset, the loop takes them by shuffle
            const bool col_in = lane < XCPT && nt + lane < g.N;
            const int fb = col_in ? g.fb[nt + lane + r0] : 0;
            const long long cn_l = col_in ? (long long)c_n[nt + lane] : 0;
            const unsigned keep = mixed ? *(volatile uint32_t*)keep_slot : ~0u;
            __syncwarp();            // (the staging is written below)
            const int fa = row_ok ? g.fa[m + r0] : 0;
            const int ea = max(fa, 1) - 1022;
            if constexpr (XT<S>::SUM) {
                weak |= __ballot_sync(0xffffffffu, field_outside(fb));
                if (field_outside(fa)) weak = ~0u;
                // of the elements that are stored
                weak = row_ok ? weak & keep : 0u;
                weak &= (1u << max(0, min(XCPT, g.N - nt))) - 1u;
                if (g.sym) weak &= ~0u << max(0, min(XCPT, m - nt));
                static_assert(!XT<S>::SUM || (XN == 32 && XCPT == 8), "a byte of a word per thread");
                ((uint8_t*)g.weak)[((size_t)nb * g.weak_rows + mb * XM + quad * 32 + lane) * 4 + colq] = (uint8_t)weak;
                if (__any_sync(0xffffffffu, weak != 0) && lane == 0) g.weak_tile[mb * g.words + nb] = g.flags[0] = 1;
            }
            const int eb_l = max(fb, 1) - 1022 - 14 - 8 * (S - 1);
            if (g.rows_fast) {
                // lanes are adjacent rows, adjacent in C
                double* cp = C + (row_ok ? c_m[m] : 0);
#pragma unroll
                for (int j = 0; j < XCPT; ++j) {
                    const int e2 = ea + __shfl_sync(0xffffffffu, eb_l, j);
                    const long long cn = __shfl_sync(0xffffffffu, cn_l, j);
                    if (row_ok && nt + j < g.N && (keep >> j & 1u)) cp[cn] = wide_to_double(w[j], e2);
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
                const int64_t cm_mirror = c_n[m];
#pragma unroll
                for (int j = 0; j < XCPT; ++j) {
                    const int n = nt + j;
                    if (n < g.N && n > m && (keep >> j & 1u)) C[c_m[n] + cm_mirror] = v[j];
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
                    const int mr = mb * XM + quad * 32 + rr - r0;
                    const unsigned kr = __shfl_sync(0xffffffffu, keep, rr);
                    if (mr < g.M && n < g.N && (!g.sym || n >= mr) && (kr >> (pass * 8 + cl) & 1u))
                        C[c_m[mr] + cn] = stg[rr * 8 + (cl ^ ((rr >> 1) & 7))];
                }
                __syncwarp();
            }
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

// ---------------------------------------------- elements left to the pipe ---
// C(m, n) of the elements that the digit product marked weak, as FP64 sums in
// order of k, the bits of k_gemm_f64.  A block takes R x 32 elements at a time,
// lists the marked ones and gives each thread up to sixteen (eight) of them, so
// its time follows their number; operands are staged as in k_gemm_f64.  Bound by
// the FP64 pipe: one FMA of a warp takes 16 clocks there, the two operands from
// shared memory about four.  R = 128 where that gives every SM eight blocks'
// worth, 32 for smaller products, whose marks lie unevenly: late in an off-critical
// solve at Dcut 24 the D^7 product takes 1.99 ms with 128 and 2.25 with 32, P and Q
// in one launch 0.35 and 0.22.
struct WeakArgs {
    int M, N, K, sym, half;
    const double* A[2]; const int64_t* a_m[2]; const int64_t* a_k[2]; int a_kfast[2];
    const double* B[2]; const int64_t* b_k[2]; const int64_t* b_n[2]; int b_nfast[2];
    double* C[2]; const int64_t* c_m[2]; const int64_t* c_n[2];
    const int* any;
    const int* tile;           // [tiles_m][words]
    const uint32_t* weak;      // [words][rows]
    int tiles_m, words, rows;
};
constexpr int WS = 32, WK = 16;                 // columns, K per stage
template <int R>
__global__ void __launch_bounds__(R == 32 ? 128 : 256, 2) k_weak_f64(const WeakArgs g) {
    constexpr int WT = R == 32 ? 128 : 256;     // threads
    constexpr int WE = R * WS / WT;             // elements a thread can be given
    if (*g.any == 0) return;
    __shared__ double As[WK][R + 1];
    __shared__ double Bs[WK][WS + 1];
    __shared__ uint16_t list[R * WS];           // row << 5 | column
    __shared__ int warp_count[R / 32];
    const int tid = threadIdx.x;
    for (int t = blockIdx.x; t < g.tiles_m * g.words * (XM / R); t += gridDim.x) {
        const int tile = t / (XM / R), row0 = tile / g.words * XM + t % (XM / R) * R, w = tile % g.words;
        if (!g.tile[tile]) continue;
        const int q = g.half && row0 >= g.half ? 1 : 0;
        const int m0 = row0 - (q ? g.half : 0), n0 = w * WS - (q ? g.half : 0);
        __syncthreads();                        // the previous list has been used
        uint32_t bits = 0;
        int at = 0;
        if (tid < R) {
            if (m0 + tid < g.M) bits = g.weak[(size_t)w * g.rows + row0 + tid];
            const int cols = g.N - n0;
            if (cols < WS) bits &= (1u << max(cols, 0)) - 1u;
            // place of this row's elements in the list: first within the warp
            at = __popc(bits);
#pragma unroll
            for (int o = 1; o < 32; o *= 2) {
                const int v = __shfl_up_sync(0xffffffffu, at, o);
                if ((tid & 31) >= o) at += v;
            }
            if ((tid & 31) == 31) warp_count[tid >> 5] = at;
            at -= __popc(bits);
        }
        __syncthreads();
        int n = 0;
#pragma unroll
        for (int i = 0; i < R / 32; ++i) {
            if (i < tid >> 5) at += warp_count[i];
            n += warp_count[i];
        }
        for (; bits; bits &= bits - 1) list[at++] = (uint16_t)(tid << 5 | (__ffs((int)bits) - 1));
        __syncthreads();
        if (n == 0) continue;
        int el[WE];
        double acc[WE];
#pragma unroll
        for (int e = 0; e < WE; ++e) {
            el[e] = tid + e * WT < n ? list[tid + e * WT] : 0;
            acc[e] = 0.0;
        }
        double ra[R * WK / WT], rb[WS * WK / WT];
        auto load = [&](int k0) {
#pragma unroll
            for (int i = 0; i < R * WK / WT; ++i) {
                const int e = tid + i * WT;
                const int r = g.a_kfast[q] ? e / WK : e % R, k = k0 + (g.a_kfast[q] ? e % WK : e / R);
                ra[i] = m0 + r < g.M && k < g.K ? g.A[q][g.a_m[q][m0 + r] + g.a_k[q][k]] : 0.0;
            }
#pragma unroll
            for (int i = 0; i < WS * WK / WT; ++i) {
                const int e = tid + i * WT;
                const int c = g.b_nfast[q] ? e % WS : e / WK, k = k0 + (g.b_nfast[q] ? e / WS : e % WK);
                rb[i] = n0 + c < g.N && k < g.K ? g.B[q][g.b_k[q][k] + g.b_n[q][n0 + c]] : 0.0;
            }
        };
        load(0);
        for (int k0 = 0; k0 < g.K; k0 += WK) {
            __syncthreads();
#pragma unroll
            for (int i = 0; i < R * WK / WT; ++i) {
                const int e = tid + i * WT;
                if (g.a_kfast[q]) As[e % WK][e / WK] = ra[i]; else As[e / R][e % R] = ra[i];
            }
#pragma unroll
            for (int i = 0; i < WS * WK / WT; ++i) {
                const int e = tid + i * WT;
                if (g.b_nfast[q]) Bs[e / WS][e % WS] = rb[i]; else Bs[e % WK][e / WK] = rb[i];
            }
            __syncthreads();
            if (k0 + WK < g.K) load(k0 + WK);
#pragma unroll
            for (int e = 0; e < WE; ++e) {
                if ((tid & ~31) + e * WT >= n) break;       // (the same for the warp)
                const int r = el[e] >> 5, c = el[e] & 31;
#pragma unroll
                for (int kk = 0; kk < WK; ++kk) acc[e] = fma(As[kk][r], Bs[kk][c], acc[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < WE; ++e) {
            if (tid + e * WT >= n) break;
            const int m = m0 + (el[e] >> 5), c = n0 + (el[e] & 31);
            g.C[q][g.c_m[q][m] + g.c_n[q][c]] = acc[e];
            if (g.sym && c > m) g.C[q][g.c_m[q][c] + g.c_n[q][m]] = acc[e];
        }
    }
}

// Which tiles hold rows (columns) that need 15 digits (1) and which hold others
// (2): out9 for the tiles of the nine-digit kernel, t9 rows (columns) long, out15
// for the other's; flags[1] and flags[2] for all of them.
__global__ void __launch_bounds__(256) k_need_tiles(const int* need, int count, int t9, int* out9, int t15, int* out15,
                                                    int* flags) {
    const int t = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;      // a warp per tile
    auto state = [&](int side) {
        unsigned s = 0;
        for (int i = t * side + lane; i < min(count, (t + 1) * side); i += 32) s |= need[i] ? 1u : 2u;
        return (int)__reduce_or_sync(0xffffffffu, s);
    };
    const int s9 = state(t9), s15 = state(t15);
    if (lane != 0) return;
    if (t * t9 < count) out9[t] = s9;
    if (t * t15 < count) {
        out15[t] = s15;
        if (s15 & 1) flags[1] = 1;
        if (s15 & 2) flags[2] = 1;
    }
}

// ------------------------------------------------------------- host side ---
// `count` planes from plane `first` on of the digits [kp / 16][XPLANES][rows][16]
// (their order in a stage: no swizzle here), four rows to a 128-byte line,
// boxes of box_rows rows and box_k K of all of them.
CUtensorMap digit_map(const uint16_t* base, int first, int count, int64_t rows, int kp, int box_rows, int box_k) {
    CUtensorMap m;
    std::memset(&m, 0, sizeof(m));
    const cuuint64_t dims[4] = {64, (cuuint64_t)rows / 4, (cuuint64_t)count, (cuuint64_t)kp / 16};
    const cuuint64_t strides[3] = {128, (cuuint64_t)rows * 32, (cuuint64_t)rows * 32 * XPLANES};
    const cuuint32_t box[4] = {64, (cuuint32_t)box_rows / 4, (cuuint32_t)count, (cuuint32_t)box_k / 16};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<uint16_t*>(base + (size_t)first * rows * 16),
                             dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) fail(TRG_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
    return m;
}

inline int64_t up(int64_t v, int64_t q) { return (v + q - 1) / q * q; }

// Exponent fields and digits of rows [0, R) of an operand, as rows of an array
// of Rs.
void digits(Ctx& ctx, const Gather& g, int R, int K, int Rp, int Kp, int* ef, uint16_t* out, int Rs) {
    if (g.c_identity && Kp <= CUT_ROWS4_MAX_K) {
        launch_cut_rows4(ctx.stream, g.base, g.off_r, R, K, Rp, Kp, ef, out, Rs);
        TRG_LAUNCHED(ctx);
        return;
    }
    TRG_CUDA(cudaMemsetAsync(ef, 0, (size_t)R * sizeof(int), ctx.stream));
    launch_row_field<true>(ctx.stream, g, R, K, ef);
    TRG_LAUNCHED(ctx);
    launch_cut<15>(ctx.stream, g, R, K, Rp, Kp, ef, nullptr, out, Rs);
    TRG_LAUNCHED(ctx);
}

// Tiles (128 rows, xn columns) that reach the diagonal or above it, and those of
// a second product whose rows start at half.
const long long* diagonal_tiles(Ctx& ctx, int tiles_m, int tiles_n, int xn, int half, int& n) {
    const std::string key = "xsym:" + std::to_string(tiles_m) + ":" + std::to_string(tiles_n) + ":" +
                            std::to_string(xn) + ":" + std::to_string(half);
    auto it = ctx.lists.find(key);
    if (it == ctx.lists.end()) {
        std::vector<long long> h;
        for (int mb = 0; mb < tiles_m; ++mb)
            for (int nb = 0; nb < tiles_n; ++nb)
                if ((int64_t)nb * xn + xn - 1 >= (int64_t)mb * XM) h.push_back(((long long)mb << 32) | nb);
        for (size_t i = 0, one = h.size(); half && i < one; ++i)
            h.push_back(h[i] + ((long long)(half / XM) << 32) + half / xn);
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

// Rows of the operands whose digits are held at a time (multiples of the tile;
// B's of XNP): at most cap bytes of them, half of it for either, and a weak bit
// for an element of C in at most a 64th of that.  One tile of each is the least;
// below XCAP_MIN the tiles of a block (256 at K = 4096) no longer fill the SMs, so
// less is taken only where more cannot be had.
constexpr int64_t XCAP = (int64_t)2 << 30, XCAP_MIN = (int64_t)256 << 20;
constexpr int64_t XNP = 64;
struct XBlock { int64_t a, b; };
XBlock block_rows(int64_t M, int64_t N, int64_t kp, int64_t cap) {
    const int64_t most = cap / 2 / (2 * XPLANES * kp);
    XBlock x;
    x.a = std::min(up(M, XM), std::max<int64_t>(XM, most / XM * XM));
    x.b = std::min(up(N, XNP), std::max<int64_t>(XNP, std::min(most, cap / 8 / x.a) / XNP * XNP));
    return x;
}
// Bytes of the flags, the weak tiles and the weak bits of an a x b block.
int64_t flag_bytes(int64_t a, int64_t b) { return up(256 + 4 * (a / XM) * (up(b, 32) / 32), 256); }
int64_t weak_bytes(int64_t a, int64_t b) { return 4 * a * (up(b, 32) / 32); }
// ... and of need[] and state[] of a product of M x N in such blocks.
int64_t need_bytes(int64_t M, int64_t N) { return 4 * std::max(M, N); }
int64_t state_bytes(int64_t a, int64_t b) { return 4 * (std::max(a, b) / 32 + 1); }

}  // namespace

int64_t exact_cap(size_t workspace_bytes) {
    return std::min(XCAP, std::max(XCAP_MIN, workspace_bytes ? (int64_t)workspace_bytes : XCAP));
}

int64_t exact_scratch_bytes(int64_t M, int64_t N, int64_t K, int64_t cap) {
    const int64_t kp = up(std::max<int64_t>(K, 1), XKP);
    const XBlock x = block_rows(M, N, kp, cap);
    return 2 * XPLANES * kp * (x.a + x.b) + 4 * (x.a + x.b) + flag_bytes(x.a, x.b) + weak_bytes(x.a, x.b) +
           need_bytes(M, N) + 2 * state_bytes(x.a, x.b) + 4096;
}

int64_t exact_pair_scratch_bytes(int64_t M, int64_t K) {
    const int64_t kp = up(std::max<int64_t>(K, 1), XKP), rows = 2 * up(M, XM);
    return 2 * XPLANES * kp * rows + 4 * rows + flag_bytes(rows, rows) + weak_bytes(rows, rows) + 2048;
}

namespace {
double tiles_of(int64_t M, int64_t N, int xn, bool sym) {
    const double tm = (double)up(M, XM) / XM, tn = (double)up(N, xn) / xn;
    return sym ? 0.5 * tm * (tn + 128.0 / xn) : tm * tn;
}
double us15(const Ctx& ctx, int64_t M, int64_t N, int64_t K, bool sym) {
    return std::ceil(tiles_of(M, N, XT<15>::N, sym) / ctx.sm_count) * (std::ceil((double)K / 64.0) * 4.4 + 3.0);
}
// Whether to look for the nine-digit form: the check and the three more launches
// have to be made good.
bool try_nine(const Ctx& ctx, int64_t M, int64_t N, int64_t K, bool sym) {
    if (K > XNINE_K) return false;
    const double nine = std::ceil(tiles_of(M, N, XT<9>::N, sym) / ctx.sm_count) * (std::ceil((double)K / 96.0) * 3.8 + 3.0);
    const double check = std::ceil(tiles_of(M, N, XT<1>::N, sym) / ctx.sm_count) * (std::ceil((double)K / 32.0) * 0.35 + 1.0);
    return nine + check + 16.0 < us15(ctx, M, N, K, sym);
}
}  // namespace

double exact_us(const Ctx& ctx, int64_t M, int64_t N, int64_t K, bool sym) {
    if (M > (1ll << 30) || N > (1ll << 30) || K > (1 << 17)) return 1e300;
    const double moved = (46.0 * (double)K * ((double)M + (sym ? 0.0 : (double)N)) + 8.0 * (double)M * (double)N) / 4.0e6;
    return 25.0 + us15(ctx, M, N, K, sym) + moved;
}

namespace {

// The kernel for S digits (S = 1: the sums of |a||b|) on the cut planes.
template <int S>
void launch_exact(Ctx& ctx, const uint16_t* sa, int64_t mp, const uint16_t* sb, int64_t np, XArgs a) {
    constexpr int first = S == 1 ? 15 : 0;
    static PerDevice prepared;
    prepared.get(ctx.device, [] {
        TRG_CUDA(cudaFuncSetAttribute(k_exact_mma<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, XT<S>::SMEM));
        return 0;
    });
    const CUtensorMap ta = digit_map(sa, first, XT<S>::P, mp, a.Kp, XM, XT<S>::K);
    const CUtensorMap tb = digit_map(sb, first, XT<S>::P, np, a.Kp, XT<S>::N, XT<S>::K);
    const int tiles_m = (a.M + XM - 1) / XM, tiles_n = (a.N + XT<S>::N - 1) / XT<S>::N;
    int tiles = tiles_m * tiles_n;
    a.acc_wait_ns = ctx.acc_wait_ns ? ctx.acc_wait_ns : WAIT_NS;
    a.tile_list = nullptr;
    a.n_list = 0;
    if (a.sym) {
        a.tile_list = diagonal_tiles(ctx, tiles_m, tiles_n, XT<S>::N, a.half, a.n_list);
        tiles = a.n_list;
    }
    // (which tiles are computed is decided on the device)
    a.flops = ctx.device_flops();
    a.tile_flops = S * (S + 1) / 2 * 2.0 * XM * XT<S>::N * a.Kp;
    // column blocks whose digits share L2 (about 40 MB of them)
    a.group_n = (int)std::max<int64_t>(1, std::min<int64_t>(tiles_n, (40ll << 20) / ((int64_t)XT<S>::N * a.Kp * 2 * S)));
    k_exact_mma<S><<<std::min(tiles, ctx.sm_count), XT<S>::THREADS, XT<S>::SMEM, ctx.stream>>>(ta, tb, a);
    TRG_LAUNCHED(ctx);
}

// The weak elements of the block at (m0, n0) of d0 (and of d1, for a pair).
void launch_weak(Ctx& ctx, const GemmDesc& d0, const GemmDesc& d1, int64_t m0, int64_t n0, const XArgs& a) {
    WeakArgs w;
    w.M = a.M; w.N = a.N; w.K = (int)d0.K; w.sym = a.sym; w.half = a.half;
    const GemmDesc* d[2] = {&d0, &d1};
    for (int q = 0; q < 2; ++q) {
        w.A[q] = d[q]->A.base; w.a_m[q] = d[q]->A.off_r + m0; w.a_k[q] = d[q]->A.off_c; w.a_kfast[q] = d[q]->A.c_fast;
        w.B[q] = d[q]->B.base; w.b_k[q] = d[q]->B.off_r; w.b_n[q] = d[q]->B.off_c + n0; w.b_nfast[q] = d[q]->B.c_fast;
        w.C[q] = d[q]->C; w.c_m[q] = d[q]->c_m + m0; w.c_n[q] = d[q]->c_n + n0;
    }
    w.any = a.flags; w.tile = a.weak_tile; w.weak = a.weak;
    w.tiles_m = (a.half + a.M + XM - 1) / XM; w.words = a.words; w.rows = a.weak_rows;
    const int tiles = w.tiles_m * w.words;
    if (tiles >= 8 * ctx.sm_count) k_weak_f64<128><<<4 * ctx.sm_count, 256, 0, ctx.stream>>>(w);
    else k_weak_f64<32><<<std::min(4 * tiles, 8 * ctx.sm_count), 128, 0, ctx.stream>>>(w);
    TRG_LAUNCHED(ctx);
}

}  // namespace

bool gemm_exact(Ctx& ctx, const GemmDesc& d) {
    const int K = (int)std::max<int64_t>(d.K, 1), Kp = (int)up(K, XKP);
    const ScratchUse use(ctx);
    // smaller blocks where there is no room for these (the bits are the same)
    XBlock blk;
    for (int64_t cap = ctx.digit_bytes ? (int64_t)ctx.digit_bytes : exact_cap(ctx.cfg.workspace_bytes);; cap /= 2) {
        blk = block_rows(d.M, d.N, Kp, cap);
        try {
            ctx.ensure(ctx.split_ws, (size_t)exact_scratch_bytes(d.M, d.N, K, cap));
            break;
        } catch (const Error& e) {
            if (e.status != TRG_ENOMEM) throw;
            if (blk.a <= XM && blk.b <= XNP) return false;    // not even for a tile: the FP64 pipe needs none
        }
    }
    const int64_t ra = blk.a, rb = blk.b;
    const bool sym = d.gram && d.M == d.N && ra >= d.M && rb >= d.N;
    uint8_t* p = ctx.split_ws.as<uint8_t>();
    auto take = [&](size_t bytes) { uint8_t* q = p; p += (bytes + 255) & ~(size_t)255; return q; };
    int* flags = (int*)take((size_t)flag_bytes(ra, rb));
    int* need = (int*)take((size_t)need_bytes(d.M, d.N));     // (cleared with the flags)
    uint32_t* weak = (uint32_t*)take((size_t)weak_bytes(ra, rb));
    int* fa = (int*)take((size_t)ra * 4);
    int* fb = sym ? fa : (int*)take((size_t)rb * 4);
    int* state9 = (int*)take((size_t)state_bytes(ra, rb));
    int* state15 = (int*)take((size_t)state_bytes(ra, rb));
    uint16_t* sa = (uint16_t*)take((size_t)(2 * XPLANES) * ra * Kp);
    uint16_t* sb = sym ? sa : (uint16_t*)take((size_t)(2 * XPLANES) * rb * Kp);

    // Nine digits or fifteen: one decision for a row (a column, if the product is
    // a slab of columns), so that it is the same from every slab and block; one
    // for all of a Gram product, which is symmetric.
    const int scope = !try_nine(ctx, d.choice_m(), d.choice_n(), K, d.gram) ? NONE : d.gram ? WHOLE : d.whole_n ? COLUMNS : ROWS;
    TRG_CUDA(cudaMemsetAsync(flags, 0, (size_t)(flag_bytes(ra, rb) + (scope ? need_bytes(d.M, d.N) : 0)), ctx.stream));
    bool cleared = true;      // the flags, for the next block
    const bool one_a = ra >= d.M, one_b = rb >= d.N;      // (an operand cut once)
    const bool check_first = scope && !(one_a && one_b) && !(scope == ROWS && one_b) && !(scope == COLUMNS && one_a);
    // B as rows n, columns k
    const Gather bt = transposed(d.B);
    auto blocks = [&](bool check, bool products) {
        for (int64_t m0 = 0; m0 < d.M; m0 += ra) {
            const int mr = (int)std::min(ra, d.M - m0), mp = (int)up(mr, XM);
            Gather ga = d.A;
            ga.off_r += m0;
            digits(ctx, ga, mr, K, mp, Kp, fa, sa, mp);
            for (int64_t n0 = 0; n0 < d.N; n0 += rb) {
                const int nr = (int)std::min(rb, d.N - n0), np = sym ? mp : (int)up(nr, XNP);
                if (!sym && (m0 == 0 || !one_b)) {
                    Gather gb = bt;
                    gb.off_r += n0;
                    digits(ctx, gb, nr, K, np, Kp, fb, sb, np);
                }
                XArgs a;
                a.M = mr; a.N = sym ? mr : nr; a.Kp = Kp;
                a.fa = fa; a.fb = fb;
                a.C = d.C; a.c_m = d.c_m + m0; a.c_n = d.c_n + n0;
                a.rows_fast = d.c_m_fast && !sym ? 1 : 0;
                a.sym = sym ? 1 : 0;
                a.half = 0;
                a.flags = flags; a.status = ctx.gave_up;
                a.weak = weak; a.weak_tile = flags + 64; a.weak_rows = mp; a.words = (a.N + 31) / 32;
                a.scope = scope;
                a.need = need + (scope == ROWS ? m0 : scope == COLUMNS ? n0 : 0);
                a.state = nullptr;
                if (check) launch_exact<1>(ctx, sa, mp, sb, np, a);
                if (!products) continue;
                if (!cleared) TRG_CUDA(cudaMemsetAsync(flags, 0, (size_t)flag_bytes(mp, a.N), ctx.stream));
                cleared = false;
                const int tok = ctx.region_begin(TRG_PHASE_MMA);
                if (scope) {
                    const int count = scope == ROWS ? mr : scope == COLUMNS ? nr : 1;
                    const int t9 = scope == COLUMNS ? XT<9>::N : XM, t15 = scope == COLUMNS ? XT<15>::N : XM;
                    const int tiles = (count + t15 - 1) / t15;
                    k_need_tiles<<<(tiles + 7) / 8, 256, 0, ctx.stream>>>(a.need, count, t9, state9, t15, state15, flags);
                    TRG_LAUNCHED(ctx);
                    a.state = state9;
                    launch_exact<9>(ctx, sa, mp, sb, np, a);
                    a.state = state15;
                }
                launch_exact<15>(ctx, sa, mp, sb, np, a);
                ctx.region_end(tok, 2.0 * (double)mr * nr * K, 0.0);    // (the kernels add their digit products)
                launch_weak(ctx, d, d, m0, n0, a);
            }
        }
    };
    if (check_first) blocks(true, false);
    blocks(scope && !check_first, true);
    return true;
}

// Two Gram products of one size whose tiles fit the chip together (the P and Q
// of an environment): one launch, which takes as long as either alone.  At (24,
// 22), 2 x 55 tiles on 152 SMs, the environment takes 228 us instead of 300.
bool gemm_exact_pair(Ctx& ctx, const GemmDesc& d0, const GemmDesc& d1) {
    const int64_t M = d0.M, K = std::max<int64_t>(d0.K, 1);
    if (!(d0.gram && d1.gram && d0.N == M && d1.M == M && d1.N == M && d1.K == d0.K)) return false;
    if (2 * tiles_of(M, M, XT<15>::N, true) > ctx.sm_count || try_nine(ctx, M, M, K, true)) return false;
    const int Kp = (int)up(K, XKP), mp = (int)up(M, XM);
    static_assert(XM % XT<15>::N == 0, "the second product starts on a column tile");
    const ScratchUse use(ctx);
    if (ctx.digit_bytes && exact_pair_scratch_bytes(M, K) > (int64_t)ctx.digit_bytes) return false;
    try {
        ctx.ensure(ctx.split_ws, (size_t)exact_pair_scratch_bytes(M, K));
    } catch (const Error& e) {
        if (e.status == TRG_ENOMEM) return false;
        throw;
    }
    const int phase = ctx.region_begin(ctx.phase);
    uint8_t* p = ctx.split_ws.as<uint8_t>();
    auto take = [&](int64_t bytes) { uint8_t* q = p; p += up(bytes, 256); return q; };
    int* flags = (int*)take(flag_bytes(2 * mp, 2 * mp));
    uint32_t* weak = (uint32_t*)take(weak_bytes(2 * mp, 2 * mp));
    int* f = (int*)take((int64_t)2 * mp * 4);
    uint16_t* s = (uint16_t*)p;
    TRG_CUDA(cudaMemsetAsync(flags, 0, (size_t)flag_bytes(2 * mp, 2 * mp), ctx.stream));
    digits(ctx, d0.A, (int)M, (int)K, mp, Kp, f, s, 2 * mp);
    digits(ctx, d1.A, (int)M, (int)K, mp, Kp, f + mp, s + (size_t)mp * 16, 2 * mp);
    XArgs a;
    a.M = (int)M; a.N = (int)M; a.Kp = Kp;
    a.fa = f; a.fb = f;
    a.C = d0.C; a.c_m = d0.c_m; a.c_n = d0.c_n;
    a.C1 = d1.C; a.c_m1 = d1.c_m; a.c_n1 = d1.c_n;
    a.rows_fast = 0;
    a.sym = 1;
    a.half = mp;
    a.scope = NONE;
    a.need = nullptr;
    a.state = nullptr;
    a.flags = flags; a.status = ctx.gave_up;
    a.weak = weak; a.weak_tile = flags + 64; a.weak_rows = 2 * mp; a.words = 2 * mp / 32;
    const int tok = ctx.region_begin(TRG_PHASE_MMA);
    launch_exact<15>(ctx, s, 2 * mp, s, 2 * mp, a);
    ctx.region_end(tok, 4.0 * (double)M * M * K, 0.0);
    launch_weak(ctx, d0, d1, 0, 0, a);
    ctx.region_end(phase, 4.0 * (double)M * M * K, 0.0);
    return true;
}

}  // namespace trg
