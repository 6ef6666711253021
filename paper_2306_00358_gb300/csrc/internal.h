// Internal declarations of libtrg (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <map>
#include <string>
#include <utility>
#include <vector>

#include "per_device.h"
#include "trg.h"

namespace trg {

// ------------------------------------------------------------ errors ----
struct Error {
    int status;
    std::string msg;
};

[[noreturn]] void fail(int status, const std::string& msg);
void check_cuda(cudaError_t e, const char* what, const char* file, int line);
#define TRG_CUDA(call) ::trg::check_cuda((call), #call, __FILE__, __LINE__)
// After every launch: catch configuration errors immediately.
#define TRG_LAUNCHED(ctx) do { (ctx).launches++; ::trg::check_cuda(cudaGetLastError(), "kernel launch", __FILE__, __LINE__); } while (0)

// Device status word bits (written by kernels, read by the host at sync points).
enum : int {
    ST_BAD_NORM = 1,       // norm <= 0, NaN or inf
    ST_BAD_TRACE = 2,      // trace <= 0 or NaN
    ST_EIG_NOCONV = 4,     // Jacobi sweeps exhausted
    ST_CHOL_BREAK = 8,     // Cholesky pivot could not be repaired
    ST_TIMEOUT = 16,       // a bounded device wait ran out (in Ctx::gave_up)
    ST_BOUNDS = 32         // a checked index fell outside its buffer (skipped)
};

// ------------------------------------------------------- device memory ----
struct Buf {
    void* p = nullptr;
    size_t bytes = 0;
    template <class T> T* as() const { return static_cast<T*>(p); }
};

// A rank-4 strided view of FP64 device memory (element strides).
struct View4 {
    double* p;
    int64_t n[4];
    int64_t s[4];
};

// A rank-6 strided view (the cubic-lattice tensor t[x, x', y, y', z, z']).
struct View6 {
    double* p;
    int64_t n[6];
    int64_t s[6];
};

// A half-step between its isometry and its contraction: step k (odd = x,
// even = y), the tensor the x formulas see (T itself, or its rotation for a
// y step), the kept dimension and eigenvalues.
struct HalfPlan {
    int k = 0;
    bool xdir = true;
    int precision = 0;
    View4 r{};
    int64_t dn = 0;
    std::vector<double> lam;   // empty when U = I
};

struct Ctx {
    int device = 0;
    int sm_count = 0;
    cudaStream_t stream = nullptr;
    trg_config cfg{};
    trg_alloc_fn alloc_fn = nullptr;
    trg_free_fn free_fn = nullptr;
    void* alloc_user = nullptr;
    std::string last_error;
    uint64_t launches = 0;
    // tensor-core products: limit of the epilogue's wait for finished accumulators
    // in ns (0 = the kernels' default of 2 s); see trg_set_wait_limit
    unsigned long long acc_wait_ns = 0;
    bool no_exact = false;   // FP64 products stay on the FP64 pipe (no room for their digits)
    size_t digit_bytes = 0;  // bound on the digits' scratch (0: exact_cap of the workspace)

    // ---- solve state
    bool have_tensor = false;
    int Dx = 0, Dy = 0;
    int steps = 0;
    double beta = 0.0;
    Buf T, Tnext;          // current / next site tensor
    // a half-step split over ranks (trg_shard_begin .. trg_shard_finish)
    bool shard_pending = false;
    HalfPlan shard;
    // impure tensor (an observable inserted at one site), blocked alongside T
    bool have_impure = false;
    int model = -1, d0 = 0;    // model of the last trg_init_tensor (-1 after a raw init)
    double h_field = 0.0;
    Buf Timp, Timp_next, Timp_tmp;
    Buf M;                 // environment
    Buf U;                 // isometry (n x Dn row-major)
    Buf scal;              // device scalars, see SC_* below
    Buf status;            // device status word (int)
    // Mapped host memory that kernels write and the host reads without a copy
    // (host_slot, api.cu): set by a product whose bounded device wait ran out
    // (check_timeout), and the isometry's answers (EigBox, eig.cu).
    int* gave_up = nullptr;
    void* box = nullptr;
    std::vector<std::vector<double>> spectra;

    // ---- scratch
    Buf ws;                // contraction workspace (X1, X2 slices)
    Buf envP, envQ;        // environment intermediates
    Buf eig;               // subspace-iteration buffers
    Buf eig_small;         // m x m buffers
    Buf flags;             // per-column flags (int)
    Buf split_ws;          // tensor-core products: exponents and BF16 slices / digits of both operands
    int split_ws_users = 0;   // a product holds pointers into it (ScratchUse)
    Buf f64_partial;       // FP64 GEMM: split-K partial sums
    Buf ksplit_ws;         // split GEMM: split-K partial fixed-point sums
    Buf bslices;           // contraction: the D^7 product's B slices, shared by its j-blocks
    Buf field_ws;          // split / exact products: exponent fields of an operand's rows
    Buf cons_ef;           // exponent fields recorded by a producing product (two halves)
    Buf eig_slices;        // split mode: M sliced once per isometry solve
    Buf s3[10];            // cubic-lattice step: P1, P2, Ux, Uy, Mx, My, then A, W, C, D of the contraction
    std::map<std::vector<std::pair<int64_t, int64_t>>, Buf> tables;   // cached offset tables
    std::map<std::string, Buf> lists;      // cached tile lists
    std::map<std::string, int> list_len;   // entries of the cached tile lists

    // ---- phase timing
    bool prof = false;
    int phase = TRG_PHASE_ENV;
    struct PhaseAcc {
        double ms = 0.0, flops = 0.0, mma_flops = 0.0;
        uint64_t calls = 0;
        std::vector<std::pair<cudaEvent_t, cudaEvent_t>> pending;
    } ph[TRG_PHASE_COUNT];
    std::vector<cudaEvent_t> event_pool;
    // diagnostics: subspace iterations, Rayleigh-Ritz solves, FP32 / FP64
    // Jacobi sweeps, Cholesky-QR column repairs
    uint64_t counters[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    // Subspace iteration: power steps that reached the tolerance in the last
    // solve of each direction (x / y half-steps), used as the next plan.
    // plan of the next isometry of one direction: the products its
    // predecessor needed and that solve's smallest Ritz value theta_m
    struct EigHint { int64_t n = -1; int m = -1; int precision = -1; int products = 0; double theta_m = 0.0; };
    EigHint eig_hint[2];
    unsigned long long box_seq = 0;
    cudaEvent_t get_event();
    void take_host_slot();
    void give_host_slot(bool idle);
    // Record the start of a timed region of phase p (no-op unless profiling).
    int region_begin(int p);
    void region_end(int token, double flops, double mma_flops);
    // Where kernels add tensor-core FLOPs that only they know (TRG_PHASE_MMA);
    // null unless profiling.
    double* device_flops();
    Buf mma_flops;
    void collect_timings();

    void* raw_alloc(size_t bytes);
    void raw_free(void* p, size_t bytes);
    void ensure(Buf& b, size_t bytes);
    void release(Buf& b);
    const int64_t* table(const std::vector<std::pair<int64_t, int64_t>>& modes);
};
constexpr size_t HOST_SLOT_BYTES = 2048, HOST_SLOT_BOX = 64;    // bytes of a slot; the box's offset

// While one lives, Ctx::ensure does not give split_ws up for another buffer.
struct ScratchUse {
    Ctx& ctx;
    explicit ScratchUse(Ctx& c) : ctx(c) { ++ctx.split_ws_users; }
    ~ScratchUse() { --ctx.split_ws_users; }
    ScratchUse(const ScratchUse&) = delete;
    ScratchUse& operator=(const ScratchUse&) = delete;
};

// Device scalar slots (doubles) in Ctx::scal.
enum : int {
    SC_LOGNORM = 0,   // sum_k 2^-k ln n_k
    SC_LN_N0 = 1,     // ln n0
    SC_NORM = 2,      // last max|T| (as the bits of a non-negative double)
    SC_TRACE = 3,     // last trace
    SC_RES = 4,       // max Ritz residual / lambda_1 (subspace iteration)
    SC_TRACE_IMP = 5, // last trace of the impure tensor
    SC_COUNT = 8
};

// ------------------------------------------------------------ GEMM ----
// C[c_m[m] + c_n[n]] = sum_k A[a_m[m] + a_k[k]] * B[b_k[k] + b_n[n]]  (+ beta*C)
// Offset tables (int64, elements) make any strided multi-index layout a
// plain matrix for the kernels.
struct Gather {
    const double* base;
    const int64_t* off_r;   // row offsets   (A: m, B: k, C: m)
    const int64_t* off_c;   // col offsets   (A: k, B: n, C: n)
    bool c_fast;            // consecutive columns are adjacent in memory
    bool c_identity = false;   // off_c[k] == k: every row is one contiguous run
    bool r_fast = false;       // consecutive rows are adjacent in memory
    bool r_identity = false;   // off_r[r] == r
};
struct GemmDesc {
    int64_t M, N, K;
    Gather A, B;
    double* C;
    const int64_t* c_m;
    const int64_t* c_n;
    double beta = 0.0;      // 0: overwrite, 1: accumulate
    // Split mode, FP64 output through staging only: the product may split K
    // over several CTAs per tile when its tiles cannot fill the SMs (the
    // n x m products of the isometry); exact partial sums, deterministic.
    bool allow_ksplit = false;
    // FP64 mode: the product may run on the tensor cores when it is large
    // enough (gemm_exact).
    bool allow_exact = false;
    // The product is a slab, some rows (whole_m > 0) or columns (whole_n > 0), of
    // one with so many: a slice of j's of a contraction, whose extent depends on
    // the workspace and on the rank.  Choices that change bits (digits or pipe,
    // nine or fifteen of them, split K) are those of the whole product, so that
    // an element comes out the same from every slab.
    int64_t whole_m = 0, whole_n = 0;
    int64_t choice_m() const { return whole_m ? whole_m : M; }
    int64_t choice_n() const { return whole_n ? whole_n : N; }
    // consecutive rows are (mostly) adjacent in C: the epilogues store row-wise,
    // without staging.  The consumer rows cons_m + cons_n are below 2^31.
    bool c_m_fast = false;
    // Split mode only.  Producer side: record, for the product that will
    // consume C as its A operand, the largest FP64 exponent field of each of
    // its rows (row of element (m, n) = cons_m[m] + cons_n[n]) into cons_ef
    // (zeroed beforehand).  Consumer side: a_ef holds those fields for this
    // product's A rows, so the exponent pass over A is skipped.  The producer
    // stores row-wise (c_m_fast).
    int* cons_ef = nullptr;
    const int64_t* cons_m = nullptr;
    const int64_t* cons_n = nullptr;
    const int* a_ef = nullptr;
    // Split mode: A arrives sliced (split_slice_operand), for an A that several
    // products share.
    const uint16_t* a_slices = nullptr;
    const int* a_e = nullptr;
    // C = A A^T (a Gram product): B is A read the other way (B(k, n) =
    // A(n, k)), M = N, and c_m, c_n address C for either index.  Split mode
    // slices A once for both operands (when their padded sizes agree),
    // computes only the tiles that reach the diagonal or above it, and
    // writes each element above the diagonal also at its mirror position,
    // so C is exactly symmetric; so does FP64 mode.
    bool gram = false;
    // Split mode: B arrives sliced (split_slice_b), for a B that several
    // products share; the product then skips B's exponent and slicing passes.
    const uint16_t* b_slices = nullptr;
    const int* b_e = nullptr;
};
// Rows and columns of the padded slice arrays a split product of M rows and
// K columns reads for its A operand.
int64_t split_rows_padded(const Ctx& ctx, int64_t M);
int64_t split_k_padded(int64_t K);
// Slice an A operand once for several split products (GemmDesc::a_slices / a_e).
void split_slice_operand(Ctx& ctx, const Gather& A, int64_t M, int64_t K, uint16_t* slices, int* e);
// Exponents (per column n) and BF16 slices of a K x N B operand in the layout
// a split product reads: [S][split_cols_padded(N)][split_k_padded(K)].
void split_slice_b(Ctx& ctx, const Gather& B, int64_t K, int64_t N, uint16_t* slices, int* e);
int64_t split_cols_padded(int64_t N);
void gemm(Ctx& ctx, const GemmDesc& g, int precision);
void gemm_f64(Ctx& ctx, const GemmDesc& g);
double f64_us(const Ctx& ctx, int64_t M, int64_t N, int64_t K, bool sym);   // modelled time of gemm_f64
// FP64 product from exact BF16 digit products (exact_gemm.cu); false if its
// scratch cannot be had (nothing computed).
bool gemm_exact(Ctx& ctx, const GemmDesc& g);
double exact_us(const Ctx& ctx, int64_t M, int64_t N, int64_t K, bool sym);
// Bound on the digits' scratch, as a rule: the workspace's, within 256 MiB .. 2 GiB
// (2 GiB if it is not set).  How the operands are cut into blocks that fit changes
// no bit.
int64_t exact_cap(size_t workspace_bytes);
int64_t exact_scratch_bytes(int64_t M, int64_t N, int64_t K, int64_t cap);
// Two Gram products in one launch; false, with nothing computed, if they do not
// fit the chip together or their scratch cannot be had.
bool gemm_exact_pair(Ctx& ctx, const GemmDesc& d0, const GemmDesc& d1);
int64_t exact_pair_scratch_bytes(int64_t M, int64_t K);

// Table helpers: enumerate all index tuples of `modes` (size, stride),
// first mode slowest, and return the device table of offsets.
std::vector<int64_t> build_table(const std::vector<std::pair<int64_t, int64_t>>& modes);

// ------------------------------------------------------ path pieces ----
// Arithmetic of half-step `step` on a tensor whose leg dimensions multiply to
// dd (Dx Dy; Dx Dy Dz on the cubic lattice).
int precision_for_step(const Ctx& ctx, int step, int64_t dd);
// BF16 slices of the split products issued now: env_slices during the
// environment and the isometry (when set), split_slices otherwise.
int slices_now(const Ctx& ctx);
void environment(Ctx& ctx, const View4& t, double* M, int precision);
// Tx = U . top . bottom . U (the upper tensor of the blocked pair is `top`,
// the lower one `bottom`; both the same tensor for the pure half-step).
// Only the output rows j in [j_begin, j_end) are computed (j_end < 0: all);
// `out` starts at j = j_out0 (its element (i, j, k, l) is at
// (j - j_out0) s[1] + ...), so a slab of j can be written on its own.
void contract(Ctx& ctx, const View4& top, const View4& bottom, const double* U, int64_t Dn, const View4& out,
              int precision, int64_t j_begin = 0, int64_t j_end = -1, int64_t j_out0 = 0);
// Returns Dn actually kept; lam (host) gets the kept eigenvalues.
int isometry(Ctx& ctx, const double* M, int64_t n, int dcut, double* U, std::vector<double>& lam,
             int step, int precision);

// Small kernels (small_kernels.cu)
// impure = 1: the observable inserted (Ising s, XY cos(theta), Potts [s = 0])
void launch_init_ising(Ctx& ctx, double* T, double beta, double h, int impure = 0);
void launch_init_xy(Ctx& ctx, double* T, int d0, double beta, double h, int impure = 0);
void launch_init_potts(Ctx& ctx, double* T, int q, double beta, double h, int impure = 0);
// x *= exp(-scal[slot]) (the impure tensor takes the pure tensor's ln n0)
void launch_scale_by_exp_neg(Ctx& ctx, double* x, int64_t n, const double* slot);
// x *= 1 / (the norm in scal[SC_NORM]), the pure tensor's last n_k
void launch_scale_by_last_norm(Ctx& ctx, double* x, int64_t n);
// y = (y + z) / 2
void launch_mean2(Ctx& ctx, double* y, const double* z, int64_t n);
// Tr T into a slot without the positivity check (an observable's trace may be <= 0)
void launch_trace_signed(Ctx& ctx, const double* T, int64_t Dx, int64_t Dy, double* slot);
void launch_maxabs(Ctx& ctx, const double* x, int64_t n, double* slot_bits);
void launch_normalise(Ctx& ctx, double* x, int64_t n, int step_weight_exp, bool initial);
void launch_trace(Ctx& ctx, const double* T, int64_t Dx, int64_t Dy, double* slot);
void launch_identity(Ctx& ctx, double* U, int64_t n);
void launch_fill(Ctx& ctx, double* x, int64_t n, double v);
void launch_copy_strided(Ctx& ctx, const View4& src, const View4& dst);

// Cubic lattice (path3d.cu, small_kernels.cu)
void launch_init_ising3d(Ctx& ctx, double* T, double beta, double h);
void launch_trace3(Ctx& ctx, const View6& t, double* slot);
// One z step of the view t into out (contiguous [X][X'][Y][Y'][z][z']);
// returns (Nx, Ny) and appends the kept eigenvalues of both isometries.
std::pair<int64_t, int64_t> step3(Ctx& ctx, const View6& t, int dcut, int step, double* out, int precision,
                                  std::vector<double>& lam_x, std::vector<double>& lam_y);

int read_status(Ctx& ctx);  // synchronises the stream
// Throws TRG_ETIMEOUT, with the word cleared for the next call, if a bounded
// device wait ran out (the stream has been synchronised).
void check_timeout(Ctx& ctx);
void trim_buffers(Ctx& ctx);  // free every solve buffer (engine.cu)

}  // namespace trg

struct trg_ctx : public trg::Ctx {};
