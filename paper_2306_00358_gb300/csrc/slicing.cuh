// Cutting FP64 operands into BF16 digits for the tensor-core products
// (split_gemm.cu: S = 2..5 slices, exact_gemm.cu: 15 digits).
//
// An operand is rows r < R of length K, element (r, k) at src[off_r[r] +
// off_c[k]]; its digits go to out[p][r][k] (r < Rp, k < Kp, zero in the
// padding; digit_at for the order of 15 digits, whose rows may be a part of a
// larger array of Rs).  With f the largest exponent field of a row and e = f - 1022
// (|x| < 2^e), X = rint(x 2^(F - e)), F = 7 + 8 (S - 1), halves away from
// zero, is the sum of d_p 2^(8 (S - 1 - p)), d_0 in [-128, 128], d_p in
// [-128, 127]; slices are stored as d_p 2^(-8p) (S <= 5) or as d_p (S = 15).
//
// All of it is bound by HBM: 8 B read (twice where the exponents take a pass
// of their own) and 2 S B written per element.
//  - Rows that are contiguous runs of at most 8192 are read once: a warp or a
//    block holds a row in registers, finds its exponent and cuts it
//    (k_cut_rows; k_cut_rows4 for 15 digits, up to 4096).  16384 x 4096, S = 4: 153 us (1.07 GB, 7.0 TB/s).
//  - Rows whose exponents the producing product recorded: a warp per row
//    (k_slice_contig).
//  - Gathered operands: k_row_field, then k_cut, both reading along the index
//    that is adjacent in memory.  4096 x 4096 read across, S = 4: 32 + 77 us.
//    (With a shared-memory atomic per element for the exponents and 2-byte
//    stores, two passes for every operand, the two above took 757 us.)
//  - A few gathered rows: one block per row reads it twice (k_slice_rows, in
//    split_gemm.cu).
#pragma once

#include <cstdint>

#include "internal.h"

namespace trg {

namespace {

// Biased exponent field; a subnormal counts as field 1 (SUB) or as zero.
template <bool SUB>
__device__ __forceinline__ unsigned exponent_field(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hi = (unsigned)(b >> 32) & 0x7fffffffu;
    if (!SUB) return hi >> 20;
    return hi >= 0x100000u ? hi >> 20 : ((hi | (unsigned)b) ? 1u : 0u);
}

// Scale exponent of a row from its largest field (-1022 for a zero row).
__device__ __forceinline__ int row_exponent(int f) { return f ? f - 1022 : -1022; }

// Planes stored for S digits: 15 digits are followed by |x| 2^(SIZE_SHIFT - e),
// cut off to BF16 (the operands of the product's |A||B|, see exact_gemm.cu).
// The shift keeps sums of up to 2^17 products of two of them below 2^127, and
// the floor, 2^-63 for any x that is not zero, keeps every product normal in
// FP32: such a sum is zero only if every |a||b| of it is.
__host__ __device__ constexpr int planes(int S) { return S == 15 ? 16 : S; }
constexpr int SIZE_SHIFT = 54, SIZE_FLOOR = -63;

// The digits of x in a row of largest field f, as the FP32 values to store
// (exact in BF16: their upper halves).
template <int S>
__device__ __forceinline__ void cut(double x, int f, float (&d)[planes(S)]) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7FF);
    const unsigned long long m53 = ex ? ((b & ((1ull << 52) - 1)) | (1ull << 52)) : 0ull;
    const bool neg = (long long)b < 0;
    // adding 128 to every digit but the first turns the signed digits into
    // bytes; a byte under the exponent of 2^23 is the FP32 number 2^23 + byte
    if constexpr (S == 15) {
        // X = mantissa 2^(66 - (f - ex)), 120 bits
        const int sh = f - ex - 66;
        typedef unsigned __int128 u128;
        const u128 m = sh <= 0 ? (u128)m53 << (-sh & 127) : sh < 60 ? (u128)((m53 + (1ull << (sh - 1))) >> sh) : (u128)0;
        const u128 y = (neg ? (u128)0 - m : m) + (((u128)0x0000808080808080ull << 64) | 0x8080808080808080ull);
        const unsigned long long ylo = (unsigned long long)y, yhi = (unsigned long long)(y >> 64);
        d[0] = (float)(int)((long long)yhi >> 48);
        const unsigned q[4] = {(unsigned)ylo, (unsigned)(ylo >> 32), (unsigned)yhi, (unsigned)(yhi >> 32)};
#pragma unroll
        for (int p = 1; p < 15; ++p) {
            const int byte = 14 - p;
            d[p] = __uint_as_float(__byte_perm(q[byte >> 2], 0x4B000000u, 0x7440u | (unsigned)(byte & 3))) - 8388736.0f;   // 2^23 + 128
        }
        // its FP32 exponent field: that of 1 is 127, |x| 2^-e = 1.mmm 2^(ex - f - 1)
        const int ea = max(ex - f + 126 + SIZE_SHIFT, 127 + SIZE_FLOOR);
        d[15] = (b << 1) ? __uint_as_float(((unsigned)ea << 23) | (((unsigned)(m53 >> 45) & 0x7Fu) << 16)) : 0.0f;
    } else {
        constexpr int F = 7 + 8 * (S - 1);
        constexpr unsigned BIAS = S == 2 ? 0x80u : S == 3 ? 0x8080u : S == 4 ? 0x808080u : 0x80808080u;
        const int sh = 53 - F + f - ex;          // > 0
        const long long m = sh < 63 ? (long long)((m53 + (1ull << (sh - 1))) >> sh) : 0ll;
        const long long y = (neg ? -m : m) + (long long)BIAS;
        d[0] = (float)(int)(y >> (8 * (S - 1)));
#pragma unroll
        for (int p = 1; p < S; ++p) {
            const unsigned v = __byte_perm((unsigned)y, 0x4B000000u, 0x7440u | (unsigned)(S - 1 - p));
            const float w = __int_as_float((127 - 8 * p) << 23);
            d[p] = fmaf(__uint_as_float(v), w, -8388736.0f * w);   // exact
        }
    }
}
// Where digit 0 of element (r, k) goes, and how far apart the digits of an
// element are: [p][r][k], but for 15 digits (and |x| 2^-e) the order in which
// their product's stages hold them in shared memory, [k / 16][p][r][k % 16] with
// the two 16-byte halves of a row's 16 k swapped in every other four rows (the
// 32-byte swizzle): a stage is a few long pieces of memory then.
template <int S>
__device__ __forceinline__ size_t digit_at(int r, int k, int Rp, int Kp) {
    if (S == 15) return ((size_t)(k >> 4) * planes(S) * Rp + r) * 16 + ((((k >> 3) ^ (r >> 2)) & 1) << 3) + (k & 7);
    return (size_t)r * Kp + k;
}
template <int S>
__device__ __forceinline__ size_t digit_stride(int Rp, int Kp) { return (size_t)Rp * (S == 15 ? 16 : Kp); }

// Two neighbours' digits as packed BF16.
template <int S>
__device__ __forceinline__ void cut2(double x0, double x1, int f, uint32_t (&w)[planes(S)]) {
    float a[planes(S)], b[planes(S)];
    cut<S>(x0, f, a);
    cut<S>(x1, f, b);
#pragma unroll
    for (int p = 0; p < planes(S); ++p) w[p] = __byte_perm(__float_as_uint(a[p]), __float_as_uint(b[p]), 0x7632);
}

// Largest exponent field of each row, maxima into ef (zeroed); a block takes 32
// rows and xf_k of their entries.  It is bound by latency where the operand is
// small: 256 entries (eight loads in flight per thread, fewest atomics) leave
// most of the chip idle there, so 64 are taken below four blocks per SM (576
// rows of 576: 11.4 -> 4.2 us).
constexpr int XF_BLOCKS = 600;
template <bool SUB>
__global__ void __launch_bounds__(256) k_row_field(const double* __restrict__ src, const int64_t* __restrict__ off_r,
                                                   const int64_t* __restrict__ off_c, int R, int K, int k_fast,
                                                   int xf_k, int* __restrict__ ef) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k0 = blockIdx.x * xf_k, k1 = min(K, k0 + xf_k);
    const int nby = (R + 31) / 32;      // row blocks, strided over grid.y (at most 65535)
    for (int by = blockIdx.y; by < nby; by += gridDim.y) {
        const int r0 = by * 32;
        if (k_fast) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r0 + warp * 4 + i;
                if (r >= R) break;
                const double* row = src + off_r[r];
                unsigned f = 0;
#pragma unroll 8
                for (int k = k0 + lane; k < k1; k += 32) f = max(f, exponent_field<SUB>(row[off_c[k]]));
                f = __reduce_max_sync(0xffffffffu, f);
                if (lane == 0 && f) atomicMax(&ef[r], (int)f);
            }
        } else {
            __shared__ unsigned red[8][32];
            const int r = r0 + lane;
            unsigned f = 0;
            if (r < R) {
                const double* row = src + off_r[r];
#pragma unroll 8
                for (int k = k0 + warp; k < k1; k += 8) f = max(f, exponent_field<SUB>(row[off_c[k]]));
            }
            red[warp][lane] = f;
            __syncthreads();
            if (warp == 0) {
#pragma unroll
                for (int w = 1; w < 8; ++w) f = max(f, red[w][lane]);
                if (r < R && f) atomicMax(&ef[r], (int)f);
            }
            __syncthreads();
        }
    }
}

// Digits of a gathered operand with known fields ef.  Elements pass through a
// 32 x 64 shared tile so that both sides are coalesced; a thread cuts eight
// adjacent k and writes 16 bytes per digit.
constexpr int XD_R = 32, XD_K = 64, XD_LD = XD_K + XD_K / 8 + 1;
template <int S>
__global__ void __launch_bounds__(256) k_cut(const double* __restrict__ src, const int64_t* __restrict__ off_r,
                                             const int64_t* __restrict__ off_c, int R, int K, int Rp, int Kp,
                                             int k_fast, const int* __restrict__ ef, int* __restrict__ e_out,
                                             uint16_t* __restrict__ out, int Rs) {
    __shared__ double tile[XD_R * XD_LD];
    const int k0 = blockIdx.x * XD_K;
    const size_t plane = digit_stride<S>(Rs, Kp);
    const int nby = (Rp + XD_R - 1) / XD_R;
    for (int by = blockIdx.y; by < nby; by += gridDim.y) {
        const int r0 = by * XD_R;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < XD_R * XD_K / 256; ++q) {
            const int e = threadIdx.x + q * 256;
            int rr, kk;
            if (k_fast) { kk = e % XD_K; rr = e / XD_K; } else { rr = e % XD_R; kk = e / XD_R; }
            const int r = r0 + rr, k = k0 + kk;
            tile[rr * XD_LD + kk + (kk >> 3)] = (r < R && k < K) ? src[off_r[r] + off_c[k]] : 0.0;
        }
        __syncthreads();
        const int rr = threadIdx.x >> 3, kg = threadIdx.x & 7;
        const int r = r0 + rr, k = k0 + kg * 8;
        if (r >= Rp || k >= Kp) continue;
        const int f = r < R ? ef[r] : 0;
        if (e_out && blockIdx.x == 0 && kg == 0 && r < R) e_out[r] = row_exponent(f);
        const double* x = tile + rr * XD_LD + kg * 9;
        uint32_t w[4][planes(S)];
#pragma unroll
        for (int h = 0; h < 4; ++h) cut2<S>(x[2 * h], x[2 * h + 1], f, w[h]);
        uint16_t* o = out + digit_at<S>(r, k, Rs, Kp);
#pragma unroll
        for (int p = 0; p < planes(S); ++p) *reinterpret_cast<uint4*>(o + p * plane) = make_uint4(w[0][p], w[1][p], w[2][p], w[3][p]);
    }
}

// Four adjacent elements of a contiguous row (zero past K).
__device__ __forceinline__ void load4(const double* row, int k, int K, bool vec, double (&v)[4]) {
    v[0] = v[1] = v[2] = v[3] = 0.0;
    if (vec && k + 3 < K) {
        const double2 a = *reinterpret_cast<const double2*>(row + k);
        const double2 b = *reinterpret_cast<const double2*>(row + k + 2);
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (k + j < K) v[j] = row[k + j];
    }
}
template <int S>
__device__ __forceinline__ void store4(const double (&v)[4], int f, uint16_t* o, size_t plane) {
    uint32_t a[planes(S)], b[planes(S)];
    cut2<S>(v[0], v[1], f, a);
    cut2<S>(v[2], v[3], f, b);
#pragma unroll
    for (int p = 0; p < planes(S); ++p) *reinterpret_cast<uint2*>(o + p * plane) = make_uint2(a[p], b[p]);
}

// Contiguous rows with known fields: a warp per row, four columns per lane.
template <int S>
__global__ void __launch_bounds__(256) k_slice_contig(const double* __restrict__ src, const int64_t* __restrict__ off_r,
                                                      int R, int K, int Rp, int Kp, const int* __restrict__ ef,
                                                      int* __restrict__ e_out, uint16_t* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (r >= Rp) return;
    const size_t plane = digit_stride<S>(Rp, Kp);
    const bool real = r < R;
    const double* row = real ? src + off_r[r] : nullptr;
    const bool vec = real && ((reinterpret_cast<uintptr_t>(row) & 15) == 0);
    const int f = real ? ef[r] : 0;
    if (e_out && lane == 0 && real) e_out[r] = row_exponent(f);
    for (int k = lane * 4; k < Kp; k += 128) {
        double v[4];
        load4(row, k, real ? K : 0, vec, v);
        store4<S>(v, f, out + digit_at<S>(r, k, Rp, Kp), plane);
    }
}

// Contiguous rows with unknown fields, K <= 4 TPR NCH: TPR threads (a warp or
// the block) hold a row in registers, so it is read once.
template <int S, int TPR, int NCH, bool SUB>
__global__ void __launch_bounds__(256) k_cut_rows(const double* __restrict__ src, const int64_t* __restrict__ off_r,
                                                  int R, int K, int Rp, int Kp, int* __restrict__ ef_out,
                                                  int* __restrict__ e_out, uint16_t* __restrict__ out) {
    __shared__ unsigned wmax[8];
    const int t = threadIdx.x % TPR;
    const int r = blockIdx.x * (256 / TPR) + threadIdx.x / TPR;
    if (TPR == 32 && r >= Rp) return;
    const size_t plane = digit_stride<S>(Rp, Kp);
    const bool real = r < R;
    const double* row = real ? src + off_r[r] : nullptr;
    const bool vec = real && ((reinterpret_cast<uintptr_t>(row) & 15) == 0);
    double v[NCH][4];
    unsigned fm = 0;
#pragma unroll
    for (int c = 0; c < NCH; ++c) load4(row, (c * TPR + t) * 4, real ? K : 0, vec, v[c]);
#pragma unroll
    for (int c = 0; c < NCH; ++c)
#pragma unroll
        for (int j = 0; j < 4; ++j) fm = max(fm, exponent_field<SUB>(v[c][j]));
    fm = __reduce_max_sync(0xffffffffu, fm);
    if (TPR == 256) {
        if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = fm;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 8; ++w) fm = max(fm, wmax[w]);
    }
    const int f = (int)fm;
    if (t == 0 && real) {
        if (ef_out) ef_out[r] = f;
        if (e_out) e_out[r] = row_exponent(f);
    }
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        const int k = (c * TPR + t) * 4;
        if (k < Kp) store4<S>(v[c], f, out + digit_at<S>(r, k, Rp, Kp), plane);
    }
}

constexpr int CUT_ROWS_MAX_K = 8192;
template <int S, bool SUB>
void launch_cut_rows(cudaStream_t stream, const double* src, const int64_t* off_r, int R, int K, int Rp, int Kp,
                     int* ef_out, int* e_out, uint16_t* out) {
    const unsigned gw = (unsigned)((Rp + 7) / 8), gb = (unsigned)Rp;
    if (Kp <= 128) k_cut_rows<S, 32, 1, SUB><<<gw, 256, 0, stream>>>(src, off_r, R, K, Rp, Kp, ef_out, e_out, out);
    else if (Kp <= 512) k_cut_rows<S, 32, 4, SUB><<<gw, 256, 0, stream>>>(src, off_r, R, K, Rp, Kp, ef_out, e_out, out);
    else if (Kp <= 2048) k_cut_rows<S, 256, 2, SUB><<<gb, 256, 0, stream>>>(src, off_r, R, K, Rp, Kp, ef_out, e_out, out);
    else if (Kp <= 4096) k_cut_rows<S, 256, 4, SUB><<<gb, 256, 0, stream>>>(src, off_r, R, K, Rp, Kp, ef_out, e_out, out);
    else k_cut_rows<S, 256, 8, SUB><<<gb, 256, 0, stream>>>(src, off_r, R, K, Rp, Kp, ef_out, e_out, out);
}

// The same for 15 digits, K <= 256 NCH: a block holds four rows, and a warp
// stores 32 k of all four at a time, so that each digit's 2 x 128 bytes are
// contiguous (digit_at; a warp per row writes eight pieces of 32 bytes, which
// takes 564 us where this takes 236: 6912 rows of 2304).
template <int NCH>
__global__ void __launch_bounds__(256) k_cut_rows4(const double* __restrict__ src, const int64_t* __restrict__ off_r,
                                                   int R, int K, int Rp, int Kp, int* __restrict__ ef_out,
                                                   uint16_t* __restrict__ out, int Rs) {
    __shared__ unsigned wmax[8][4];
    const int warp = threadIdx.x >> 5, rr = (threadIdx.x >> 3) & 3, kc = threadIdx.x & 7;
    const int r = blockIdx.x * 4 + rr;                   // Rp is a multiple of four
    const size_t plane = digit_stride<15>(Rs, Kp);
    const bool real = r < R;
    const double* row = real ? src + off_r[r] : nullptr;
    const bool vec = real && ((reinterpret_cast<uintptr_t>(row) & 15) == 0);
    double v[NCH][4];
    unsigned fm = 0;
#pragma unroll
    for (int c = 0; c < NCH; ++c) load4(row, ((c * 8 + warp) * 8 + kc) * 4, real ? K : 0, vec, v[c]);
#pragma unroll
    for (int c = 0; c < NCH; ++c)
#pragma unroll
        for (int j = 0; j < 4; ++j) fm = max(fm, exponent_field<true>(v[c][j]));
#pragma unroll
    for (int m = 1; m < 8; m *= 2) fm = max(fm, __shfl_xor_sync(0xffffffffu, fm, m));
    if (kc == 0) wmax[warp][rr] = fm;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) fm = max(fm, wmax[w][rr]);
    const int f = (int)fm;
    if (warp == 0 && kc == 0 && real) ef_out[r] = f;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        const int k = ((c * 8 + warp) * 8 + kc) * 4;
        if (k < Kp) store4<15>(v[c], f, out + digit_at<15>(r, k, Rs, Kp), plane);
    }
}

constexpr int CUT_ROWS4_MAX_K = 4096;
inline void launch_cut_rows4(cudaStream_t stream, const double* src, const int64_t* off_r, int R, int K, int Rp, int Kp,
                             int* ef_out, uint16_t* out, int Rs) {
    const unsigned grid = (unsigned)(Rp / 4);
    if (Kp <= 256) k_cut_rows4<1><<<grid, 256, 0, stream>>>(src, off_r, R, K, Rp, Kp, ef_out, out, Rs);
    else if (Kp <= 512) k_cut_rows4<2><<<grid, 256, 0, stream>>>(src, off_r, R, K, Rp, Kp, ef_out, out, Rs);
    else if (Kp <= 1024) k_cut_rows4<4><<<grid, 256, 0, stream>>>(src, off_r, R, K, Rp, Kp, ef_out, out, Rs);
    else if (Kp <= 2048) k_cut_rows4<8><<<grid, 256, 0, stream>>>(src, off_r, R, K, Rp, Kp, ef_out, out, Rs);
    else if (Kp <= 3072) k_cut_rows4<12><<<grid, 256, 0, stream>>>(src, off_r, R, K, Rp, Kp, ef_out, out, Rs);
    else k_cut_rows4<16><<<grid, 256, 0, stream>>>(src, off_r, R, K, Rp, Kp, ef_out, out, Rs);
}

template <bool SUB>
void launch_row_field(cudaStream_t stream, const Gather& g, int R, int K, int* ef) {
    const int64_t by = (R + 31) / 32;
    const int xf_k = by * ((K + 255) / 256) < XF_BLOCKS ? 64 : 256;
    dim3 grid((unsigned)((K + xf_k - 1) / xf_k), (unsigned)std::min<int64_t>(by, 65535));
    k_row_field<SUB><<<grid, 256, 0, stream>>>(g.base, g.off_r, g.off_c, R, K, g.c_fast ? 1 : 0, xf_k, ef);
}

template <int S>
void launch_cut(cudaStream_t stream, const Gather& g, int R, int K, int Rp, int Kp, const int* ef, int* e_out,
                uint16_t* out, int Rs = 0) {
    dim3 grid((unsigned)((Kp + XD_K - 1) / XD_K), (unsigned)std::min((Rp + XD_R - 1) / XD_R, 65535));
    k_cut<S><<<grid, 256, 0, stream>>>(g.base, g.off_r, g.off_c, R, K, Rp, Kp, g.c_fast ? 1 : 0, ef, e_out, out,
                                         Rs ? Rs : Rp);
}

// B operand as rows n, columns k: the roles of its two tables swapped.
inline Gather transposed(const Gather& b) {
    Gather t = b;
    t.off_r = b.off_c;
    t.off_c = b.off_r;
    t.c_fast = b.r_fast && !b.c_fast;
    t.r_fast = b.c_fast;
    t.c_identity = b.r_identity;
    t.r_identity = b.c_identity;
    return t;
}

}  // namespace

}  // namespace trg
