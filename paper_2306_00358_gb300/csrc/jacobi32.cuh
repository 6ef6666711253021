// FP32 cyclic Jacobi on a symmetric m x m matrix in one CTA's shared memory
// (the first stage of the Rayleigh-Ritz eigensolve, eig.cu).
//
// Round-robin ordering, rotation (p, q): tau = (h_qq - h_pp) / (2 h_pq),
// t = sign(tau) / (|tau| + sqrt(1 + tau^2)), c = 1 / sqrt(1 + t^2), s = t c,
// H <- J^T H J, W <- W J.
//
// What bounds it: the chain of rounds.  A round's rotations are a serial
// chain of three divisions and two square roots, its update touches all of H
// and W.  The two run side by side here: H is held twice, the update warps
// take round r from one copy to the other (column and row pass of a 2 x 2
// block in registers, a lane per block), and two warps work out the rotations
// of round r + 1 from the old copy and the rotations of round r by updating
// just the three elements that each needs.  One barrier a round instead of
// three.  The loops stay short: unrolled bodies were slower, since one CTA
// runs through them once a round.  All elements go through the operations of
// the plain form (columns first, then rows) in its order, so the bits are the
// plain form's.  Measured, a pair of calls in a solve (Q^T M Q of the last
// power steps) at m = 40 / 56: 132 / 207 us a call, the plain form 195 / 301; with every pair rotating at
// m = 33 / 40 / 56 / 64: 207 / 248 / 473 / 603 us, the plain form 264 / 384 /
// 700 / 678.  Above m = 72 (JAC_PIPE_M) the plain form is used: it skips the
// pairs below the threshold, which are most in late sweeps, where this one
// copies them (m = 88 in a solve: 487 us plain, 571 here).
#pragma once

#include <cstdint>

namespace trg {

namespace {

constexpr int JAC_PIPE_M = 72;
constexpr int JAC_MAX_PAIRS = JAC_PIPE_M / 2;

__device__ __forceinline__ void rr_pair(int r, int i, int mp, int& p, int& q) {
    if (i == 0) { p = mp - 1; q = r; }
    else {
        p = r + i; if (p >= mp - 1) p -= mp - 1;
        q = r - i; if (q < 0) q += mp - 1;
    }
    if (p > q) { const int x = p; p = q; q = x; }
}

template <typename T>
__device__ __forceinline__ bool jacobi_rotates(T hpq, T hpp, T hqq, T tol) {
    return fabs(hpq) > tol * sqrt(fabs(hpp * hqq)) && fabs(hpq) > (T)(sizeof(T) == 4 ? 0.0 : 1e-300);
}

// the two outputs of a rotation, rounded as the plain expressions c a - s b and s a + c b are
__device__ __forceinline__ float rot_p(float c, float s, float a, float b) { return fmaf(c, a, -(s * b)); }
__device__ __forceinline__ float rot_q(float c, float s, float a, float b) { return fmaf(s, a, c * b); }

struct JacShared {
    float2 cs[2][JAC_MAX_PAIRS];     // c, s of the rounds' pairs (round parity)
    short2 pq[2][JAC_MAX_PAIRS];
    int rot;
};

// Without branches (the lanes of a warp would take both sides).  A pair below
// the threshold goes through with harmless numbers: zeros and infinities would
// take the slow paths of the divisions and square roots.
__device__ __forceinline__ float2 jac_rotation(float hpq, float hpp, float hqq, float tol) {
    const bool rot = jacobi_rotates<float>(hpq, hpp, hqq, tol);
    const float tau = (rot ? hqq - hpp : 1.0f) / (rot ? 2 * hpq : 1.0f);
    const float ta = 1 / (fabsf(tau) + sqrtf(1 + tau * tau));
    const float t = (tau >= 0) ? ta : -ta;
    const float c = 1 / sqrtf(1 + t * t);
    return rot ? make_float2(c, t * c) : make_float2(1.0f, 0.0f);
}

// Pair that player x belongs to in round r.
__device__ __forceinline__ int jac_pair_of(int r, int x, int mp) {
    if (x == mp - 1 || x == r) return 0;
    int d = x - r;
    if (d < 0) d += mp - 1;
    return min(d, mp - 1 - d);
}

// H is m rows of ld floats in Ha (Hb: scratch of the same size), W column-major
// m x m.  Rotations with |h_pq| <= tol sqrt(|h_pp h_qq|) are skipped; the loop
// ends when a scan finds no pair above the threshold.  Returns the sweeps that
// rotated (max_sweeps + 1 at the limit).  All NT threads of the block call it.
template <int NT>
__device__ int jacobi_sweeps_f32(float* Ha, float* Hb, int ld, float* W, int m, float tol, int max_sweeps,
                                 JacShared& sh) {
    const int mp = m + (m & 1), npair = mp / 2;
    const int warp = threadIdx.x >> 5;
    float* H = Ha;
    float* Hn = Hb;
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        if (threadIdx.x == 0) sh.rot = 0;
        __syncthreads();
        for (int e = threadIdx.x; e < m * m; e += NT) {
            const int p = e / m, q = e % m;
            if (p < q && jacobi_rotates<float>(H[p * ld + q], H[p * ld + p], H[q * ld + q], tol)) *(volatile int*)&sh.rot = 1;
        }
        if (threadIdx.x < npair) {      // the first round's rotations
            int p, q;
            rr_pair(0, threadIdx.x, mp, p, q);
            sh.cs[0][threadIdx.x] = q < m ? jac_rotation(H[p * ld + q], H[p * ld + p], H[q * ld + q], tol) : make_float2(1.0f, 0.0f);
            sh.pq[0][threadIdx.x] = make_short2((short)p, (short)q);
        }
        __syncthreads();
        if (sh.rot == 0) return sweep;
        for (int r = 0; r < mp - 1; ++r) {
            const float2* cs = sh.cs[r & 1];
            const short2* pq = sh.pq[r & 1];
            if (warp < 2) {
                const int i = threadIdx.x;
                if (i < npair && r + 1 < mp - 1) {
                    int P, Q;
                    rr_pair(r + 1, i, mp, P, Q);
                    float2 o = make_float2(1.0f, 0.0f);
                    if (Q < m) {
                        // element (x, y) after this round, x and y in the pairs (a, ca) and
                        // (b, cb): both outputs of a rotation are alpha u + beta v
                        auto element = [&](int x, int y, short2 a, float2 ca, short2 b, float2 cb) {
                            const bool bp = y == b.x, ap = x == a.x;
                            const float ba = bp ? cb.x : cb.y, bb = bp ? -cb.y : cb.x;
                            const float aa = ap ? ca.x : ca.y, ab = ap ? -ca.y : ca.x;
                            const int ay = min((int)a.y, m - 1), by = min((int)b.y, m - 1);   // dummy: not used below
                            const float* h0 = H + a.x * ld;
                            const float* h1 = H + ay * ld;
                            const float u0 = h0[b.x], u1 = h0[by], w0 = h1[b.x], w1 = h1[by];
                            const float v0 = cb.y == 0.0f ? (bp ? u0 : u1) : fmaf(ba, u0, bb * u1);
                            const float v1 = cb.y == 0.0f ? (bp ? w0 : w1) : fmaf(ba, w0, bb * w1);
                            return ca.y == 0.0f ? (ap ? v0 : v1) : fmaf(aa, v0, ab * v1);
                        };
                        const int ip = jac_pair_of(r, P, mp), iq = jac_pair_of(r, Q, mp);
                        const short2 a = pq[ip], b = pq[iq];
                        const float2 ca = cs[ip], cb = cs[iq];
                        const float hpq = element(P, Q, a, ca, b, cb);
                        const float hpp = element(P, P, a, ca, a, ca);
                        const float hqq = element(Q, Q, b, cb, b, cb);
                        o = jac_rotation(hpq, hpp, hqq, tol);
                    }
                    sh.cs[(r + 1) & 1][i] = o;
                    sh.pq[(r + 1) & 1][i] = make_short2((short)P, (short)Q);
                }
            } else {
                constexpr int NW = NT / 32 - 2;
                const int lane = threadIdx.x & 31;
                // a warp per row pair, a lane per column pair (two of them for
                // npair > 32), whose places and rotation stay in registers
                short2 b[2];
                float2 cb[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int j = lane + 32 * u;
                    b[u] = j < npair ? pq[j] : make_short2(0, 0);
                    cb[u] = j < npair ? cs[j] : make_float2(1.0f, 0.0f);
                }
#pragma unroll 1
                for (int i = warp - 2; i < npair; i += NW) {
                    const short2 a = pq[i];
                    const float2 ca = cs[i];
                    const bool qa = a.y < m;
                    const float* h0 = H + a.x * ld;
                    const float* h1 = H + (qa ? a.y : a.x) * ld;
                    float* n0 = Hn + a.x * ld;
                    float* n1 = Hn + a.y * ld;
#pragma unroll 1
                    for (int u = 0; u < 2; ++u) {
                        const int j = lane + 32 * u;
                        if (j >= npair) break;
                        const short2 bu = u ? b[1] : b[0];
                        const float2 cu = u ? cb[1] : cb[0];
                        const bool qb = bu.y < m;
                        const int c0 = bu.x, c1 = qb ? bu.y : bu.x;
                        float x00 = h0[c0], x01 = h0[c1], x10 = h1[c0], x11 = h1[c1];
                        const float e = rot_p(cu.x, cu.y, x00, x01), f = rot_q(cu.x, cu.y, x00, x01);
                        const float g = rot_p(cu.x, cu.y, x10, x11), h = rot_q(cu.x, cu.y, x10, x11);
                        x00 = rot_p(ca.x, ca.y, e, g); x10 = rot_q(ca.x, ca.y, e, g);
                        x01 = rot_p(ca.x, ca.y, f, h); x11 = rot_q(ca.x, ca.y, f, h);
                        if (i == j && ca.y != 0.0f) x01 = x10 = 0.0f;
                        n0[c0] = x00;
                        if (qb) n0[c1] = x01;
                        if (qa) { n1[c0] = x10; if (qb) n1[c1] = x11; }
                    }
                    if (ca.y != 0.0f) {
                        float* wp = W + a.x * m;
                        float* wq = W + a.y * m;
#pragma unroll 1
                        for (int k = lane; k < m; k += 32) {
                            const float vp = wp[k], vq = wq[k];
                            wp[k] = rot_p(ca.x, ca.y, vp, vq);
                            wq[k] = rot_q(ca.x, ca.y, vp, vq);
                        }
                    }
                }
            }
            __syncthreads();
            float* x = H; H = Hn; Hn = x;
        }
    }
    return max_sweeps + 1;
}

}  // namespace

}  // namespace trg
