// jacobi_wv.cu -- one-sided Jacobi SVD of FP32 matrices with up to 64 columns and 64 or 128 rows, the
// matrix W and the accumulated rotations V held by different warps in different layouts (Algorithm 2,
// Section 2.2; the register tier of Section 4).
//
// The method, the pair ordering (odd-even transposition with exchange, 32 pair slots), the scaled
// rotations, the carried norms and the order of every sum are those of jacobi_reg.cu, so results are
// the same bit for bit.  What differs is who holds what:
//   W warps  lane (h, i), h = lane / 16, holds 32 rows (part h of the warp's 64) of four columns, the
//            ones at positions 4 i .. 4 i + 3, as pairs of consecutive rows (packed FP32 FMAs; each
//            half rounds as the scalar one).  Even steps and every other pair of the odd steps then
//            stay inside a lane; one column in four moves to the neighbouring lane each step (half a
//            shuffle per element and step of what one slot per lane would take).  Slot 2 i + h's scales,
//            norms and rotation parameters are lane (h, i)'s: the two halves exchange one partial sum
//            and two multipliers, and no parameter is computed twice.  A 64-row matrix has one W warp,
//            and its steps need no barrier.
//   V warp   lane t holds rows t and t + 32 of V, all 64 columns in registers by position, so that a
//            step is two FMAs per pair and row and no exchange: the swap of positions is a renaming of
//            registers.  The steps' multipliers arrive in a ring in shared memory, broadcast to all
//            lanes; the V warp runs up to kRing double steps behind the W warps.
// Why: with W and V in the same lanes (jacobi_reg.cu) a preconditioned 64 x 64 matrix takes 759 k warp
// instructions (1400 a step, of which 366 are FP32 FMAs); the rest is the exchange of W and V (a shuffle
// per element, two selects per element on odd steps, moves), parameters computed by both row parts, and
// spills.  Here it takes 357 k (660 a step), and the step's dependent chain of exchange, parameters and dot
// products bounds it: 1550 cycles a step for a matrix alone; with 12 warps in 168 registers each on an SM
// 41 % of the issue slots and 32 % of the FMA pipe are busy, and barrier waits (the V warps', for the
// ring) and fixed latencies lead the stalls.
// Measured (GB300, before -> after): 20 000 preconditioned 64 x 64 matrices 18.6 -> 13.8 ms; 500 of
// 512 x 512 by the block tier, whose inner SVDs these are, 230 -> 212 ms; a depth-12 basis tree (128-row
// form) 16.0 -> 12.4 ms.
#include <cuda_runtime.h>

#include <type_traits>

#include "common.cuh"
#include "launch.cuh"
#include "rnmath.cuh"

namespace bsvd {

namespace {

constexpr int kRing = 2;      // double steps (even, odd) in flight between the W and the V warps
constexpr int kCols = 64;     // column capacity (32 slots of two)
constexpr int kLdV = 65;      // leading dimension of the V exchange area (QR-preconditioned form)
constexpr unsigned kFullWarp = 0xffffffffu;

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 shfl2(float2 v, int src)
{
    return make_float2(__shfl_sync(kFullWarp, v.x, src), __shfl_sync(kFullWarp, v.y, src));
}
__device__ __forceinline__ float2 sel2(bool w, float2 a, float2 b) { return make_float2(w ? a.x : b.x, w ? a.y : b.y); }

// the three Gram entries of a pair over 32 rows, two chains (even, odd rows) each
__device__ __forceinline__ void dot3(const float2 (&x)[16], const float2 (&y)[16], float& a, float& b, float& c)
{
    float2 ca = both(0.f), cb = both(0.f), cc = both(0.f);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        ca = fma2(x[j], x[j], ca);
        cb = fma2(y[j], y[j], cb);
        cc = fma2(x[j], y[j], cc);
    }
    a = ca.x + ca.y;
    b = cb.x + cb.y;
    c = cc.x + cc.y;
}

// gamma alone, four chains (rows mod 4)
__device__ __forceinline__ float dot1(const float2 (&x)[16], const float2 (&y)[16])
{
    float2 c0 = both(0.f), c1 = both(0.f);
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
        c0 = fma2(x[j], y[j], c0);
        c1 = fma2(x[j + 1], y[j + 1], c1);
    }
    return (c0.x + c1.x) + (c0.y + c1.y);
}

// rows r .. r + 3 of a column: 16 bytes where aligned
__device__ __forceinline__ void store4(float* p, bool vec, int left, float a, float b, float c, float d)
{
    if (vec && left >= 4) {
        *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
    } else {
        if (left > 0) p[0] = a;
        if (left > 1) p[1] = b;
        if (left > 2) p[2] = c;
        if (left > 3) p[3] = d;
    }
}
__device__ __forceinline__ float4 load4(const float* p, bool vec, int left)
{
    if (vec && left >= 4) return *reinterpret_cast<const float4*>(p);
    return make_float4(left > 0 ? p[0] : 0.f, left > 1 ? p[1] : 0.f, left > 2 ? p[2] : 0.f, left > 3 ? p[3] : 0.f);
}
__device__ __forceinline__ int again(const int* p) { return *reinterpret_cast<const volatile int*>(p); }
__device__ __forceinline__ bool vec16(const void* p, int ld)
{
    return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld & 3) == 0;
}

// named barriers of `threads` threads: producers arrive, consumers wait.  The ids are literals: a kernel
// with a computed id is charged all 16 barriers, and an SM has 64.
template <int ID>
__device__ __forceinline__ void bar_wait(int threads)
{
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "r"(threads) : "memory");
}
template <int ID>
__device__ __forceinline__ void bar_arrive(int threads)
{
    asm volatile("bar.arrive %0, %1;" ::"n"(ID), "r"(threads) : "memory");
}
constexpr int kBarFull = 1, kBarEmpty = 3, kBarSweep = 5, kBarRed = 6, kBarRanks = 7;   // + ring slot for the first two
static_assert(kRing == 2, "two literal ids each");
__device__ __forceinline__ void wait_full(int slot) { slot ? bar_wait<kBarFull + 1>(64) : bar_wait<kBarFull>(64); }
__device__ __forceinline__ void wait_empty(int slot) { slot ? bar_wait<kBarEmpty + 1>(64) : bar_wait<kBarEmpty>(64); }
__device__ __forceinline__ void arrive_full(int slot) { slot ? bar_arrive<kBarFull + 1>(64) : bar_arrive<kBarFull>(64); }
__device__ __forceinline__ void arrive_empty(int slot) { slot ? bar_arrive<kBarEmpty + 1>(64) : bar_arrive<kBarEmpty>(64); }

struct WvShared {
    float4 ring[kRing][2][32];  // per double step, parity and pair: mL, mL, mR, mR
};

// QR of the preconditioned form: the matrix (leading dimension 64; reflector i in rows >= i of column i,
// R above the diagonal), R's diagonal, the reflector being applied and the reduction slots.  The ring
// is idle while V passes through vs, so the two share their memory.
struct WvQr {
    float qs[kCols * kCols];
    float v[2][kCols];        // the reflector being applied
    float2 red[2][2][32];
    float qdiag[kCols];
    float qred[2];
};

template <int WW>
struct WvRed {
    float4 g[2][2 * WW][32];  // per parity, row part and slot: partial sums (alpha, beta, gamma)
};

// A W warp's step.  Even: pairs A = (c0, c1) and B = (c2, c3), positions (4 i, 4 i + 1) and (4 i + 2,
// 4 i + 3).  Odd: A = (c0, c3) and B = (c2, c1), positions (4 i + 1, 4 i + 2) and (4 i + 3, 4 i + 4).
struct WvState {
    float dL, dR;   // scales of slot 2 i + h's columns
    float nL, nR;   // carried norms: true squared norms (negative: stale)
};

template <int WW, bool ODD, bool P64, bool CARRY, typename P>
__device__ __forceinline__ unsigned wv_step(float2 (&c0)[16], float2 (&c1)[16], float2 (&c2)[16], float2 (&c3)[16],
                                            WvState& q, int lane, int warp, P tol, WvRed<WW>& red, int& par,
                                            float4* ring)
{
    const int h = lane >> 4, i = lane & 15;
    // partial Gram entries of both pairs over this lane's rows: the three products, or -- carried norms,
    // neither norm stale -- gamma alone
    bool mineA = true, mineB = true;
    const bool mine = !CARRY || q.nL < 0.f || q.nR < 0.f;
    if (CARRY) {
        const unsigned mb = __ballot_sync(kFullWarp, mine);
        mineA = (mb >> i) & 1u;
        mineB = (mb >> (16 + i)) & 1u;
    }
    float aA = 0.f, bA = 0.f, gA, aB = 0.f, bB = 0.f, gB;
    if (mineA)
        ODD ? dot3(c0, c3, aA, bA, gA) : dot3(c0, c1, aA, bA, gA);
    else
        gA = ODD ? dot1(c0, c3) : dot1(c0, c1);
    if (mineB)
        ODD ? dot3(c2, c1, aB, bB, gB) : dot3(c2, c3, aB, bB, gB);
    else
        gB = ODD ? dot1(c2, c1) : dot1(c2, c3);
    // this lane's pair: slot 2 i + h
    float sa = 0.f, sb = 0.f, sc;
    if constexpr (WW == 1) {
        if (!CARRY || __any_sync(kFullWarp, mine)) {
            sa = (h ? aB : aA) + __shfl_xor_sync(kFullWarp, h ? aA : aB, 16);
            sb = (h ? bB : bA) + __shfl_xor_sync(kFullWarp, h ? bA : bB, 16);
        }
        sc = (h ? gB : gA) + __shfl_xor_sync(kFullWarp, h ? gA : gB, 16);
    } else {
        red.g[par][2 * warp + h][2 * i] = make_float4(aA, bA, gA, 0.f);
        red.g[par][2 * warp + h][2 * i + 1] = make_float4(aB, bB, gB, 0.f);
        bar_wait<kBarRed>(32 * WW);
        sa = sb = sc = 0.f;
#pragma unroll
        for (int p = 0; p < 2 * WW; ++p) {
            const float4 x = red.g[par][p][2 * i + h];
            sa += x.x;
            sb += x.y;
            sc += x.z;
        }
        par ^= 1;
    }
    float tnL = q.nL, tnR = q.nR;
    if (CARRY && mine) {
        tnL = q.dL * q.dL * sa;
        tnR = q.dR * q.dR * sb;
    }
    // rotation of the pair, in the unscaled frame; the wrap slot idles on odd steps.  With carried norms or
    // two W warps the parameters are computed by every lane without branches (a lane that does not
    // rotate drops them), so that the reciprocals and the test run under the dot product and the cosine
    // under the exchange (128 rows: a depth-12 basis tree 12.9 -> 12.4 ms);
    // with one warp and three sums a step the built-in operations' fewer instructions are faster
    // (20 000 of 54 x 45: 23.4 against 22.6 ms).
    const P alpha = CARRY ? P(tnL) : P(q.dL) * P(q.dL) * P(sa);
    const P beta = CARRY ? P(tnR) : P(q.dR) * P(q.dR) * P(sb);
    const P gamma = P(q.dL) * P(q.dR) * P(sc);
    const bool rot = !(ODD && lane == 31) && alpha > P(0) && beta > P(0) && off_diagonal_large(alpha, beta, gamma, tol);
    const unsigned rots = __ballot_sync(kFullWarp, rot);
    float mL = 0.f, mR = 0.f, cth = 1.f, tth = 0.f;
    if constexpr (P64 || (!CARRY && WW == 1)) {
        if (rot) {
            const P t = jacobi_t(alpha, beta, gamma);
            tth = float(t);
            cth = float(drsqrt(P(1) + t * t));
            mL = -float(t) * (q.dR * rcp_rn(q.dL));
            mR = float(t) * (q.dL * rcp_rn(q.dR));
        }
    } else if (rots) {  // (most steps of the last sweeps rotate nothing)
        // scale ratios from the current scales (correctly rounded reciprocals; 2^-33 < d <= 1)
        const float kL = q.dR * rn_rcp(q.dL), kR = q.dL * rn_rcp(q.dR);
        // jacobi_t: the larger of |dn| and |gn| is in [1, 2), the divisor in [1, 5)
        const float d = beta - alpha, g2 = 2.f * gamma;
        const float ad = fabsf(d), ag = fabsf(g2);
        const float sl = pow2_scale(ad > ag ? ad : ag);
        const float dn = ad * sl, gn = g2 * sl;
        const float den = dn + rn_sqrt(fmaf(dn, dn, gn * gn));
        float t = rn_div(gn, den);
        if (__any_sync(kFullWarp, rot && !(fabsf(gn) >= 0x1p-100f && den < 8.f))) t = gn / den;
        t = rot ? (d >= 0.f ? t : -t) : 0.f;
        mL = -t * kL;  // -t d_j / d_i
        mR = t * kR;   //  t d_i / d_j
        cth = rn_rsqrt12(fmaf(t, t, 1.f));
        tth = t;
    }
    q.dL *= cth;
    q.dR *= cth;
    q.nL = tnL;
    q.nR = tnR;
    if (CARRY) {
        // alpha' = alpha - t gamma, beta' = beta + t gamma; a cancelling update is stale
        const float aN = fmaf(-tth, float(gamma), tnL), bN = fmaf(tth, float(gamma), tnR);
        q.nL = rot && aN < 0.25f * tnL ? -1.f : aN;
        q.nR = rot && bN < 0.25f * tnR ? -1.f : bN;
    }
    if (ring) ring[2 * i + h] = make_float4(mL, mL, mR, mR);
    const float oL = __shfl_xor_sync(kFullWarp, mL, 16), oR = __shfl_xor_sync(kFullWarp, mR, 16);
    const float2 mLA = both(h ? oL : mL), mRA = both(h ? oR : mR), mLB = both(h ? mL : oL), mRB = both(h ? mR : oR);
    // rotate and exchange.  A skipped pair has multipliers 0, which leaves its columns as they are.
    if (!ODD) {
        // the right column of pair A (position 4 i after the swap) moves one lane down
        const int src = (lane & 16) | ((i + 1) & 15);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float2 t = fma2(mRA, c0[j], c1[j]);
            c0[j] = fma2(mLA, c1[j], c0[j]);
            c1[j] = shfl2(t, src);
            const float2 l = fma2(mLB, c3[j], c2[j]);
            c3[j] = fma2(mRB, c2[j], c3[j]);
            c2[j] = l;
        }
        // slot p takes slot p + 1's right column
        const int ssrc = h ? (i + 1) & 15 : 16 + i;
        q.dR = __shfl_sync(kFullWarp, q.dR, ssrc);
        if (CARRY) q.nR = __shfl_sync(kFullWarp, q.nR, ssrc);
    } else {
        // the left column of pair B (position 4 i + 4) moves one lane up; the last lane, whose pair B
        // (positions 63 and 0) idled, hands position 0's column back and keeps position 63's
        const int src = (lane & 16) | ((i + 15) & 15);
        const bool last = i == 15;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float2 x = c1[j], y = c2[j], l = c0[j], r = c3[j];
            const float2 t = fma2(mLB, x, y), u = fma2(mRB, y, x);
            c3[j] = sel2(last, t, u);
            c0[j] = shfl2(sel2(last, u, t), src);
            c2[j] = fma2(mLA, r, l);
            c1[j] = fma2(mRA, l, r);
        }
        // slot p takes slot p - 1's left column; the wrap slot hands over its right one and keeps its
        // left one as the right
        const int ssrc = h ? i : 16 + ((i + 15) & 15);
        const bool wrap = lane == 31;
        const float d = __shfl_sync(kFullWarp, wrap ? q.dR : q.dL, ssrc);
        q.dR = wrap ? q.dL : q.dR;
        q.dL = d;
        if (CARRY) {
            const float n = __shfl_sync(kFullWarp, wrap ? q.nR : q.nL, ssrc);
            q.nR = wrap ? q.nL : q.nR;
            q.nL = n;
        }
    }
    return rots;
}

}  // namespace

// WW: W warps (64 rows each); MINB: CTAs per SM the register allocation is capped for.  One matrix per
// CTA of 32 (WW + 1) threads, the last warp the V warp.
template <int WW, int MINB, bool PRE, bool P64, bool CARRY>
__global__ void __launch_bounds__(32 * (WW + 1), MINB)
    jacobi_wv_kernel(int batch, float* const* A, const int* M, const int* N, const int* LDA, float* const* Sout,
                     float* const* U, const int* LDU, float* const* V, const int* LDV, double tol_in, int max_sweeps,
                     int* info, long long* rot_out, ItemList wl)
{
    static_assert(!PRE || WW == 1, "the preconditioned form is square: 64 rows");
    constexpr int PARTS = 2 * WW;      // parts of 32 rows
    typedef typename std::conditional<P64, double, float>::type P;

    constexpr size_t kRingBytes = sizeof(WvShared);
    constexpr size_t kVsBytes = PRE ? sizeof(float) * kCols * kLdV : 0;
    __shared__ __align__(16) unsigned char sh_raw[kRingBytes > kVsBytes ? kRingBytes : kVsBytes];
    WvShared& sh = *reinterpret_cast<WvShared*>(sh_raw);
    float* vs = reinterpret_cast<float*>(sh_raw);
    __shared__ __align__(16) unsigned char qr_raw[PRE ? sizeof(WvQr) : 16];
    WvQr& q = *reinterpret_cast<WvQr*>(qr_raw);
    __shared__ __align__(16) unsigned char red_raw[WW > 1 ? sizeof(WvRed<WW>) : 16];
    WvRed<WW>& red = *reinterpret_cast<WvRed<WW>*>(red_raw);
    __shared__ float sig_s[kCols];
    __shared__ int rank_s[kCols];      // by position
    __shared__ float2 fold_s[32];      // a sweep's scales of the slots' columns
    __shared__ int more_s;             // another sweep follows

    const int tid = threadIdx.x;
    const int s = tid & 31;            // lane: slot (W warps), row (V warp)
    int warp = tid >> 5;
    if constexpr (WW == 1) {
        // W and V warps on every scheduler of the SM: warps go to schedulers by their hardware slot, so
        // with W always first in its CTA, two schedulers would run all the W warps
        if (tid == 0) {
            unsigned hw;
            asm volatile("mov.u32 %0, %%warpid;" : "=r"(hw));
            more_s = (hw >> 2) & 1;
        }
        __syncthreads();
        warp ^= more_s;
        __syncthreads();
    }
    const bool is_v = warp == WW;

    for (int b = item_first(wl, batch); b >= 0; b = item_next(wl, batch, b)) {
        const int m = M[b], n = N[b], lda = LDA[b];
        const bool tr = m < n;
        const int mm = tr ? n : m;
        const int nn = tr ? m : n;
        const bool wantU = U != nullptr, wantV = V != nullptr;
        const int ldu = wantU ? LDU[b] : 1, ldvo = wantV ? LDV[b] : 1;
        const bool bad = m < 0 || n < 0 || mm > 32 * PARTS || nn > kCols || lda < (m > 1 ? m : 1) ||
                         (wantU && ldu < (m > 1 ? m : 1)) || (wantV && ldvo < (n > 1 ? n : 1));
        if (bad) {
            if (tid == 0) info[b] = BSVD_INFO_BAD_SHAPE;
            continue;
        }
        if (nn == 0) {
            if (tid == 0) {
                info[b] = 0;
                if (rot_out) rot_out[b] = 0;
            }
            continue;
        }
        // preconditioned: the sweeps run on R^T, whose rotations give U (through Q) and whose
        // normalised columns give V, so the roles of the two outputs swap as for A^T
        const bool pre = PRE && m == n && n > 1;
        const bool sw = tr || pre;
        const bool accV = sw ? wantU : wantV;
        const float* a = A[b];
        // the outputs' pointers and sizes are read where they are used: kept through the sweeps they would
        // spill the columns
        auto w_out = [&](int& ld) -> float* {   // receives W / sigma
            if (!(sw ? wantV : wantU)) return nullptr;
            ld = again((sw ? LDV : LDU) + b);
            return (sw ? V : U)[b];
        };
        auto v_out = [&](int& ld) -> float* {   // receives V (PRE: Q V_w)
            ld = again((sw ? LDU : LDV) + b);
            return (sw ? U : V)[b];
        };

        if constexpr (PRE) {
            if (pre) {
                // Householder QR, warp p holding rows 32 p .. of the columns 2 s and 2 s + 1 (Algorithm
                // 1): column i's owner lanes publish it with their share of its squared norm; lane t
                // of warp p forms element 32 p + t of the reflector v_i (normalised for I - 2 v v^T),
                // every lane reads it as a broadcast and applies it to its columns right of i.
                const int p = warp, cl = 2 * s, cr = 2 * s + 1;
                float aL[32], aR[32];
                const bool va = vec16(a, lda);
#pragma unroll
                for (int k = 0; k < 32; k += 4) {
                    const int r = p * 32 + k;
                    const float4 x = cl < n ? load4(a + (size_t)cl * lda + r, va, n - r) : make_float4(0.f, 0.f, 0.f, 0.f);
                    const float4 y = cr < n ? load4(a + (size_t)cr * lda + r, va, n - r) : make_float4(0.f, 0.f, 0.f, 0.f);
                    aL[k] = x.x;
                    aL[k + 1] = x.y;
                    aL[k + 2] = x.z;
                    aL[k + 3] = x.w;
                    aR[k] = y.x;
                    aR[k + 1] = y.y;
                    aR[k + 2] = y.z;
                    aR[k + 3] = y.w;
                }
                const int rt = p * 32 + s;
#pragma unroll 1
                for (int i = 0; i < n; ++i) {
                    if (s == (i >> 1)) {
                        // (rows past n hold zeros; entries above the diagonal are R's)
                        const bool odd_col = i & 1;
                        float ss = 0.f;
#pragma unroll
                        for (int k = 0; k < 32; k += 4) {
                            float x[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                x[e] = odd_col ? aR[k + e] : aL[k + e];
                                const float y = p * 32 + k + e >= i ? x[e] : 0.f;
                                ss = fmaf(y, y, ss);
                            }
                            *reinterpret_cast<float4*>(q.qs + i * kCols + p * 32 + k) = make_float4(x[0], x[1], x[2], x[3]);
                        }
                        q.qred[p] = ss;
                    }
                    __syncthreads();
                    const float ss = q.qred[0] + q.qred[1];
                    const float x0 = q.qs[i * kCols + i];
                    const float xt = q.qs[i * kCols + rt];
                    const float alpha = dsqrt(ss);
                    const float sg = x0 >= 0.f ? 1.f : -1.f;
                    const float inv = alpha > 0.f ? drsqrt(2.f * alpha * (alpha + dabs(x0))) : 0.f;
                    const float vt = rt < i ? 0.f : (rt == i ? x0 + sg * alpha : xt) * inv;
                    float* vb = q.v[i & 1] + p * 32;
                    vb[s] = vt;
                    __syncwarp();
                    float wl_ = 0.f, wr_ = 0.f;
#pragma unroll
                    for (int k = 0; k < 32; k += 4) {
                        const float4 x = *reinterpret_cast<const float4*>(vb + k);
                        wl_ = fmaf(x.x, aL[k], wl_);
                        wr_ = fmaf(x.x, aR[k], wr_);
                        wl_ = fmaf(x.y, aL[k + 1], wl_);
                        wr_ = fmaf(x.y, aR[k + 1], wr_);
                        wl_ = fmaf(x.z, aL[k + 2], wl_);
                        wr_ = fmaf(x.z, aR[k + 2], wr_);
                        wl_ = fmaf(x.w, aL[k + 3], wl_);
                        wr_ = fmaf(x.w, aR[k + 3], wr_);
                    }
                    q.red[i & 1][p][s] = make_float2(wl_, wr_);
                    __syncthreads();
                    const float2 w0 = q.red[i & 1][0][s], w1 = q.red[i & 1][1][s];
                    // columns right of i take the reflector (column i itself is final: R(i, i) to qdiag)
                    wl_ = cl > i ? -2.f * (w0.x + w1.x) : 0.f;
                    wr_ = cr > i ? -2.f * (w0.y + w1.y) : 0.f;
#pragma unroll
                    for (int k = 0; k < 32; k += 4) {
                        const float4 x = *reinterpret_cast<const float4*>(vb + k);
                        aL[k] = fmaf(wl_, x.x, aL[k]);
                        aR[k] = fmaf(wr_, x.x, aR[k]);
                        aL[k + 1] = fmaf(wl_, x.y, aL[k + 1]);
                        aR[k + 1] = fmaf(wr_, x.y, aR[k + 1]);
                        aL[k + 2] = fmaf(wl_, x.z, aL[k + 2]);
                        aR[k + 2] = fmaf(wr_, x.z, aR[k + 2]);
                        aL[k + 3] = fmaf(wl_, x.w, aL[k + 3]);
                        aR[k + 3] = fmaf(wr_, x.w, aR[k + 3]);
                    }
                    if (rt >= i) q.qs[i * kCols + rt] = vt;
                    if (rt == i) q.qdiag[i] = -sg * alpha;
                }
                __syncthreads();
            }
        }

        const int sweeps_cap = max_sweeps > 0 ? max_sweeps : 30;
        int sweep = 0;

        if (!is_v) {
            // ================================ W ================================
            const P tol = tol_in > 0.0 ? P(tol_in) : P(dsqrt(double(mm)) * Unit<float>::value);
            const int h = s >> 4, i = s & 15, p0 = 4 * i;  // columns (positions) p0 .. p0 + 3
            const int r0 = warp * 64 + h * 32;
            float2 c0[16], c1[16], c2[16], c3[16];
            {
                const bool va = !tr && vec16(a, lda);
#pragma unroll
                for (int j = 0; j < 16; j += 2) {
                    const int r = r0 + 2 * j;
                    float x[4][4];  // [column][row]
                    if (PRE && pre) {  // W = R^T: W(r, c) = R(c, r)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int rr = r + e;
                            const float4 y = *reinterpret_cast<const float4*>(q.qs + rr * kCols + p0);
                            const float d = q.qdiag[rr];
                            const bool in = rr < n;
                            x[0][e] = in && p0 <= rr ? (p0 < rr ? y.x : d) : 0.f;
                            x[1][e] = in && p0 + 1 <= rr ? (p0 + 1 < rr ? y.y : d) : 0.f;
                            x[2][e] = in && p0 + 2 <= rr ? (p0 + 2 < rr ? y.z : d) : 0.f;
                            x[3][e] = in && p0 + 3 <= rr ? (p0 + 3 < rr ? y.w : d) : 0.f;
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            if (!tr) {
                                const float4 y = p0 + e < nn ? load4(a + (size_t)(p0 + e) * lda + r, va, mm - r)
                                                             : make_float4(0.f, 0.f, 0.f, 0.f);
                                x[e][0] = y.x;
                                x[e][1] = y.y;
                                x[e][2] = y.z;
                                x[e][3] = y.w;
                            } else {
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    x[e][k] = (p0 + e < nn && r + k < mm) ? a[(size_t)(r + k) * lda + p0 + e] : 0.f;
                            }
                        }
                    }
                    c0[j] = make_float2(x[0][0], x[0][1]);
                    c0[j + 1] = make_float2(x[0][2], x[0][3]);
                    c1[j] = make_float2(x[1][0], x[1][1]);
                    c1[j + 1] = make_float2(x[1][2], x[1][3]);
                    c2[j] = make_float2(x[2][0], x[2][1]);
                    c2[j + 1] = make_float2(x[2][2], x[2][3]);
                    c3[j] = make_float2(x[3][0], x[3][1]);
                    c3[j + 1] = make_float2(x[3][2], x[3][3]);
                }
            }
            WvState z;
            z.dL = z.dR = 1.f;
            z.nL = z.nR = 0.f;
            bool converged = false;
            long long total_rot = 0;
            int par = 0;               // parity of the cross-warp reduction slot
            const bool feed = accV && warp == 0;

            while (sweep < sweeps_cap) {
                int rot_sweep = 0;
                if (CARRY) z.nL = z.nR = -1.f;  // every sweep starts from norms summed afresh
#pragma unroll 1
                for (int it = 0; it < 32; ++it) {
                    const int slot = it & 1;
                    if (feed && (sweep > 0 || it >= kRing)) wait_empty(slot);
                    float4* ring = feed ? sh.ring[slot][0] : nullptr;
                    rot_sweep += __popc(wv_step<WW, false, P64, CARRY, P>(c0, c1, c2, c3, z, s, warp, tol, red, par, ring));
                    ring = feed ? sh.ring[slot][1] : nullptr;
                    rot_sweep += __popc(wv_step<WW, true, P64, CARRY, P>(c0, c1, c2, c3, z, s, warp, tol, red, par, ring));
                    if (feed) arrive_full(slot);
                }
                // fold the scales back into the columns
                {
                    const float oL = __shfl_xor_sync(kFullWarp, z.dL, 16), oR = __shfl_xor_sync(kFullWarp, z.dR, 16);
                    const float d0 = h ? oL : z.dL, d1 = h ? oR : z.dR, d2 = h ? z.dL : oL, d3 = h ? z.dR : oR;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        c0[j] = make_float2(c0[j].x * d0, c0[j].y * d0);
                        c1[j] = make_float2(c1[j].x * d1, c1[j].y * d1);
                        c2[j] = make_float2(c2[j].x * d2, c2[j].y * d2);
                        c3[j] = make_float2(c3[j].x * d3, c3[j].y * d3);
                    }
                }
                ++sweep;
                total_rot += rot_sweep;
                converged = rot_sweep == 0;
                if (feed) {
                    // (the V warp has read the previous sweep's scales: it has since emptied ring slots)
                    fold_s[2 * i + h] = make_float2(z.dL, z.dR);
                    if (s == 0) more_s = !converged && sweep < sweeps_cap;
                    bar_arrive<kBarSweep>(64);
                }
                z.dL = z.dR = 1.f;
                if (converged) break;
            }
            if (feed) {  // the last kRing double steps' "empty" arrivals
                wait_empty(0);
                wait_empty(1);
            }

            // ---- sigma = column norms of slot 2 i + h; position p holds column p after an even number of
            // sweeps, 63 - p after an odd one (every sweep reverses the order) ----
            const int sl = 2 * i + h;
            const int colL = sweep & 1 ? kCols - 1 - 2 * sl : 2 * sl, colR = sweep & 1 ? colL - 1 : colL + 1;
            float na, nb;
            {
                auto norm2 = [](const float2(&c)[16]) {
                    float x = 0.f;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        x = fmaf(c[j].x, c[j].x, x);
                        x = fmaf(c[j].y, c[j].y, x);
                    }
                    return x;
                };
                const float x0 = norm2(c0), x1 = norm2(c1), x2 = norm2(c2), x3 = norm2(c3);
                if constexpr (WW == 1) {
                    na = (h ? x2 : x0) + __shfl_xor_sync(kFullWarp, h ? x0 : x2, 16);
                    nb = (h ? x3 : x1) + __shfl_xor_sync(kFullWarp, h ? x1 : x3, 16);
                } else {
                    red.g[par][2 * warp + h][2 * i] = make_float4(x0, x1, 0.f, 0.f);
                    red.g[par][2 * warp + h][2 * i + 1] = make_float4(x2, x3, 0.f, 0.f);
                    bar_wait<kBarRed>(32 * WW);
                    na = nb = 0.f;
#pragma unroll
                    for (int p = 0; p < PARTS; ++p) {
                        na += red.g[par][p][sl].x;
                        nb += red.g[par][p][sl].y;
                    }
                }
            }
            const float sgL = dsqrt(na), sgR = dsqrt(nb);
            const int nn = tr ? again(M + b) : again(N + b);
            if (warp == 0) {
                sig_s[colL] = sgL;
                sig_s[colR] = sgR;
            }
            if constexpr (WW > 1) bar_wait<kBarRed>(32 * WW);
            __syncwarp();
            int rkL = 0, rkR = 0;
            for (int j = 0; j < nn; ++j) {
                const float sj = sig_s[j];
                rkL += (sj > sgL) || (sj == sgL && j < colL);
                rkR += (sj > sgR) || (sj == sgR && j < colR);
            }
            if (colL >= nn) rkL = -1;  // padding columns are not written
            if (colR >= nn) rkR = -1;
            if (warp == 0) {
                float* s_out = Sout[b];
                if (rkL >= 0) s_out[rkL] = sgL;
                if (rkR >= 0) s_out[rkR] = sgR;
                rank_s[2 * sl] = rkL;
                rank_s[2 * sl + 1] = rkR;
                const bool finite = __all_sync(kFullWarp, (rkL < 0 || isfinite(sgL)) && (rkR < 0 || isfinite(sgR)));
                if (s == 0) {
                    info[b] = !finite ? BSVD_INFO_NONFINITE : (converged ? sweep : BSVD_INFO_NOT_CONVERGED + sweep);
                    if (rot_out) rot_out[b] = total_rot;
                }
            }
            int lduw = 0;
            if (float* uw = w_out(lduw)) {
                const int mm = tr ? again(N + b) : again(M + b);
                const float iL = sgL > 0.f ? 1.f / sgL : 0.f, iR = sgR > 0.f ? 1.f / sgR : 0.f;
                const float oL = __shfl_xor_sync(kFullWarp, iL, 16), oR = __shfl_xor_sync(kFullWarp, iR, 16);
                const int ol = __shfl_xor_sync(kFullWarp, rkL, 16), or_ = __shfl_xor_sync(kFullWarp, rkR, 16);
                const bool vu = vec16(uw, lduw);
                auto put = [&](const float2(&c)[16], int rk, float inv) {
                    if (rk < 0) return;
                    float* col = uw + (size_t)rk * lduw + r0;
#pragma unroll
                    for (int j = 0; j < 16; j += 2)
                        store4(col + 2 * j, vu, mm - r0 - 2 * j, c[j].x * inv, c[j].y * inv, c[j + 1].x * inv,
                               c[j + 1].y * inv);
                };
                put(c0, h ? ol : rkL, h ? oL : iL);
                put(c1, h ? or_ : rkR, h ? oR : iR);
                put(c2, h ? rkL : ol, h ? iL : oL);
                put(c3, h ? rkR : or_, h ? iR : oR);
            }
            // V's output follows: preconditioned, the W warp waits for V in vs, else the V warp for the ranks
            if (PRE && pre && accV)
                bar_wait<kBarRanks>(32 * (WW + 1));
            else
                bar_arrive<kBarRanks>(32 * (WW + 1));
        } else {
            // ================================ V ================================
            float2 v[kCols];  // rows s and s + 32 of the column at each position
#pragma unroll
            for (int p = 0; p < kCols; ++p) v[p] = make_float2(p == s ? 1.f : 0.f, p == s + 32 ? 1.f : 0.f);
            {
                // (not a branch around the loop: its second path would keep W's registers live beside V's)
                bool more = accV;
                while (more) {
                    // a double step in one pass over the pairs: the odd step's pair (2p - 1, 2p) follows
                    // the even step's pair (2p, 2p + 1), so every result goes to a register whose old
                    // value has been used, and the swaps of positions cost no moves
#pragma unroll 1
                    for (int it = 0; it < 32; ++it) {
                        const int slot = it & 1;
                        wait_full(slot);
                        float2 up = both(0.f);  // the column at position 2p - 1 between the two steps
#pragma unroll
                        for (int p = 0; p < 32; ++p) {
                            const float4 me = sh.ring[slot][0][p];
                            const float2 x = v[2 * p], y = v[2 * p + 1];
                            const float2 lo = fma2(make_float2(me.z, me.w), x, y);
                            const float2 hi = fma2(make_float2(me.x, me.y), y, x);
                            if (p == 0) {
                                v[0] = lo;
                            } else {
                                const float4 mo = sh.ring[slot][1][p - 1];
                                v[2 * p - 1] = fma2(make_float2(mo.z, mo.w), up, lo);
                                v[2 * p] = fma2(make_float2(mo.x, mo.y), lo, up);
                            }
                            up = hi;
                        }
                        v[kCols - 1] = up;
                        arrive_empty(slot);
                    }
                    bar_wait<kBarSweep>(64);
#pragma unroll
                    for (int p = 0; p < 32; ++p) {
                        const float2 d = fold_s[p];
                        v[2 * p] = make_float2(v[2 * p].x * d.x, v[2 * p].y * d.x);
                        v[2 * p + 1] = make_float2(v[2 * p + 1].x * d.y, v[2 * p + 1].y * d.y);
                    }
                    more = more_s != 0;
                }
            }
            if (PRE && pre && accV) {
#pragma unroll
                for (int p = 0; p < kCols; ++p) {
                    vs[p * kLdV + s] = v[p].x;
                    vs[p * kLdV + s + 32] = v[p].y;
                }
                __syncwarp();
                bar_arrive<kBarRanks>(32 * (WW + 1));
            } else {
                bar_wait<kBarRanks>(32 * (WW + 1));
                int ldvw = 0;
                float* vw = accV ? v_out(ldvw) : nullptr;
                const int nn = tr ? again(M + b) : again(N + b);
#pragma unroll
                for (int p = 0; p < kCols; ++p) {
                    const int rk = vw ? rank_s[p] : -1;   // (null also where the pointer array has a null entry)
                    if (rk >= 0) {
                        if (s < nn) vw[(size_t)rk * ldvw + s] = v[p].x;
                        if (s + 32 < nn) vw[(size_t)rk * ldvw + s + 32] = v[p].y;
                    }
                }
            }
        }

        if constexpr (PRE) {
            // ---- U = Q V_w = H_0 H_1 ... H_{n-1} V_w, the reflectors applied last first, in the QR's layout ----
            if (pre && accV) {
                const int p = warp, cl = 2 * s, cr = 2 * s + 1, rt = p * 32 + s;
                float vL[32], vR[32];
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                    vL[k] = vs[cl * kLdV + p * 32 + k];
                    vR[k] = vs[cr * kLdV + p * 32 + k];
                }
#pragma unroll 1
                for (int j = n - 1; j >= 0; --j) {
                    // the reflector occupies rows j .. n - 1 of column j
                    const float vt = (rt >= j && rt < n) ? q.qs[j * kCols + rt] : 0.f;
                    float* vb = q.v[j & 1] + p * 32;
                    vb[s] = vt;
                    __syncwarp();
                    float dl = 0.f, dr = 0.f;
#pragma unroll
                    for (int k = 0; k < 32; k += 4) {
                        const float4 x = *reinterpret_cast<const float4*>(vb + k);
                        dl = fmaf(x.x, vL[k], dl);
                        dr = fmaf(x.x, vR[k], dr);
                        dl = fmaf(x.y, vL[k + 1], dl);
                        dr = fmaf(x.y, vR[k + 1], dr);
                        dl = fmaf(x.z, vL[k + 2], dl);
                        dr = fmaf(x.z, vR[k + 2], dr);
                        dl = fmaf(x.w, vL[k + 3], dl);
                        dr = fmaf(x.w, vR[k + 3], dr);
                    }
                    q.red[j & 1][p][s] = make_float2(dl, dr);
                    __syncthreads();
                    const float2 w0 = q.red[j & 1][0][s], w1 = q.red[j & 1][1][s];
                    dl = (w0.x + w1.x) * -2.f;
                    dr = (w0.y + w1.y) * -2.f;
#pragma unroll
                    for (int k = 0; k < 32; k += 4) {
                        const float4 x = *reinterpret_cast<const float4*>(vb + k);
                        vL[k] = fmaf(dl, x.x, vL[k]);
                        vR[k] = fmaf(dr, x.x, vR[k]);
                        vL[k + 1] = fmaf(dl, x.y, vL[k + 1]);
                        vR[k + 1] = fmaf(dr, x.y, vR[k + 1]);
                        vL[k + 2] = fmaf(dl, x.z, vL[k + 2]);
                        vR[k + 2] = fmaf(dr, x.z, vR[k + 2]);
                        vL[k + 3] = fmaf(dl, x.w, vL[k + 3]);
                        vR[k + 3] = fmaf(dr, x.w, vR[k + 3]);
                    }
                }
                int ldvw = 0;
                float* vw = v_out(ldvw);
                const int rkL = vw ? rank_s[cl] : -1, rkR = vw ? rank_s[cr] : -1;
                const bool vv = vec16(vw, ldvw);
#pragma unroll
                for (int k = 0; k < 32; k += 4) {
                    const int r = p * 32 + k;
                    if (rkL >= 0)
                        store4(vw + (size_t)rkL * ldvw + r, vv, nn - r, vL[k], vL[k + 1], vL[k + 2], vL[k + 3]);
                    if (rkR >= 0)
                        store4(vw + (size_t)rkR * ldvw + r, vv, nn - r, vR[k], vR[k + 1], vR[k + 2], vR[k + 3]);
                }
            }
        }
        __syncthreads();  // the shared areas are reused by the next item
    }
}

template <int WW, int MINB, bool PRE, bool P64, bool CARRY>
static int launch_wv(int batch, void* const* A, const int* M, const int* N, const int* LDA, void* const* S,
                     void* const* U, const int* LDU, void* const* V, const int* LDV, double tol, int max_sweeps,
                     int* info, long long* rot, cudaStream_t st, ItemList wl)
{
    auto kern = jacobi_wv_kernel<WW, MINB, PRE, P64, CARRY>;
    // the whole of the SM's shared memory for the CTAs that the registers allow
    if (cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) !=
        cudaSuccess)
        return BSVD_ERR_CUDA;
    const int grid = item_grid(kern, 32 * (WW + 1), 0, wl, batch, st);
    if (grid == 0) return BSVD_ERR_CUDA;
    kern<<<grid, 32 * (WW + 1), 0, st>>>(batch, (float* const*)A, M, N, LDA, (float* const*)S, (float* const*)U, LDU,
                                        (float* const*)V, LDV, tol, max_sweeps, info, rot, wl);
    return cudaGetLastError() == cudaSuccess ? BSVD_SUCCESS : BSVD_ERR_CUDA;
}

int launch_jacobi_wv(bool rows128, bool pre, bool p64, bool carry, int batch, void* const* A, const int* M,
                     const int* N, const int* LDA, void* const* S, void* const* U, const int* LDU, void* const* V,
                     const int* LDV, double tol, int max_sweeps, int* info, long long* rot, cudaStream_t st,
                     ItemList wl)
{
#define BSVD_WV(WW_, MINB_, PRE_, P64_, CARRY_)                                                                     \
    launch_wv<WW_, MINB_, PRE_, P64_, CARRY_>(batch, A, M, N, LDA, S, U, LDU, V, LDV, tol, max_sweeps, info, rot, st, wl)
    if (rows128) return pre || p64 || carry ? BSVD_ERR_UNSUPPORTED : BSVD_WV(2, 4, false, false, false);
    if (p64) return carry ? BSVD_ERR_UNSUPPORTED : (pre ? BSVD_WV(1, 6, true, true, false) : BSVD_WV(1, 6, false, true, false));
    if (pre) return carry ? BSVD_WV(1, 6, true, false, true) : BSVD_WV(1, 6, true, false, false);
    return carry ? BSVD_WV(1, 6, false, false, true) : BSVD_WV(1, 6, false, false, false);
#undef BSVD_WV
}

}  // namespace bsvd
