// jacobi_rx.cu -- one-sided Jacobi SVD of FP32 matrices up to 128 x 128, one CTA per matrix, W and the
// accumulated rotations V in registers of different warps (Algorithm 2, Section 2.2; the shared-memory
// kernel of Section 5, re-arranged for sm_103a).
//
// The pair ordering is the odd-even transposition with exchange of the register tier: 2 NS positions,
// even steps pair (2s, 2s + 1), odd steps (2s + 1, 2s + 2), every processed pair swaps positions, 2 NS
// steps per sweep; on odd steps the wrap slot NS - 1, holding positions 2 NS - 1 and 0, idles.
//   W warps      (a warp per eight slots) slot s is lanes 4 s .. 4 s + 3; lane h holds the rows 4 q + h of the slot's two columns,
//                pairs of q packed for two-element FMAs.  A Gram entry is summed in eight chains (rows mod 8)
//                and a tree, the order in which eight lanes per slot would sum it.  One column per slot moves
//                to the neighbouring slot each step, through a double-buffered area in shared memory (16-byte
//                accesses) and one barrier of the W warps.
//   V warps      (a warp per 16 slots) thread t holds row t of V, the columns in registers by position: a step is two rotations'
//                worth of FMAs per pair and no exchange (the swap renames registers).  The steps' (c, s) come
//                through a ring in shared memory; the V warps run up to two double steps behind.
// Bound by the W warps' dependent chain of a step (dot products, parameters, rotation, exchange); the V
// warps fill the schedulers meanwhile.  With W and V in the same lanes, eight lanes a slot, both exchanged
// through shared memory and the parameters computed eight times over, 1000 matrices of 127 x 100 took
// 18.6 ms; it takes 12.2 ms here.  Up to 16 columns that form is the better one and the second kernel below.
#include <cuda_runtime.h>

#include "common.cuh"
#include "launch.cuh"
#include "rnmath.cuh"

namespace bsvd {

namespace {

constexpr int kRxRows = 128;
constexpr int kRxQuarter = 36, kRxLd = 4 * kRxQuarter;  // exchange area: strides of a lane's quarter column and of a
                                                        // slot: eight lanes' 16-byte accesses in distinct banks
// threads of the form for up to SLOTS slots: W, V (a row each), both
template <int SLOTS>
struct RxThreads {
    static constexpr int w = 4 * SLOTS, v = (2 * SLOTS + 31) / 32 * 32, all = w + v;
};
constexpr unsigned kRxFull = 0xffffffffu;

template <int SLOTS>
struct RxShared {
    float x[2][SLOTS * kRxLd];          // columns on the move, by step parity and sending slot
    float4 ring[2][2][SLOTS / 2];       // per double step and step: (c, s) of two pairs
    float sig[2 * SLOTS];               // singular values by column
    int rank[2 * SLOTS];                // by position (-1: padding)
    int count[RxThreads<SLOTS>::w / 32];   // rotations of a sweep, per W warp
    int more[2];                        // another sweep follows (by sweep parity)
};

// named barriers (0 is the CTA's): the W warps' own; ring slots full and empty, a sweep's end
template <int ID, int N>
__device__ __forceinline__ void rx_wait() { asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(N) : "memory"); }
template <int ID, int N>
__device__ __forceinline__ void rx_arrive() { asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(N) : "memory"); }
constexpr int kRxW = 1, kRxFullBar = 2, kRxEmptyBar = 4, kRxSweep = 6, kRxRanks = 7;
// (a barrier that both sides would reach with the same instruction is merged by the compiler into one block,
// where W's and V's registers would be live together)
template <int N> __device__ __forceinline__ void rx_wait_full(int slot) { slot ? rx_wait<kRxFullBar + 1, N>() : rx_wait<kRxFullBar, N>(); }
template <int N> __device__ __forceinline__ void rx_wait_empty(int slot) { slot ? rx_wait<kRxEmptyBar + 1, N>() : rx_wait<kRxEmptyBar, N>(); }
template <int N> __device__ __forceinline__ void rx_arrive_full(int slot) { slot ? rx_arrive<kRxFullBar + 1, N>() : rx_arrive<kRxFullBar, N>(); }
template <int N> __device__ __forceinline__ void rx_arrive_empty(int slot) { slot ? rx_arrive<kRxEmptyBar + 1, N>() : rx_arrive<kRxEmptyBar, N>(); }

__device__ __forceinline__ float2 rx_both(float x) { return make_float2(x, x); }

// this lane's two chains of x . y, added as eight lanes' butterfly over 4 would; then the butterflies over 2 and 1
__device__ __forceinline__ float rx_dot(const float2 (&x)[16], const float2 (&y)[16])
{
    float2 a = rx_both(0.f);
#pragma unroll
    for (int q = 0; q < 16; ++q) a = __ffma2_rn(x[q], y[q], a);
    float s = a.x + a.y;
    s += __shfl_xor_sync(kRxFull, s, 2);
    s += __shfl_xor_sync(kRxFull, s, 1);
    return s;
}

__device__ __noinline__ bool rx_rotation_slow(float al, float be, float ga, float tol, float* cs)
{
    return jacobi_rotation<float>(al, be, ga, tol, cs[0], cs[1]);
}

// rot(G) of jacobi_rotation<float>, the same numbers: by branch-free correctly rounded operations when every
// lane of the warp is inside their range, else by jacobi_rotation itself
template <typename P>
__device__ __forceinline__ bool rx_rotation(float al, float be, float ga, P tol, float& c, float& s)
{
    c = 1.f;
    s = 0.f;
    if constexpr (sizeof(P) == 8) {
        P cp, sp;
        if (!jacobi_rotation<P>(P(al), P(be), P(ga), tol, cp, sp)) return false;
        c = float(cp);
        s = float(sp);
        return true;
    } else {
        const bool pos = al > 0.f && be > 0.f;
        const float d = be - al, g2 = 2.f * ga;
        const bool rot = pos && !(fabsf(ga) <= tol * rn_sqrt(al) * rn_sqrt(be));
        const float zeta = rn_div(d, g2), az = fabsf(zeta);
        float t = rn_rcp(az + rn_sqrt(fmaf(zeta, zeta, 1.f)));
        t = zeta >= 0.f ? t : -t;
        const float cf = rn_rsqrt12(fmaf(t, t, 1.f));
        auto in = [](float x) { return x >= 0x1p-100f && x <= 0x1p100f; };
        // (the test itself needs the norms' range, the parameters the rest; zeta, 0 or at least 2^-26 since d is a
        // multiple of a last place and |ga| at most the norms, is then a quotient in range, and its square plus 1
        // below 2^118)
        const bool safe = in(al) && in(be) && (!rot || (in(fabsf(g2)) && (d == 0.f || in(fabsf(d))) && az < 0x1p59f));
        if (__any_sync(kRxFull, pos && !safe)) {
            float cs[2];
            if (!rx_rotation_slow(al, be, ga, tol, cs)) return false;
            c = cs[0];
            s = cs[1];
            return true;
        }
        if (rot) {
            c = cf;
            s = cf * t;
        }
        return rot;
    }
}

}  // namespace

// P: precision of the rotation parameters and the rotation test (float, or double)
template <typename P, int SLOTS, int MINB>
__global__ void __launch_bounds__(RxThreads<SLOTS>::all, MINB)
    jacobi_rx_kernel(int batch, int max_mm, int max_np, float* const* A, const int* M, const int* N, const int* LDA,
                     float* const* Sout, float* const* U, const int* LDU, float* const* V, const int* LDV,
                     double tol_in, int max_sweeps, int* info, long long* rot_out, ItemList wl)
{
    constexpr int kW = RxThreads<SLOTS>::w, kAll = RxThreads<SLOTS>::all;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RxShared<SLOTS>& sh = *reinterpret_cast<RxShared<SLOTS>*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool is_v = tid >= kW;

    for (int b = item_first(wl, batch); b >= 0; b = item_next(wl, batch, b)) {
        const int m = M[b], n = N[b], lda = LDA[b];
        const bool tr = m < n;
        const int mm = tr ? n : m;  // working rows
        const int nn = tr ? m : n;  // working columns
        const int np = nn + (nn & 1);
        const int ns = np / 2;      // slots of this matrix
        const bool wantU = U != nullptr, wantV = V != nullptr;
        const int ldu = wantU ? LDU[b] : 1, ldvo = wantV ? LDV[b] : 1;
        const bool bad = m < 0 || n < 0 || mm > max_mm || np > max_np || mm > kRxRows || np > 2 * SLOTS ||
                         lda < (m > 1 ? m : 1) || (wantU && ldu < (m > 1 ? m : 1)) ||
                         (wantV && ldvo < (n > 1 ? n : 1));
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
        const bool accV = tr ? wantU : wantV;
        float* uw = tr ? (wantV ? V[b] : nullptr) : (wantU ? U[b] : nullptr);  // receives W / sigma
        const int lduw = tr ? ldvo : ldu;
        float* vw = tr ? (wantU ? U[b] : nullptr) : (wantV ? V[b] : nullptr);  // receives V
        const int ldvw = tr ? ldu : ldvo;

        if (!is_v) {
            // ================================ W ================================
            const int s = tid >> 2, h = tid & 3;
            const bool live = s < ns, wrap = s == ns - 1;
            const bool wrap_warp = (ns - 1) >> 3 == warp;
            const float* a = A[b];
            float2 L[16], R[16];   // element q: rows 8 q + h and 8 q + 4 + h
            {
                auto elem = [&](int c, int r) -> float {
                    if (!live || c >= nn || r >= mm) return 0.f;
                    return tr ? a[(size_t)r * lda + c] : a[(size_t)c * lda + r];
                };
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const int r = 8 * q + h;
                    L[q] = make_float2(elem(2 * s, r), elem(2 * s, r + 4));
                    R[q] = make_float2(elem(2 * s + 1, r), elem(2 * s + 1, r + 4));
                }
            }
            const P tol = tol_in > 0.0 ? P(tol_in) : P(dsqrt(double(mm)) * Unit<float>::value);
            const int sweeps_cap = max_sweeps > 0 ? max_sweeps : 30;
            int sweep = 0, slot = 0;
            bool converged = false;
            long long total_rot = 0, sent = 0;
            float4* out = reinterpret_cast<float4*>(sh.x[0] + s * kRxLd + h * kRxQuarter);
            // (slots past NS exchange zeros with themselves)
            const int up = !live ? s : (wrap ? 0 : s + 1), down = !live ? s : (s == 0 ? ns - 1 : s - 1);
            const float4* from_up = reinterpret_cast<const float4*>(sh.x[0] + up * kRxLd + h * kRxQuarter);
            const float4* from_dn = reinterpret_cast<const float4*>(sh.x[1] + down * kRxLd + h * kRxQuarter);
            float4* out1 = reinterpret_cast<float4*>(sh.x[1] + s * kRxLd + h * kRxQuarter);
            float2* ring = reinterpret_cast<float2*>(sh.ring);

            while (sweep < sweeps_cap) {
                int rot_sweep = 0;
#pragma unroll 1
                for (int it = 0; it < ns; ++it) {
                    if (accV && sent >= 2) rx_wait_empty<kAll>(slot);
                    // even step: positions 2s and 2s + 1; the right column moves one slot down
                    {
                        const float al = rx_dot(L, L), be = rx_dot(R, R), ga = rx_dot(L, R);
                        float c, sn;
                        const bool rot = rx_rotation<P>(live ? al : 0.f, be, ga, tol, c, sn);
                        const unsigned rots = __ballot_sync(kRxFull, rot && h == 0);
                        rot_sweep += __popc(rots);
                        if (accV && h == 0) ring[(2 * slot) * SLOTS + s] = make_float2(c, sn);
                        const float2 c2 = rx_both(c), s2 = rx_both(sn), m2 = rx_both(-sn);
                        if (rots) {
#pragma unroll
                            for (int q = 0; q < 16; ++q) {
                                const float2 y = __ffma2_rn(s2, L[q], __fmul2_rn(c2, R[q]));
                                L[q] = __ffma2_rn(c2, L[q], __fmul2_rn(m2, R[q]));
                                R[q] = y;
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 16; q += 2) out[q / 2] = make_float4(R[q].x, R[q].y, R[q + 1].x, R[q + 1].y);
                        rx_wait<kRxW, kW>();
#pragma unroll
                        for (int q = 0; q < 16; q += 2) {
                            const float4 v = from_up[q / 2];
                            R[q] = make_float2(v.x, v.y);
                            R[q + 1] = make_float2(v.z, v.w);
                        }
                    }
                    // odd step: positions 2s + 1 and 2s + 2; the left column moves one slot up.  The wrap slot
                    // does not rotate: it hands over its right column and keeps its left one as the right
                    {
                        const float al = rx_dot(L, L), be = rx_dot(R, R), ga = rx_dot(L, R);
                        float c, sn;
                        const bool rot = rx_rotation<P>(live && !wrap ? al : 0.f, be, ga, tol, c, sn);
                        const unsigned rots = __ballot_sync(kRxFull, rot && h == 0);
                        rot_sweep += __popc(rots);
                        // (0, 1) keeps position 2 NS - 1 apart from the zero columns past it in V
                        if (accV && h == 0) ring[(2 * slot + 1) * SLOTS + s] = wrap ? make_float2(0.f, 1.f) : make_float2(c, sn);
                        const float2 c2 = rx_both(c), s2 = rx_both(sn), m2 = rx_both(-sn);
                        if (rots) {
#pragma unroll
                            for (int q = 0; q < 16; ++q) {
                                const float2 x = __ffma2_rn(c2, L[q], __fmul2_rn(m2, R[q]));
                                R[q] = __ffma2_rn(s2, L[q], __fmul2_rn(c2, R[q]));
                                L[q] = x;
                            }
                        }
                        if (wrap_warp) {
#pragma unroll
                            for (int q = 0; q < 16; ++q) {
                                const float2 l = L[q], r = R[q];
                                L[q] = make_float2(wrap ? r.x : l.x, wrap ? r.y : l.y);
                                R[q] = make_float2(wrap ? l.x : r.x, wrap ? l.y : r.y);
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 16; q += 2) out1[q / 2] = make_float4(L[q].x, L[q].y, L[q + 1].x, L[q + 1].y);
                        rx_wait<kRxW, kW>();
#pragma unroll
                        for (int q = 0; q < 16; q += 2) {
                            const float4 v = from_dn[q / 2];
                            L[q] = make_float2(v.x, v.y);
                            L[q + 1] = make_float2(v.z, v.w);
                        }
                    }
                    if (accV) {
                        rx_arrive_full<kAll>(slot);
                        slot ^= 1;
                        ++sent;
                    }
                }
                if (lane == 0) sh.count[warp] = rot_sweep;
                rx_wait<kRxW, kW>();
                rot_sweep = 0;
#pragma unroll
                for (int w = 0; w < kW / 32; ++w) rot_sweep += sh.count[w];
                ++sweep;
                total_rot += rot_sweep;
                converged = rot_sweep == 0;
                if (accV) {   // (a sweep of few columns has fewer double steps than the ring: both sides wait)
                    if (tid == 0) sh.more[sweep & 1] = !converged && sweep < sweeps_cap;
                    rx_wait<kRxSweep, kAll>();
                }
                if (converged) break;
                rx_wait<kRxW, kW>();   // the counts have been read
            }
            // the last double steps' "empty" arrivals
            if (sent >= 2) rx_wait_empty<kAll>(slot);
            if (sent >= 1) rx_wait_empty<kAll>(slot ^ 1);

            // ---- sigma_j = ||w_j||; position p holds column p after an even number of sweeps, 2 NS - 1 - p
            // after an odd one (every sweep reverses the order) ----
            const int colL = sweep & 1 ? np - 1 - 2 * s : 2 * s, colR = sweep & 1 ? colL - 1 : colL + 1;
            const float sl = rx_dot(L, L), sr = rx_dot(R, R);
            const float sgL = dsqrt(sl), sgR = dsqrt(sr);
            if (live && h == 0) {
                if (colL < nn) sh.sig[colL] = sgL;
                if (colR < nn) sh.sig[colR] = sgR;
            }
            rx_wait<kRxW, kW>();
            // ---- descending rank, ties in column order ----
            int rkL = 0, rkR = 0;
            for (int j = 0; j < nn; ++j) {
                const float sj = sh.sig[j];
                rkL += (sj > sgL) || (sj == sgL && j < colL);
                rkR += (sj > sgR) || (sj == sgR && j < colR);
            }
            if (!live || colL >= nn) rkL = -1;
            if (!live || colR >= nn) rkR = -1;
            if (live && h == 0) {
                sh.rank[2 * s] = rkL;
                sh.rank[2 * s + 1] = rkR;
                float* s_out = Sout[b];
                if (rkL >= 0) s_out[rkL] = sgL;
                if (rkR >= 0) s_out[rkR] = sgR;
            }
            if (tid == 0) {
                bool finite = true;
                for (int j = 0; j < nn; ++j) finite = finite && isfinite(sh.sig[j]);
                info[b] = !finite ? BSVD_INFO_NONFINITE : (converged ? sweep : BSVD_INFO_NOT_CONVERGED + sweep);
                if (rot_out) rot_out[b] = total_rot;
            }
            rx_arrive<kRxRanks, kAll>();   // the ranks are there
            if (uw) {
                auto put = [&](const float2(&x)[16], int rk, float sg) {
                    if (rk < 0) return;
                    const float inv = sg > 0.f ? 1.f / sg : 0.f;
                    float* col = uw + (size_t)rk * lduw;
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const int r = 8 * q + h;
                        if (r < mm) col[r] = x[q].x * inv;
                        if (r + 4 < mm) col[r + 4] = x[q].y * inv;
                    }
                };
                put(L, rkL, sgL);
                put(R, rkR, sgR);
            }
        } else {
            // ================================ V ================================
            const int row = tid - kW;
            float v[2 * SLOTS];   // row `row` of the column at each position
#pragma unroll
            for (int p = 0; p < 2 * SLOTS; ++p) v[p] = p == row ? 1.f : 0.f;
            {
                int slot = 0, sweep = 0;
                // (not a branch around the loop: its second path would keep W's registers live beside V's)
                bool more = accV;
                while (more) {
#pragma unroll 1
                    for (int it = 0; it < ns; ++it) {
                        // a double step in one pass: the odd step's pair (2p - 1, 2p) follows the even step's
                        // pair (2p, 2p + 1), so every result goes to a register whose old value has been used
                        rx_wait_full<kAll>(slot);
                        const float4* re = sh.ring[slot][0];
                        const float4* ro = sh.ring[slot][1];
                        float up = 0.f, oc = 1.f, os = 0.f;   // position 2p - 1 between the steps; its (c, s)
#pragma unroll
                        for (int p = 0; p < SLOTS; p += 2) {
                            const float4 e = re[p / 2], o = ro[p / 2];
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                const float c = k ? e.z : e.x, sn = k ? e.w : e.y;
                                const float x = v[2 * (p + k)], y = v[2 * (p + k) + 1];
                                const float lo = fmaf(sn, x, c * y), hi = fmaf(c, x, -sn * y);   // R', L'
                                if (p + k == 0) {
                                    v[0] = lo;
                                } else {
                                    v[2 * (p + k) - 1] = fmaf(os, up, oc * lo);
                                    v[2 * (p + k)] = fmaf(oc, up, -os * lo);
                                }
                                up = hi;
                                oc = k ? o.z : o.x;
                                os = k ? o.w : o.y;
                            }
                        }
                        v[2 * SLOTS - 1] = up;
                        rx_arrive_empty<kAll>(slot);
                        slot ^= 1;
                    }
                    rx_wait<kRxSweep, kAll>();
                    ++sweep;
                    more = sh.more[sweep & 1] != 0;
                }
            }
            rx_wait<kRxRanks, kAll>();   // the ranks are there
            if (accV && vw && row < nn) {   // (a null entry of the pointer array: that matrix's V is not written)
#pragma unroll
                for (int p = 0; p < 2 * SLOTS; ++p) {
                    const int rk = p < np ? sh.rank[p] : -1;
                    if (rk >= 0) vw[(size_t)rk * ldvw + row] = v[p];
                }
            }
        }
        __syncthreads();   // the shared areas are reused by the next item
    }
}

template <typename P, int SLOTS, int MINB>
static int launch_rx(int batch, int max_mm, int max_np, void* const* A, const int* M, const int* N, const int* LDA,
                     void* const* S, void* const* U, const int* LDU, void* const* V, const int* LDV, double tol,
                     int max_sweeps, int* info, long long* rot, cudaStream_t st, ItemList wl)
{
    auto kern = jacobi_rx_kernel<P, SLOTS, MINB>;
    const size_t smem = sizeof(RxShared<SLOTS>);
    constexpr int threads = RxThreads<SLOTS>::all;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return BSVD_ERR_CUDA;
    const int grid = item_grid(kern, threads, smem, wl, batch, st);
    if (grid == 0) return BSVD_ERR_CUDA;
    kern<<<grid, threads, smem, st>>>(batch, max_mm, max_np, (float* const*)A, M, N, LDA, (float* const*)S,
                                      (float* const*)U, LDU, (float* const*)V, LDV, tol, max_sweeps, info, rot, wl);
    return cudaGetLastError() == cudaSuccess ? BSVD_SUCCESS : BSVD_ERR_CUDA;
}

// ---- up to 16 columns: W and V in the same lanes ----
//
// Eight lanes per slot, as many slots as the batch's bound has pairs: slot s (lanes 8 s .. 8 s + 7) keeps rows
// g + 8 k of its two columns of W and of V, and one column of each moves to the neighbouring slot per step,
// through a double-buffered area in shared memory and one barrier.  The sums, parameters and rotations
// are the form's above, so results are the same bit for bit.  A matrix of n columns takes 4 n
// threads and n / 2 slots of shared memory and no warp waits for another's ring, so far more matrices share an SM:
// 20 000 matrices of 128 x 4 take 0.14 ms, 2.6 ms in the form above with 48 slots; of 128 x 16 1.08 ms, 1.39 ms in the
// form above with 8 slots (1.61 ms with room for 128 rows of V in these lanes).
constexpr int kRx8Cols = 16, kRx8Lanes = 8;
constexpr int kRx8W = kRxRows / kRx8Lanes, kRx8V = kRx8Cols / kRx8Lanes;         // rows per lane
constexpr int kRx8LdW = kRxRows + 8, kRx8LdV = kRx8Cols + 8;                      // slots 8 banks apart

__global__ void __launch_bounds__(kRx8Cols / 2 * kRx8Lanes)
    jacobi_rx8_kernel(int batch, int max_mm, int max_np, float* const* A, const int* M, const int* N, const int* LDA,
                      float* const* Sout, float* const* U, const int* LDU, float* const* V, const int* LDV,
                      double tol_in, int max_sweeps, int* info, long long* rot_out, ItemList wl)
{
    constexpr int G = kRx8Lanes;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nslot_max = max_np / 2;
    float* xw = reinterpret_cast<float*>(smem_raw);              // [2][nslot_max][kRx8LdW]
    float* xv = xw + 2 * nslot_max * kRx8LdW;                    // [2][nslot_max][kRx8LdV]
    int* xc = reinterpret_cast<int*>(xv + 2 * nslot_max * kRx8LdV);   // [2][nslot_max] column ids
    float* sig = reinterpret_cast<float*>(xc + 2 * nslot_max);   // [max_np] singular values by column id
    const int tid = threadIdx.x;
    const int s = tid / G, g = tid % G;

    for (int b = item_first(wl, batch); b >= 0; b = item_next(wl, batch, b)) {
        const int m = M[b], n = N[b], lda = LDA[b];
        const bool tr = m < n;
        const int mm = tr ? n : m, nn = tr ? m : n;
        const int np = (nn + 1) & ~1, ns = np / 2;
        const bool wantU = U != nullptr, wantV = V != nullptr;
        const int ldu = wantU ? LDU[b] : 1, ldvo = wantV ? LDV[b] : 1;
        const bool bad = m < 0 || n < 0 || mm > max_mm || np > max_np || mm > kRxRows || np > kRx8Cols ||
                         lda < (m > 1 ? m : 1) || (wantU && ldu < (m > 1 ? m : 1)) ||
                         (wantV && ldvo < (n > 1 ? n : 1));
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
        const bool live = s < ns, wrap = s == ns - 1;
        int colL = 2 * s, colR = 2 * s + 1;
        const float* a = A[b];
        float L[kRx8W], R[kRx8W], vL[kRx8V], vR[kRx8V];
#pragma unroll
        for (int k = 0; k < kRx8W; ++k) {
            const int r = g + G * k;
            auto elem = [&](int c) -> float {
                if (!live || c >= nn || r >= mm) return 0.f;
                return tr ? a[(size_t)r * lda + c] : a[(size_t)c * lda + r];
            };
            L[k] = elem(colL);
            R[k] = elem(colR);
        }
#pragma unroll
        for (int k = 0; k < kRx8V; ++k) {
            const int r = g + G * k;
            vL[k] = r == colL ? 1.f : 0.f;
            vR[k] = r == colR ? 1.f : 0.f;
        }
        const float tol = tol_in > 0.0 ? float(tol_in) : float(dsqrt(double(mm)) * Unit<float>::value);
        const int sweeps_cap = max_sweeps > 0 ? max_sweeps : 30;
        int sweep = 0, par = 0;
        bool converged = false;
        long long total_rot = 0;
        while (sweep < sweeps_cap) {
            int rot_sweep = 0;
            for (int st = 0; st < 2 * ns; ++st) {
                const bool odd = st & 1;
                float al = 0.f, be = 0.f, ga = 0.f;
#pragma unroll
                for (int k = 0; k < kRx8W; ++k) {
                    al = fmaf(L[k], L[k], al);
                    be = fmaf(R[k], R[k], be);
                    ga = fmaf(L[k], R[k], ga);
                }
                al = group_sum<G>(al);
                be = group_sum<G>(be);
                ga = group_sum<G>(ga);
                float c, sn;
                const bool rot = live && !(odd && wrap) && jacobi_rotation<float>(al, be, ga, tol, c, sn);
                if (rot) {
#pragma unroll
                    for (int k = 0; k < kRx8W; ++k) {
                        const float x = fmaf(c, L[k], -sn * R[k]);
                        R[k] = fmaf(sn, L[k], c * R[k]);
                        L[k] = x;
                    }
#pragma unroll
                    for (int k = 0; k < kRx8V; ++k) {
                        const float x = fmaf(c, vL[k], -sn * vR[k]);
                        vR[k] = fmaf(sn, vL[k], c * vR[k]);
                        vL[k] = x;
                    }
                }
                // even -> odd: the right column moves one slot down; odd -> even: the left column moves one
                // slot up, except the wrap slot's right column (it did not rotate)
                if (live) {
                    float* ow = xw + (par * nslot_max + s) * kRx8LdW + g;
                    float* ov = xv + (par * nslot_max + s) * kRx8LdV + g;
                    if (!odd || wrap) {
#pragma unroll
                        for (int k = 0; k < kRx8W; ++k) ow[G * k] = R[k];
#pragma unroll
                        for (int k = 0; k < kRx8V; ++k) ov[G * k] = vR[k];
                        if (g == 0) xc[par * nslot_max + s] = colR;
                    } else {
#pragma unroll
                        for (int k = 0; k < kRx8W; ++k) ow[G * k] = L[k];
#pragma unroll
                        for (int k = 0; k < kRx8V; ++k) ov[G * k] = vL[k];
                        if (g == 0) xc[par * nslot_max + s] = colL;
                    }
                }
                rot_sweep += __syncthreads_count(rot && g == 0);
                if (live) {
                    const int src = !odd ? (wrap ? 0 : s + 1) : (s == 0 ? ns - 1 : s - 1);
                    const float* iw = xw + (par * nslot_max + src) * kRx8LdW + g;
                    const float* iv = xv + (par * nslot_max + src) * kRx8LdV + g;
                    const int col = xc[par * nslot_max + src];
                    if (!odd) {
#pragma unroll
                        for (int k = 0; k < kRx8W; ++k) R[k] = iw[G * k];
#pragma unroll
                        for (int k = 0; k < kRx8V; ++k) vR[k] = iv[G * k];
                        colR = col;
                    } else {
                        if (wrap) {   // the wrap slot keeps its left column as the right one
#pragma unroll
                            for (int k = 0; k < kRx8W; ++k) R[k] = L[k];
#pragma unroll
                            for (int k = 0; k < kRx8V; ++k) vR[k] = vL[k];
                            colR = colL;
                        }
#pragma unroll
                        for (int k = 0; k < kRx8W; ++k) L[k] = iw[G * k];
#pragma unroll
                        for (int k = 0; k < kRx8V; ++k) vL[k] = iv[G * k];
                        colL = col;
                    }
                }
                par ^= 1;
            }
            ++sweep;
            total_rot += rot_sweep;
            if (rot_sweep == 0) {
                converged = true;
                break;
            }
        }
        // ---- sigma_j = ||w_j|| by column id, descending rank, ties in column order ----
        float sl = 0.f, sr = 0.f;
#pragma unroll
        for (int k = 0; k < kRx8W; ++k) {
            sl = fmaf(L[k], L[k], sl);
            sr = fmaf(R[k], R[k], sr);
        }
        const float sgL = dsqrt(group_sum<G>(sl)), sgR = dsqrt(group_sum<G>(sr));
        if (live && g == 0) {
            if (colL < nn) sig[colL] = sgL;
            if (colR < nn) sig[colR] = sgR;
        }
        __syncthreads();
        if (live) {
            int rkL = 0, rkR = 0;
            for (int j = 0; j < nn; ++j) {
                const float sj = sig[j];
                rkL += (sj > sgL) || (sj == sgL && j < colL);
                rkR += (sj > sgR) || (sj == sgR && j < colR);
            }
            if (g == 0) {
                if (colL < nn) Sout[b][rkL] = sgL;
                if (colR < nn) Sout[b][rkR] = sgR;
            }
            float* uw = tr ? (wantV ? V[b] : nullptr) : (wantU ? U[b] : nullptr);   // receives W / sigma
            const int lduw = tr ? ldvo : ldu;
            float* vw = tr ? (wantU ? U[b] : nullptr) : (wantV ? V[b] : nullptr);   // receives V
            const int ldvw = tr ? ldu : ldvo;
            auto put = [&](const float(&w)[kRx8W], const float(&v)[kRx8V], int rk, float sg) {
                const float inv = sg > 0.f ? 1.f / sg : 0.f;
                if (uw) {
#pragma unroll
                    for (int k = 0; k < kRx8W; ++k)
                        if (g + G * k < mm) uw[(size_t)rk * lduw + g + G * k] = w[k] * inv;
                }
                if (vw) {
#pragma unroll
                    for (int k = 0; k < kRx8V; ++k)
                        if (g + G * k < nn) vw[(size_t)rk * ldvw + g + G * k] = v[k];
                }
            };
            if (colL < nn) put(L, vL, rkL, sgL);
            if (colR < nn) put(R, vR, rkR, sgR);
        }
        if (tid == 0) {
            bool finite = true;
            for (int j = 0; j < nn; ++j) finite = finite && isfinite(sig[j]);
            info[b] = !finite ? BSVD_INFO_NONFINITE : (converged ? sweep : BSVD_INFO_NOT_CONVERGED + sweep);
            if (rot_out) rot_out[b] = total_rot;
        }
        __syncthreads();
    }
}

static int launch_rx8(int batch, int max_mm, int max_np, void* const* A, const int* M, const int* N, const int* LDA,
                      void* const* S, void* const* U, const int* LDU, void* const* V, const int* LDV, double tol,
                      int max_sweeps, int* info, long long* rot, cudaStream_t st, ItemList wl)
{
    auto kern = jacobi_rx8_kernel;
    const int ns = max_np / 2;
    const size_t smem = sizeof(float) * (2 * ns * (kRx8LdW + kRx8LdV) + 2 * ns + max_np);
    const int threads = (ns * kRx8Lanes + 31) & ~31;
    const int grid = item_grid(kern, threads, smem, wl, batch, st);
    if (grid == 0) return BSVD_ERR_CUDA;
    kern<<<grid, threads, smem, st>>>(batch, max_mm, max_np, (float* const*)A, M, N, LDA, (float* const*)S,
                                      (float* const*)U, LDU, (float* const*)V, LDV, tol, max_sweeps, info, rot, wl);
    return cudaGetLastError() == cudaSuccess ? BSVD_SUCCESS : BSVD_ERR_CUDA;
}

// FP32 matrices with max(m, n) <= 128.  Returns BSVD_ERR_UNSUPPORTED for other shapes (the caller then takes
// the shared tier).  Threads, shared memory and the V warps' work grow with the slots, so the instances follow the
// bound's columns: 1000 of 127 x 100 take 13.1 ms with room for 128 columns, 12.2 ms with 112; up to 64 columns
// two to five matrices share an SM (2000 matrices, eight lanes a slot for W and V / here: 64 x 32 0.85 / 0.52 ms,
// 40 x 40 1.75 / 1.37 ms, 64 x 64 4.40 / 3.03 ms).  FP64 parameters, which only the randomized SVD's small SVDs of
// more than 64 columns take, bound a step by themselves: one instance.
int launch_jacobi_rx(int batch, int max_m, int max_n, void* const* A, const int* M, const int* N, const int* LDA,
                     void* const* S, void* const* U, const int* LDU, void* const* V, const int* LDV, double tol,
                     int max_sweeps, int* info, long long* rot, cudaStream_t st, ItemList wl, bool p64)
{
    const int max_mm = max_m > max_n ? max_m : max_n;
    const int max_nn = max_m > max_n ? max_n : max_m;
    const int max_np = (max_nn + 1) & ~1;
    if (max_mm > kRxRows || max_np > kRxRows || max_np < 2) return BSVD_ERR_UNSUPPORTED;
#define BSVD_RX(P_, SLOTS_, MINB_)                                                                                  \
    launch_rx<P_, SLOTS_, MINB_>(batch, max_mm, max_np, A, M, N, LDA, S, U, LDU, V, LDV, tol, max_sweeps, info, rot, \
                                 st, wl)
    if (p64) return BSVD_RX(double, 64, 1);
    if (max_np <= kRx8Cols)
        return launch_rx8(batch, max_mm, max_np, A, M, N, LDA, S, U, LDU, V, LDV, tol, max_sweeps, info, rot, st, wl);
    if (max_np <= 32) return BSVD_RX(float, 16, 5);
    if (max_np <= 48) return BSVD_RX(float, 24, 3);
    if (max_np <= 64) return BSVD_RX(float, 32, 2);
    return max_np <= 96 ? BSVD_RX(float, 48, 1) : (max_np <= 112 ? BSVD_RX(float, 56, 1) : BSVD_RX(float, 64, 1));
#undef BSVD_RX
}

}  // namespace bsvd
