// jacobi_rx.cu -- one-sided Jacobi SVD of FP32 matrices up to 128 x 128, one CTA per matrix, W and the
// accumulated rotations V in registers of different warps (Algorithm 2, Section 2.2; the shared-memory
// kernel of Section 5, re-arranged for sm_103a).
//
// The pair ordering is the odd-even transposition with exchange of the register tier: 2 NS positions,
// even steps pair (2s, 2s + 1), odd steps (2s + 1, 2s + 2), every processed pair swaps positions, 2 NS
// steps per sweep; on odd steps the wrap slot NS - 1, holding positions 2 NS - 1 and 0, idles.
//   W warps (8)  slot s is lanes 4 s .. 4 s + 3; lane h holds the rows 4 q + h of the slot's two columns,
//                pairs of q packed for two-element FMAs.  A Gram entry is summed in eight chains (rows mod 8)
//                and a tree, the order in which eight lanes per slot would sum it.  One column per slot moves
//                to the neighbouring slot each step, through a double-buffered area in shared memory (16-byte
//                accesses) and one barrier of the eight warps.
//   V warps (4)  thread t holds row t of V, the columns in registers by position: a step is two rotations'
//                worth of FMAs per pair and no exchange (the swap renames registers).  The steps' (c, s) come
//                through a ring in shared memory; the V warps run up to two double steps behind.
// Bound by the W warps' dependent chain of a step (dot products, parameters, rotation, exchange); the V
// warps fill the schedulers meanwhile.  With W and V in the same lanes, eight lanes a slot, both exchanged
// through shared memory and the parameters computed eight times over, 1000 matrices of 127 x 100 took
// 18.6 ms; it takes 12.2 ms here.
#include <cuda_runtime.h>

#include "common.cuh"
#include "launch.cuh"
#include "rnmath.cuh"

namespace bsvd {

namespace {

constexpr int kRxRows = 128, kRxSlots = 64;
constexpr int kRxQuarter = 36, kRxLd = 4 * kRxQuarter;  // exchange area: strides of a lane's quarter column and of a
                                                        // slot: eight lanes' 16-byte accesses in distinct banks
// threads of the form for up to SLOTS slots: W, V (a row each), both
template <int SLOTS>
struct RxThreads {
    static constexpr int w = 4 * SLOTS, v = (2 * SLOTS + 31) / 32 * 32, all = w + v;
};
constexpr unsigned kRxFull = 0xffffffffu;

struct RxShared {
    float x[2][kRxSlots * kRxLd];       // columns on the move, by step parity and sending slot
    float4 ring[2][2][kRxSlots / 2];    // per double step and step: (c, s) of two pairs
    float sig[kRxRows];                 // singular values by column
    int rank[kRxRows];                  // by position (-1: padding)
    int count[8];                       // rotations of a sweep, per W warp
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
        // (the test itself needs the norms' range, the parameters the rest)
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
template <typename P, int SLOTS>
__global__ void __launch_bounds__(RxThreads<SLOTS>::all, 1)
    jacobi_rx_kernel(int batch, int max_mm, int max_np, float* const* A, const int* M, const int* N, const int* LDA,
                     float* const* Sout, float* const* U, const int* LDU, float* const* V, const int* LDV,
                     double tol_in, int max_sweeps, int* info, long long* rot_out, ItemList wl)
{
    constexpr int kW = RxThreads<SLOTS>::w, kAll = RxThreads<SLOTS>::all;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RxShared& sh = *reinterpret_cast<RxShared*>(smem_raw);
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
                        if (accV && h == 0) ring[(2 * slot) * kRxSlots + s] = make_float2(c, sn);
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
                        if (accV && h == 0) ring[(2 * slot + 1) * kRxSlots + s] = wrap ? make_float2(0.f, 1.f) : make_float2(c, sn);
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

template <typename P, int SLOTS>
static int launch_rx(int batch, int max_mm, int max_np, void* const* A, const int* M, const int* N, const int* LDA,
                     void* const* S, void* const* U, const int* LDU, void* const* V, const int* LDV, double tol,
                     int max_sweeps, int* info, long long* rot, cudaStream_t st, ItemList wl)
{
    auto kern = jacobi_rx_kernel<P, SLOTS>;
    const size_t smem = sizeof(RxShared);
    constexpr int threads = RxThreads<SLOTS>::all;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return BSVD_ERR_CUDA;
    const int grid = item_grid(kern, threads, smem, wl, batch, st);
    if (grid == 0) return BSVD_ERR_CUDA;
    kern<<<grid, threads, smem, st>>>(batch, max_mm, max_np, (float* const*)A, M, N, LDA, (float* const*)S,
                                      (float* const*)U, LDU, (float* const*)V, LDV, tol, max_sweeps, info, rot, wl);
    return cudaGetLastError() == cudaSuccess ? BSVD_SUCCESS : BSVD_ERR_CUDA;
}

// FP32 matrices with max(m, n) <= 128.  Returns BSVD_ERR_UNSUPPORTED for other shapes (the caller then takes
// the shared tier).  Up to 112 columns V leaves registers free and the V warps' work shrinks with the columns:
// 1000 of
// 127 x 100 take 13.1 ms with room for 128 columns (V spilling), 12.2 ms with 112.
int launch_jacobi_rx(int batch, int max_m, int max_n, void* const* A, const int* M, const int* N, const int* LDA,
                     void* const* S, void* const* U, const int* LDU, void* const* V, const int* LDV, double tol,
                     int max_sweeps, int* info, long long* rot, cudaStream_t st, ItemList wl, bool p64)
{
    const int max_mm = max_m > max_n ? max_m : max_n;
    const int max_nn = max_m > max_n ? max_n : max_m;
    const int max_np = (max_nn + 1) & ~1;
    if (max_mm > kRxRows || max_np > kRxRows || max_np < 2) return BSVD_ERR_UNSUPPORTED;
#define BSVD_RX(P_, SLOTS_) \
    launch_rx<P_, SLOTS_>(batch, max_mm, max_np, A, M, N, LDA, S, U, LDU, V, LDV, tol, max_sweeps, info, rot, st, wl)
    if (p64) return BSVD_RX(double, 64);
    return max_np <= 96 ? BSVD_RX(float, 48) : (max_np <= 112 ? BSVD_RX(float, 56) : BSVD_RX(float, 64));
#undef BSVD_RX
}

}  // namespace bsvd
