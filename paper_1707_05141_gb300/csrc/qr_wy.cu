// qr_wy.cu -- batched Householder QR of wider FP32 matrices, one CTA per matrix: 32-column panels in
// registers, compact WY block reflectors on the columns in shared memory (Algorithm 1, Section 2.1;
// the blocked form of Section 3.2 on chip).
//
// qr_kernel (qr.cu) applies one reflector at a time: two shared-memory passes and a warp reduction per
// reflector and column, for the factorisation and again for Q, so it runs at the shared memory's rate
// and not at the FMA units'.  Here
//   panel   warp w holds the panel's columns 2 w and 2 w + 1 (lane: rows lane + 32 t).  The raw pivot
//           column, multiplied with all 32 columns at once, gives its norm, the updates of the columns
//           behind it and the entries of V^T V for T in one reduction; two barriers per column.
//   update  V^T C and C - V Y in register blocks from shared memory (16 and 32 FMAs per four and three
//           16-byte loads), up to 128 columns at a time.
//   Q       the panels' block reflectors on [I; 0], last panel first, in place of V.
// The order of the sums differs from qr_kernel's, so the randomized SVD, whose singular vectors move
// with the last bit of R, keeps that one.
// Their error does not grow: the products are summed in parts of 16 rows and an update's products by themselves before
// they reach the column (Q of 250 x 149 Gaussian matrices against 64 bits: qr_kernel 4.06e-7, here 2.95e-7; 4.61e-7 with
// one chain per thread through the products and through the column, for 2 % less time).
// Measured (GB300, before -> here): 2000 matrices of 250 x 149 7.54 -> 3.69 ms, of 180 x 80 3.08 -> 1.64,
// 20 of 250 x 149 0.54 -> 0.26.  One CTA per SM; by its code, the panels' chain of
// barriers and the shared-memory loads of the updates bound it.
#include <cuda_runtime.h>

#include "common.cuh"
#include "house.cuh"
#include "launch.cuh"

namespace bsvd {

namespace {

constexpr int kPw = 32;                         // panel width
constexpr int kWarps = 16;                      // warps that own two panel columns each
constexpr int kThreads = 32 * (kWarps + 1);     // and one that forms T
constexpr int kWork = 32 * kWarps;
constexpr int kChunk = 128;                     // columns a block reflector is applied to at once
constexpr int kLdW = kChunk + 4;
constexpr int kLdT = kPw + 1;

// leading dimension in shared memory: an odd number of 16-byte vectors, so that a vector from each of
// eight consecutive columns lies in distinct banks
__host__ __device__ inline int wy_ld(int m) { return (((m + 3) / 4) | 1) * 4; }

inline size_t wy_smem(int max_m, int max_n)
{
    const int panels = (max_n + kPw - 1) / kPw;
    return sizeof(float) * ((size_t)wy_ld(max_m) * max_n + (size_t)kPw * kLdW + (size_t)panels * kPw * kLdT);
}

struct Vec4 {
    float v[4];
};
__device__ __forceinline__ Vec4 ld4(const float* p)
{
    const float4 x = *reinterpret_cast<const float4*>(p);
    return Vec4{{x.x, x.y, x.z, x.w}};
}

}  // namespace

template <int RPL>
__global__ void __launch_bounds__(kThreads, 1)
    qr_wy_kernel(int max_m, int max_n, float* const* A, const int* M, const int* N, const int* LDA, float* const* Q,
                 const int* LDQ, float* const* R, const int* LDR, int* info)
{
    extern __shared__ __align__(16) float wy_sm[];
    __shared__ float pub[2][RPL * 32];          // the pivot column, zero above its row
    __shared__ float sum[2][kPw], row[2][kPw];  // its products with the panel's columns; its row of the panel
    __shared__ float Gs[kPw][kLdT], Ts[kPw][kLdT];   // V^T V (above the diagonal) and T (row i, column c)
    __shared__ float diag[kPw], back[kPw];      // R's diagonal; powers of two that a column's entries of R are multiplied by

    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m = M[b], n = N[b], lda = LDA[b];
    const int ldq = Q ? LDQ[b] : m, ldr = R ? LDR[b] : n;
    if (m < 0 || n < 0 || m < n || m > max_m || n > max_n || lda < (m > 1 ? m : 1) ||
        (Q && ldq < (m > 1 ? m : 1)) || (R && ldr < (n > 1 ? n : 1))) {
        if (tid == 0) info[b] = BSVD_INFO_BAD_SHAPE;
        return;
    }
    if (tid == 0) info[b] = 0;
    if (n == 0) return;

    const int ld = wy_ld(max_m), m4 = (m + 3) & ~3;   // (rows m .. m4 - 1 are zero throughout)
    float* S = wy_sm;
    float* Ws = S + (size_t)ld * max_n;               // (i, c) at i kLdW + c
    float* Tm = Ws + kPw * kLdW;                      // panel p's T(i, k) at (p kPw + i) kLdT + k

    // ---- load: eight rows of a column in flight per lane ----
    {
        const float* a = A[b];
        int nonfinite = 0;
        for (int j = warp; j < n; j += kWarps + 1)
            for (int i0 = 0; i0 < m4; i0 += 256) {
                float x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int i = i0 + lane + 32 * u;
                    x[u] = i < m ? a[(size_t)j * lda + i] : 0.f;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int i = i0 + lane + 32 * u;
                    nonfinite |= !isfinite(x[u]);
                    if (i < m4) S[j * ld + i] = x[u];
                }
            }
        if (__syncthreads_or(nonfinite) && tid == 0) info[b] = BSVD_INFO_NONFINITE;
    }

    // C = (I - V op(T) V^T) C on the columns c0 .. n - 1, V panel j0 (32 columns, zero above the diagonal)
    auto apply = [&](int j0, int c0, bool trans) {
        const int rows4 = (m4 - j0) >> 2;
        const float* Tp = Tm + (size_t)(j0 / kPw) * kPw * kLdT;
        for (int cc = c0; cc < n; cc += kChunk) {
            const int nc = n - cc < kChunk ? n - cc : kChunk;
            const int tiles = (nc + 31) >> 5, groups = 8 / tiles;   // row groups of a 32-column tile: 64 threads each
            const int tile = (tid >> 6) / groups, g = (tid >> 6) % groups;
            const bool on = tile < tiles && tid < kWork;
            const int ti = tid & 7, tj = (tid >> 3) & 7;
            float acc[4][4];
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = 0.f;
            if (on) {
                const float *vp[4], *cp[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int c = cc + 32 * tile + tj + 8 * x;   // (a column past the last one: any, not stored)
                    vp[x] = S + (size_t)(j0 + ti + 8 * x) * ld + j0;
                    cp[x] = S + (size_t)(c < n ? c : n - 1) * ld + j0;
                }
                // partial sums of 16 rows, then added: a single chain per thread (up to 128 rows) would err by more
                // than the one-reflector form's 32 lanes and tree
                for (int r0 = g; r0 < rows4; r0 += 4 * groups) {
                    const int r1 = r0 + 4 * groups < rows4 ? r0 + 4 * groups : rows4;
                    float part[4][4];
#pragma unroll
                    for (int x = 0; x < 4; ++x)
#pragma unroll
                        for (int z = 0; z < 4; ++z) part[x][z] = 0.f;
#pragma unroll 2
                    for (int r = r0; r < r1; r += groups) {
                        Vec4 v[4], y[4];
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            v[x] = ld4(vp[x] + 4 * r);
                            y[x] = ld4(cp[x] + 4 * r);
                        }
#pragma unroll
                        for (int k = 0; k < 4; ++k)
#pragma unroll
                            for (int x = 0; x < 4; ++x)
#pragma unroll
                                for (int z = 0; z < 4; ++z) part[x][z] = fmaf(v[x].v[k], y[z].v[k], part[x][z]);
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x)
#pragma unroll
                        for (int z = 0; z < 4; ++z) acc[x][z] += part[x][z];
                }
            }
            for (int k = 0; k < groups; ++k) {   // the row groups, one after the other
                if (on && g == k) {
#pragma unroll
                    for (int x = 0; x < 4; ++x)
#pragma unroll
                        for (int z = 0; z < 4; ++z) {
                            float* w = Ws + (ti + 8 * x) * kLdW + 32 * tile + tj + 8 * z;
                            *w = k == 0 ? acc[x][z] : *w + acc[x][z];
                        }
                }
                __syncthreads();
            }
            // Y = op(T) W: thread (row i, four columns), twice
            float y[2][4];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int i = warp + kWarps * q, c = 4 * lane;
#pragma unroll
                for (int z = 0; z < 4; ++z) y[q][z] = 0.f;
                if (tid < kWork && c < 32 * tiles) {
#pragma unroll 8
                    for (int k = 0; k < kPw; ++k) {
                        const float t = trans ? Tp[k * kLdT + i] : Tp[i * kLdT + k];
                        const Vec4 w = ld4(Ws + k * kLdW + c);
#pragma unroll
                        for (int z = 0; z < 4; ++z) y[q][z] = fmaf(t, w.v[z], y[q][z]);
                    }
                }
            }
            __syncthreads();
            if (tid < kWork) {
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    *reinterpret_cast<float4*>(Ws + (warp + kWarps * q) * kLdW + 4 * lane) =
                        make_float4(y[q][0], y[q][1], y[q][2], y[q][3]);
            }
            __syncthreads();
            // C -= V Y: four rows, eight columns; the product is summed by itself, so that C is rounded once per
            // panel and not once per reflector
            const int units = rows4 * ((nc + 7) >> 3);
            for (int u = tid; u < units; u += kThreads) {
                const int cg = u / rows4, r = j0 + 4 * (u - cg * rows4);
                Vec4 o[8];
#pragma unroll
                for (int z = 0; z < 8; ++z) o[z] = Vec4{};
#pragma unroll 4
                for (int i = 0; i < kPw; ++i) {
                    const Vec4 v = ld4(S + (size_t)(j0 + i) * ld + r);
                    const Vec4 y0 = ld4(Ws + i * kLdW + 8 * cg), y1 = ld4(Ws + i * kLdW + 8 * cg + 4);
#pragma unroll
                    for (int z = 0; z < 4; ++z)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            o[z].v[e] = fmaf(v.v[e], y0.v[z], o[z].v[e]);
                            o[z + 4].v[e] = fmaf(v.v[e], y1.v[z], o[z + 4].v[e]);
                        }
                }
#pragma unroll
                for (int z = 0; z < 8; ++z) {
                    const int c = cc + 8 * cg + z;
                    if (c < n) {
                        float* d = S + (size_t)c * ld + r;
                        const Vec4 x = ld4(d);
                        *reinterpret_cast<float4*>(d) = make_float4(x.v[0] - o[z].v[0], x.v[1] - o[z].v[1],
                                                                    x.v[2] - o[z].v[2], x.v[3] - o[z].v[3]);
                    }
                }
            }
            __syncthreads();
        }
    };

    // ---- factorisation ----
    for (int j0 = 0; j0 < n; j0 += kPw) {
        const int vcols = n - j0 < kPw ? n - j0 : kPw, rows = m - j0;
        float* P = S + (size_t)j0 * ld + j0;
        const bool owner = warp < kWarps, busy = 2 * warp < vcols;   // (vcols <= 2 kWarps)
        float x[2][RPL];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int t = 0; t < RPL; ++t) {
                const int c = 2 * warp + q, r = lane + 32 * t;
                x[q][t] = (owner && c < vcols && r < rows) ? P[(size_t)c * ld + r] : 0.f;
            }
        // the columns are scaled (house.cuh)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float sc = column_scale(warp_magnitude(x[q]), 0.f);
            if (owner && lane == 0) back[2 * warp + q] = 1.f / sc;
#pragma unroll
            for (int t = 0; t < RPL; ++t) x[q][t] *= sc;
        }
        if (warp == 0) {
#pragma unroll
            for (int t = 0; t < RPL; ++t) pub[0][lane + 32 * t] = x[0][t];
        }
        for (int e = tid; e < kPw * kLdT; e += kThreads) (&Ts[0][0])[e] = 0.f;
        // T's column k (lane i: row i): T(k, k) = 2, T(0:k, k) = -2 T(0:k, 0:k) G(0:k, k)
        auto t_column = [&](int k) {
            float s = 0.f;
            for (int e = 0; e < k; ++e) s = fmaf(Ts[lane][e], Gs[e][k], s);
            if (lane <= k) Ts[lane][k] = lane == k ? 2.f : -2.f * s;
        };
        __syncthreads();
        for (int c = 0; c < vcols; ++c) {
            const int buf = c & 1;
            if (busy) {
                float s0 = 0.f, s1 = 0.f;
#pragma unroll
                for (int t = 0; t < RPL; ++t) {
                    const float v = pub[buf][lane + 32 * t];
                    s0 = fmaf(v, x[0][t], s0);
                    s1 = fmaf(v, x[1][t], s1);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    s0 += __shfl_xor_sync(0xffffffffu, s0, o);
                    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                }
                const float e0 = __shfl_sync(0xffffffffu, x[0][0], c), e1 = __shfl_sync(0xffffffffu, x[1][0], c);
                if (lane == 0) {
                    sum[buf][2 * warp] = s0;
                    sum[buf][2 * warp + 1] = s1;
                    row[buf][2 * warp] = e0;
                    row[buf][2 * warp + 1] = e1;
                }
            } else if (!owner && c > 0) {
                t_column(c - 1);
                __syncwarp();
            }
            __syncthreads();
            if (busy) {
                const float tot = sum[buf][c], x0 = row[buf][c];
                const float alpha = dsqrt(tot);
                const float sa = x0 >= 0.f ? alpha : -alpha;   // sign(x0) alpha
                const float inv = alpha > 0.f ? drsqrt(2.f * alpha * (alpha + dabs(x0))) : 0.f;
                const float vc = (x0 + sa) * inv;              // v's entry in row c
                float w[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int j = 2 * warp + q;
                    // v^T x_j = inv (x^T x_j + sign(x0) alpha x_j(c))
                    const float z = inv * fmaf(sa, row[buf][j], sum[buf][j]);
                    w[q] = j > c ? -2.f * z : 0.f;
                    if (j < c && lane == 0) Gs[j][c] = z;
                }
                if (tid == 0) diag[c] = alpha > 0.f ? -sa : 0.f;
                if (2 * warp + 1 >= c) {   // (the columns of the other warps are finished)
#pragma unroll
                    for (int t = 0; t < RPL; ++t) {
                        float v = pub[buf][lane + 32 * t] * inv;
                        if (t == 0 && lane == c) v = vc;
                        x[0][t] = fmaf(w[0], v, x[0][t]);
                        x[1][t] = fmaf(w[1], v, x[1][t]);
                        if (c >> 1 == warp && !(t == 0 && lane < c)) {   // column c becomes v
                            if (c & 1) x[1][t] = v;
                            else x[0][t] = v;
                        }
                    }
                }
                if ((c + 1) >> 1 == warp && c + 1 < vcols) {   // publish the next pivot
#pragma unroll
                    for (int t = 0; t < RPL; ++t) {
                        const float y = (c + 1) & 1 ? x[1][t] : x[0][t];
                        pub[buf ^ 1][lane + 32 * t] = t == 0 && lane <= c ? 0.f : y;
                    }
                }
            }
            __syncthreads();
        }
        float* Tp = Tm + (size_t)(j0 / kPw) * kPw * kLdT;
        if (owner) {
            // V to shared memory, zero above the diagonal; R's entries there straight to R
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int t = 0; t < RPL; ++t) {
                    const int c = 2 * warp + q, r = lane + 32 * t;
                    if (c >= vcols || r >= rows) continue;
                    P[(size_t)c * ld + r] = t == 0 && r < c ? 0.f : x[q][t];
                    if (t == 0 && R && r < vcols)
                        R[b][(size_t)(j0 + c) * ldr + j0 + r] =
                            (r < c ? x[q][t] : (r == c ? diag[c] : 0.f)) * back[c];
                }
            if (R) {
                float* r_out = R[b];
                for (int j = j0 + warp; j < j0 + vcols; j += kWarps)
                    for (int i = lane; i < n; i += 32)
                        if (i < j0 || i >= j0 + vcols) r_out[(size_t)j * ldr + i] = i < j0 ? S[(size_t)j * ld + i] : 0.f;
            }
        } else {
            t_column(vcols - 1);
            __syncwarp();
            for (int k = 0; k < kPw; ++k) Tp[lane * kLdT + k] = Ts[lane][k];   // (past vcols: 0)
        }
        __syncthreads();
        if (j0 + kPw < n) apply(j0, j0 + kPw, true);
    }
    if (!Q) return;

    // ---- Q = H_0 ... H_{n-1} [I; 0] ----
    for (int j0 = (n - 1) / kPw * kPw; j0 >= 0; j0 -= kPw) {
        const int vcols = n - j0 < kPw ? n - j0 : kPw;
        if (j0 + kPw < n) {
            // (R's rows of the columns behind become [I; 0]'s)
            for (int j = j0 + kPw + warp; j < n; j += kWarps + 1) S[(size_t)j * ld + j0 + lane] = 0.f;
            __syncthreads();
            apply(j0, j0 + kPw, false);
        }
        // the panel's own columns: I - V Y, Y = T V_top^T, a row (or half of one) per thread, in place
        const float* Tp = Tm + (size_t)(j0 / kPw) * kPw * kLdT;
        for (int e = tid; e < kPw * kPw; e += kThreads) {
            const int i = e >> 5, c = e & 31;
            float s = 0.f;
            if (c < vcols)
                for (int k = i; k <= c; ++k) s = fmaf(Tp[i * kLdT + k], S[(size_t)(j0 + k) * ld + j0 + c], s);
            Ws[i * kLdW + c] = s;
        }
        const int rows = m - j0, per = rows <= kWork / 2 ? 2 : 1;
        const int r = per == 2 ? tid & (kWork / 2 - 1) : tid, half = per == 2 ? tid / (kWork / 2) : 0;
        const bool on = tid < kWork && r < rows;
        float v[kPw];
#pragma unroll
        for (int i = 0; i < kPw; ++i) v[i] = on && i < vcols ? S[(size_t)(j0 + i) * ld + j0 + r] : 0.f;
        __syncthreads();
        if (on) {
            const int cb = half * (kPw / 2), ce = per == 2 ? cb + kPw / 2 : kPw;
            for (int c = cb; c < ce; c += 4) {
                float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int i = 0; i < kPw; ++i) {
                    const Vec4 y = ld4(Ws + i * kLdW + c);
#pragma unroll
                    for (int z = 0; z < 4; ++z) o[z] = fmaf(-v[i], y.v[z], o[z]);
                }
#pragma unroll
                for (int z = 0; z < 4; ++z)
                    if (c + z < vcols) S[(size_t)(j0 + c + z) * ld + j0 + r] = (r == c + z ? 1.f : 0.f) + o[z];
            }
        }
        __syncthreads();
    }
    float* q_out = Q[b];
    for (int j = warp; j < n; j += kWarps + 1)
        for (int i = lane; i < m; i += 32) q_out[(size_t)j * ldq + i] = S[(size_t)j * ld + i];
}

// Which bounds take this kernel.  It holds an SM alone, so it loses to qr_kernel, several CTAs of which share
// one, where a matrix is small (2000 matrices, before / here: 100 x 70 1.19 / 1.33 ms, 128 x 70 1.22 /
// 1.36, 256 x 64 1.11 / 1.19, 300 x 34 0.78 / 0.97), and wins beyond (160 x 70 2.50 / 1.47, 200 x 66 2.35
// / 1.47, 300 x 66 3.82 / 1.87, 257 x 64 2.18 / 1.46, 500 x 40 1.99 / 1.18).  At the line, 48 to 51 columns, it
// loses where R alone is wanted of thousands (2000 of 300 x 50 0.84 / 0.89 ms; with Q 1.46 / 1.21, 20 of them 0.144
// / 0.064): both calls give the same R, so both take it.  Matrices that are nearly square
// keep qr_kernel's order of sums: the last column of Q of a random square matrix is determined only
// to the size of R(n, n), which over a batch comes close to zero.
int launch_qr_wy(int batch, int max_m, int max_n, void* const* A, const int* M, const int* N, const int* LDA,
                 void* const* Q, const int* LDQ, void* const* R, const int* LDR, int* info, cudaStream_t st)
{
    const size_t smem = wy_smem(max_m, max_n);
    const bool wide = max_n > 64 ? max_m > 128 : (max_n >= 48 && max_m > 256);
    if (!wide || max_m > 512 || 4 * max_m < 5 * max_n || smem > 210 * 1024) return BSVD_ERR_UNSUPPORTED;
    auto kern = max_m <= 256 ? qr_wy_kernel<8> : qr_wy_kernel<16>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return BSVD_ERR_CUDA;
    kern<<<batch, kThreads, smem, st>>>(max_m, max_n, (float* const*)A, M, N, LDA, (float* const*)Q, LDQ,
                                        (float* const*)R, LDR, info);
    return cudaGetLastError() == cudaSuccess ? BSVD_SUCCESS : BSVD_ERR_CUDA;
}

}  // namespace bsvd
