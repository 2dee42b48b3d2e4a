// qt_apply.cuh -- the SVD sweep's C_s = M_{s-1} Q_s without forming Q_s.
//
// The QR sweep leaves site s factored in place: X_s^T = Q R with the
// reflectors V below the diagonal of the m x kk column-major matrix A (unit
// diagonal implicit; R on and above it) and the compact-WY panel matrices T_p
// (Schreiber & Van Loan) in Tw.  The site tensor is the row-orthonormal
// Q^T = [I_kk 0] H_{kk-1} ... H_0 (real reflectors, H_j = H_j^T), so with
// P_p = H_{p0} ... H_{p0+pw-1} = I - V_p T_p V_p^T,
//     C = M Q^T = [M 0] P_{np-1}^T ... P_0^T,   P_p^T = I - V_p T_p^T V_p^T,
// applied from the last panel:  X <- X - (X V_p) T_p^T V_p^T,  X = [M 0].
// For out rows of M this is 4 out m kk flops, against 4 m kk^2 - 4 kk^3 / 3
// for forming Q plus 2 out m kk for the product M Q^T.
//
// One CTA of 512 threads per 32 rows of X (held in shared memory with a row
// pitch of m + 4 floats) and term:
//   * Z = X V_p: warp w takes a contiguous range of quads of the K = m - p0
//     rows of V_p; lane (rq, cq) accumulates the 8 x 4 tile rows rq + 4 i,
//     columns 4 cq.. with 16-byte loads of X (shared) and of V's columns
//     (global, loaded 8 quads ahead, a warp
//     at a time in full lines, and staged in the space of its partial sums; the
//     zero/one substitution of V's triangle only on the panel's first 32 rows);
//     the 16 warp partials are summed in shared memory;
//   * Z <- Z T_p^T (T upper triangular, held at a pitch of 33: a warp reads one
//     entry of every row of T at a time);
//   * X[:, p0:] -= Z V_p^T: two adjacent columns of X per thread, V's rows
//     k, k+1 read with one 8-byte load per panel column, coalesced across the
//     warp; multiply-adds on the packed pair.  With fewer than 512 (256) columns
//     left, two (four) groups of threads share the rows.
// Bound by shared-memory reads and issue beside the FMA pipe (one CTA of 16 warps
// per SM).  Measured: 608 x (m = 1024, kk = 256, out = 128) 4.05 -> 3.05 ms when V was
// staged (a lane reading V's columns directly used half of each 32-byte sector);
// all launches of 608 terms at L = 16, D = 128: 133 -> 121 ms by T's pitch (32 was a
// 16-way bank conflict), loads ahead, W written along its columns and row groups in
// narrow updates, -> 93 ms by the staging.
// Real float32 only, panels of 32 columns, m <= 1024 (the LQ-sweep shapes of
// the float paths up to D_max = 256); other shapes form Q in the QR kernel.
#pragma once

#include "common.cuh"

namespace thc {

constexpr int QT_THREADS = 512;
constexpr int QT_RB = 32;  // rows of X per CTA
constexpr int QT_NB = 32;  // panel width
constexpr int QT_LDT = QT_NB + 1;  // pitch of T in shared memory

template <class T>
struct QtJob {
    const T* M;   // out x kk rows, row-major, leading dimension ldM
    long strideM;
    int ldM;
    const T* A;   // m x kk reflectors, column-major, leading dimension ld
    long strideA;
    int ld;
    const T* Tw;  // panel p's T at Tw + p * QT_NB * QT_NB (row-major)
    long strideT;
    int out, m, kk;
    T* C;         // out x m result, row-major, leading dimension ldC
    long strideC;
    int ldC;
    T* W;         // optional column-major copy of C viewed as (4 out) x nW
    long strideW;
    int nW;
};

__host__ __device__ inline int qt_ldx(int m) { return m + 4; }

__host__ inline size_t qt_smem_bytes(int m) {
    return sizeof(float) * ((size_t)QT_RB * qt_ldx(m) + (size_t)(QT_THREADS / 32) * QT_RB * QT_NB +
                            2 * QT_RB * QT_NB + QT_NB * QT_LDT);
}

// V_p's element (row k of A, panel column j): zero above the diagonal, one on it
__device__ __forceinline__ float qt_v(int p0, int j, int k, float loaded) {
    const int kr = k - p0;
    return kr < j ? 0.f : (kr == j ? 1.f : loaded);
}

static __global__ void __launch_bounds__(QT_THREADS, 1) k_apply_qt(QtJob<float> job) {
    extern __shared__ __align__(16) unsigned char qt_raw[];
    const int b = blockIdx.y, r0 = blockIdx.x * QT_RB;
    const int m = job.m, kk = job.kk, ldx = qt_ldx(m);
    const int rows = min(QT_RB, job.out - r0);
    float* X = reinterpret_cast<float*>(qt_raw);                 // QT_RB x ldx
    float* Zp = X + (size_t)QT_RB * ldx;                          // 16 warps x (QT_RB x QT_NB)
    float* Z = Zp + (size_t)(QT_THREADS / 32) * QT_RB * QT_NB;    // QT_RB x QT_NB
    float* Z2 = Z + QT_RB * QT_NB;                                // Z T^T
    float* Tm = Z2 + QT_RB * QT_NB;                               // QT_NB x QT_LDT
    const float* M = job.M + (long)b * job.strideM;
    const float* A = job.A + (long)b * job.strideA;
    const float* Tw = job.Tw + (long)b * job.strideT;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = QT_THREADS / 32;
    for (int r = 0; r < QT_RB; ++r)
        for (int c = tid; c < m; c += QT_THREADS)
            X[(size_t)r * ldx + c] = (r < rows && c < kk) ? M[(long)(r0 + r) * job.ldM + c] : 0.f;
    // tile of lane (rq, cq): rows rq + 4 i (i < 8), columns 4 cq .. 4 cq + 3; the
    // four rows a quarter-warp reads together are consecutive, and the pitch
    // m + 4 puts them in distinct bank quads
    const int rq = lane >> 3, cq = lane & 7;
    const int np = ceil_div(kk, QT_NB);
    for (int p = np - 1; p >= 0; --p) {
        const int p0 = p * QT_NB, pw = min(QT_NB, kk - p0);
        for (int i = tid; i < QT_NB * QT_NB; i += QT_THREADS)
            Tm[i / QT_NB * QT_LDT + i % QT_NB] = Tw[(long)p * QT_NB * QT_NB + i];
        __syncthreads();
        // ---- Z = X[:, p0:m] V_p, K split over the warps in quads of rows
        {
            const int R4 = (m - p0) >> 2;  // m and p0 are multiples of 4
            const int qpw = ceil_div(R4, nw);
            const int q0 = wid * qpw, q1 = min(R4, q0 + qpw);
            float acc[8][4];
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
            // V's next 8 quads of rows: a warp's load covers 32 rows of 4 columns; staged
            // in the warp's own part of Zp with the row quad XORed by column / 4
            float4* Vs = reinterpret_cast<float4*>(Zp + (size_t)wid * QT_RB * QT_NB);
            const int lc = lane >> 3, lq = lane & 7;
            float4 nv[8];
            auto fetch = [&](int qc) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    nv[i] = 4 * i + lc < pw && qc + lq < q1
                                ? *reinterpret_cast<const float4*>(A + (long)(p0 + 4 * i + lc) * job.ld + p0 + 4 * (qc + lq))
                                : make_float4(0.f, 0.f, 0.f, 0.f);
            };
            fetch(q0);
            for (int qc = q0; qc < q1; qc += 8) {
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    float4 v = nv[i];
                    const int col = 4 * i + lc, k = p0 + 4 * (qc + lq);
                    if (k < p0 + QT_NB)  // the panel's triangle: zeros above the diagonal, ones on it
                        v = make_float4(qt_v(p0, col, k, v.x), qt_v(p0, col, k + 1, v.y), qt_v(p0, col, k + 2, v.z),
                                        qt_v(p0, col, k + 3, v.w));
                    Vs[col * 8 + (lq ^ i)] = v;
                }
                __syncwarp();
                fetch(qc + 8);
                const int nq = min(8, q1 - qc);
                for (int t = 0; t < nq; ++t) {
                    const int k = p0 + 4 * (qc + t);
                    float4 v[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[j] = Vs[(4 * cq + j) * 8 + (t ^ cq)];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float4 x = *reinterpret_cast<const float4*>(X + (size_t)(rq + 4 * i) * ldx + k);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            float a = acc[i][j];
                            a = fmaf(x.x, v[j].x, a);
                            a = fmaf(x.y, v[j].y, a);
                            a = fmaf(x.z, v[j].z, a);
                            acc[i][j] = fmaf(x.w, v[j].w, a);
                        }
                    }
                }
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<float4*>(Zp + (size_t)wid * QT_RB * QT_NB + (rq + 4 * i) * QT_NB + 4 * cq) =
                    make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        }
        __syncthreads();
        for (int o = tid; o < QT_RB * QT_NB; o += QT_THREADS) {
            float s = 0.f;
            for (int w = 0; w < nw; ++w) s += Zp[(size_t)w * QT_RB * QT_NB + o];
            Z[o] = s;
        }
        __syncthreads();
        // ---- Z2 = Z T^T: Z2(r, j) = sum_{i >= j} Z(r, i) T(j, i)
        for (int o = tid; o < QT_RB * QT_NB; o += QT_THREADS) {
            const int r = o / QT_NB, j = o - r * QT_NB;
            float s = 0.f;
            if (j < pw)
                for (int i = j; i < pw; ++i) s += Z[r * QT_NB + i] * Tm[j * QT_LDT + i];
            Z2[o] = s;
        }
        __syncthreads();
        // ---- X[:, p0:m] -= Z2 V_p^T, two adjacent columns per thread (p0 and m
        // are even): V's rows k, k+1 come with one 8-byte load per panel column
        const int split = m - p0 > QT_THREADS ? 1 : m - p0 > QT_THREADS / 2 ? 2 : 4;  // groups sharing the rows
        const int per = QT_THREADS / split, rg = tid / per;
        for (int k = p0 + 2 * (tid - rg * per); k < m; k += 2 * per) {
            float2 v[QT_NB];
#pragma unroll
            for (int j = 0; j < QT_NB; ++j)
                v[j] = j < pw ? *reinterpret_cast<const float2*>(A + (long)(p0 + j) * job.ld + k)
                              : make_float2(0.f, 0.f);
            if (k < p0 + QT_NB) {  // the panel's triangle
#pragma unroll
                for (int j = 0; j < QT_NB; ++j) {
                    v[j].x = qt_v(p0, j, k, v[j].x);
                    v[j].y = qt_v(p0, j, k + 1, v[j].y);
                }
            }
#pragma unroll 2
            for (int r = rg * (QT_RB / split); r < (rg + 1) * (QT_RB / split); ++r) {
                const float4* zr = reinterpret_cast<const float4*>(Z2 + r * QT_NB);
                float2 sum = make_float2(0.f, 0.f);
#pragma unroll
                for (int j4 = 0; j4 < QT_NB / 4; ++j4) {
                    const float4 z = zr[j4];
                    sum = __ffma2_rn(make_float2(z.x, z.x), v[4 * j4], sum);
                    sum = __ffma2_rn(make_float2(z.y, z.y), v[4 * j4 + 1], sum);
                    sum = __ffma2_rn(make_float2(z.z, z.z), v[4 * j4 + 2], sum);
                    sum = __ffma2_rn(make_float2(z.w, z.w), v[4 * j4 + 3], sum);
                }
                float2* xr = reinterpret_cast<float2*>(X + (size_t)r * ldx + k);
                float2 x = *xr;
                x.x -= sum.x;
                x.y -= sum.y;
                *xr = x;
            }
        }
        __syncthreads();
    }
    // ---- C (and its column-major copy for the preconditioning QR)
    float* C = job.C + (long)b * job.strideC;
    for (int r = 0; r < rows; ++r)
        for (int c = tid; c < m; c += QT_THREADS) C[(long)(r0 + r) * job.ldC + c] = X[(size_t)r * ldx + c];
    if (job.W) {
        // W viewed as (4 out) x nW column-major; m = 4 nW
        float* W = job.W + (long)b * job.strideW;
        const int mW = 4 * job.out;
        // (r, qb) fastest: a column of W gets 4 rows contiguous floats
        for (int i = tid; i < QT_RB * 4 * job.nW; i += QT_THREADS) {
            const int rb = i % (QT_RB * 4), j = i / (QT_RB * 4);
            if (rb < 4 * rows)
                W[(long)j * mW + r0 * 4 + rb] = X[(size_t)(rb >> 2) * ldx + (rb & 3) * job.nW + j];
        }
    }
}

}  // namespace thc
