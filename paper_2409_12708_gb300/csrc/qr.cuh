// qr.cuh -- batched blocked Householder QR, one CTA per matrix.
//
// A (m x n, column-major, leading dimension ld, in global memory, m a multiple
// of 4) is factored as A = Q R with Q = H_0 H_1 ... H_{kk-1}, kk = min(m, n),
// H_j = I - tau_j v_j v_j^H, v_j(j) = 1, v_j(i < j) = 0 (Golub & Van Loan,
// Householder QR; for complex A the reflector of LAPACK's convention, with a
// real beta and a complex tau, and H_j^H applied to the trailing columns; the
// blocked form uses the compact WY representation H_0 ... H_{b-1} =
// I - V T V^H of Schreiber & Van Loan).  Real and complex scalars share the
// code (scalar.cuh).
//
// Work split.  Columns are held in registers, four ("a quad") per group of S
// warps: lane l of warp h of the group holds 16-byte chunks of rows
// ((q S + h) 32 + l) VEC, q < NQ, of the four columns (16 NQ 32-bit registers).  The
// panel of nb columns (QR_SHAPES) is factored by all nb / 4 groups at once, each on
// its own quad; the finished reflectors V go to shared memory, and every trailing quad
// then is loaded into registers once, updated (W = V^H Y, W <- T^H W,
// Y -= V W) and stored once.  A group needs only its own warps for that (a
// named barrier), so the groups run free of each other between panels and hide
// one another's load latency; the CTA-wide barriers are one per panel column
// (two when pivoting).  A 16-byte load of V from shared memory feeds four
// columns, so the FMA pipe and the shared-memory pipe are about evenly loaded.
// What bounds it.  float32: about half the panel columns' serial chain (norm, scalars,
// barrier, dots, update), half the updates.  Shares of a warp's time by the clock, one
// 1024 x 256 matrix (beside 303 others within two points the same): panel columns 44 %
// (3160 cycles a column), W 23 %, Y -= V W 15 %, T^H W with its barriers 5 %, T 4 %, loads
// of quads and panels 4 %, stores and outputs 4 %, waiting at the end of a panel 1 %;
// 512 x 256 pivoted: 50 (3400 cycles), 16, 10, 6, 5, 7, 6, 1.  Neither pipe is full: issue
// 0.38 a scheduler (pivoted 0.48), FMA-pipe instructions 21 (24) % of peak, most of them packed
// pairs, warps waiting at barriers first, then for the arithmetic itself.  float64: the
// FP64 pipe (2 FMAs a clock and SM): W 42 %, Y -= V W 33 %, panel columns 15 %.
// Measured (GB300, float32): 304 matrices of 1024 x 256 in 2.04 ms, one alone in
// 0.97 ms (4.55 and 2.14 ms with groups of 16 columns updated straight from global
// memory behind four CTA barriers each); 304 of 512 x 256 pivoted in 1.06 ms, one in
// 0.75 ms (3.43 and 1.69 ms).
//
// Modes (after the factorisation):
//   QR_L_AND_Q : writes L = R^T (n x kk, row-major) and overwrites the first kk
//                columns of A with the thin Q (used to right-canonicalise a site:
//                A holds X^T, so X = L Q^T and Q^T becomes the site tensor; for
//                complex X the plain transpose keeps Q^T's rows orthonormal).
//   QR_R_ROWS  : writes R (n x n, row-major, zero below the diagonal) of A with
//                its columns reordered by block pivoting, and the order; m >= n.
//   QR_L_ONLY  : writes L as QR_L_AND_Q and leaves the reflectors in A and the
//                panel T matrices in Tw (Q is applied later without being formed).
#pragma once

#include <type_traits>

#include "common.cuh"
#include "scalar.cuh"

namespace thc {

enum QRMode : int { QR_L_AND_Q = 1, QR_R_ROWS = 2, QR_L_ONLY = 3 };

template <class T>
struct QRJob {
    T* A;          // term 0 matrix; term b at A + b * strideA; columns 16-byte aligned
    long strideA;
    int m, n, ld;
    T* Tw;         // per-term panel T matrices, [ceil(kk/nb) * nb * nb]
    long strideT;
    T* out;        // L or R output
    long strideOut;
    int mode;
    int* colmap;   // QR_R_ROWS: output, the column order block pivoting chose (n ints, stride n)
};

constexpr int QR_NC = 4;  // columns of a quad

template <class T>
struct QrVec {  // rows per 16-byte chunk
    static constexpr int V = 16 / (int)sizeof(T);
};

// A launch shape: panels of NB columns, S warps per quad, NQ chunks per lane and
// column.  It covers 32 VEC S NQ rows with 32 S NB / 4 threads.
struct QrShape {
    int nb, s, nq;
    int threads() const { return 32 * s * nb / QR_NC; }
    int units() const { return s * nq; }  // rows covered, in 32 VEC
};
// The first that covers the matrix is taken.  One warp per quad needs no barrier
// between the warps of a quad, and two CTAs fit on an SM, so that one's panel (a
// serial chain) overlaps the other's update: 304 pivoted 512 x 256 float32
// matrices take 1.07 ms that way and 1.57 ms with two warps per quad, and one
// matrix alone 0.75 against 0.77 ms.
constexpr QrShape QR_SHAPES[] = {{32, 1, 2}, {32, 1, 4}, {32, 2, 4}, {16, 4, 4}, {8, 8, 4}, {4, 16, 4},
                                 {16, 2, 2}, {16, 2, 4}};
constexpr int QR_NSHAPES = 8;

// Chunks per lane and column that a panel of R rows works on: all or half of
// them, so that the inner loops have no branch per chunk.
__host__ __device__ inline int qr_active(int R, int vec, int s, int nq) {
    return R > 32 * vec * s * (nq / 2) ? nq : nq / 2;
}
// Column stride of V in shared memory: the rows those chunks cover.
template <class T>
__host__ __device__ inline int qr_ldp(int m, int s, int nq) {
    return 32 * QrVec<T>::V * s * qr_active(m, QrVec<T>::V, s, nq);
}

// Shared memory: norm partials and alphas (16 bytes a warp), V, panel dots, the
// groups' W and W partials, T and G = V^H V; then the pivoting state.
template <class T>
__host__ inline size_t qr_smem_bytes(const QrShape& sh, int m, int n, bool pivot) {
    const size_t nb = sh.nb, warps = sh.threads() / 32;
    const size_t elems = nb * qr_ldp<T>(m, sh.s, sh.nq) + 2 * warps * QR_NC + (nb / QR_NC) * (sh.s + 1) * QR_NC * nb + 2 * nb * (nb + 4);
    const size_t piv = pivot ? (nb + n) * sizeof(real_t<T>) + 2 * (size_t)n * sizeof(int) : 0;
    return elems * sizeof(T) + 3 * warps * 16 + ((piv + 15) & ~(size_t)15);
}

// Pivoted matrices of 8- and 16-byte scalars with n >= 128 take panels of 16 columns:
// columns are sorted once per panel, so a narrower one pivots better and saves the
// Jacobi sweeps, which cost most where rows are long.  float64 factors with n >= 128
// of 16 terms at L = 16, D = 128: 3296 sweeps against 3411, 7.12 against 7.52 s, the QR
// itself 787 against 790 ms.  Below, 16 columns cost as much or more: 11344 against
// 11199 sweeps at L = 6, D = 16 float64, 344.6 against 341.6 ms for H|psi> at L = 6,
// D = 32 complex128.
template <class T>
constexpr bool qr_narrow(bool pivot) { return pivot && sizeof(T) >= 8; }

// The shape for m rows (negative: none).
template <class T>
__host__ inline int qr_shape(int m, int n, bool pivot, size_t smem_max) {
    const bool narrow = qr_narrow<T>(pivot) && n >= 128;
    for (int i : {narrow ? 6 : 0, narrow ? 7 : 1, 2, 3, 4, 5}) {
        if (narrow && i == 2) continue;
        if (QR_SHAPES[i].units() * 32 * QrVec<T>::V < m) continue;
        if (qr_smem_bytes<T>(QR_SHAPES[i], m, n, pivot) <= smem_max) return i;
    }
    return -1;
}

// 16-byte chunk load / store
template <class T>
__device__ __forceinline__ void qr_ld(T (&x)[QrVec<T>::V], const T* p) {
    const uint4 u = *reinterpret_cast<const uint4*>(p);
    const T* pu = reinterpret_cast<const T*>(&u);
#pragma unroll
    for (int e = 0; e < QrVec<T>::V; ++e) x[e] = pu[e];
}
template <class T>
__device__ __forceinline__ void qr_st(T* p, const T (&x)[QrVec<T>::V]) {
    uint4 u;
    T* pu = reinterpret_cast<T*>(&u);
#pragma unroll
    for (int e = 0; e < QrVec<T>::V; ++e) pu[e] = x[e];
    *reinterpret_cast<uint4*>(p) = u;
}

// Squared norm with about twice the storage precision.  A Householder
// reflector is orthogonal only if beta^2 = alpha^2 + ||x||^2 holds to working
// precision, and a plain float32 sum over ~10^3 entries misses that by ~1e-6,
// which then compounds through the sweeps.  float: float-float accumulation
// (Knuth's TwoSum with the exact product error from an FMA), no float64
// arithmetic on the hot path; double: a plain sum.
template <class T>
struct SqAcc;
template <>
struct SqAcc<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x * x; }
    __device__ __forceinline__ void merge(const SqAcc& o) { s += o.s; }
};
template <>
struct SqAcc<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float p = x * x, e = fmaf(x, x, -p);
        const float s = hi + p, bp = s - hi;
        lo += ((hi - (s - bp)) + (p - bp)) + e;
        hi = s;
    }
    __device__ __forceinline__ void merge(const SqAcc& o) {
        const float s = hi + o.hi, bp = s - hi;
        lo = (lo + o.lo) + ((hi - (s - bp)) + (o.hi - bp));
        hi = s;
    }
    // butterfly of float-float pairs; every lane ends with the same total
    __device__ __forceinline__ void warp_fold() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            SqAcc b;
            b.hi = __shfl_xor_sync(0xffffffffu, hi, o);
            b.lo = __shfl_xor_sync(0xffffffffu, lo, o);
            merge(b);
        }
    }
};

// complex: both parts of every entry go through the accumulator of the real type
template <class R>
struct SqAcc<cplx<R>> {
    SqAcc<R> a;
    __device__ __forceinline__ void add(cplx<R> x) {
        a.add(x.x);
        a.add(x.y);
    }
    __device__ __forceinline__ void merge(const SqAcc& o) { a.merge(o.a); }
};



// |x|^2 evaluated in float64
template <class T>
__device__ __forceinline__ double dabs2(T x) {
    if constexpr (is_complex_v<T>) return (double)x.x * (double)x.x + (double)x.y * (double)x.y;
    else return (double)x * (double)x;
}

// acc += sum_e conj(v_e) y_e over one chunk, y -= v w over one chunk.  float32
// runs on packed pairs (two IEEE FMAs per instruction).
template <class T>
struct QrAcc {
    T a = tzero<T>();
    __device__ __forceinline__ void add(const T (&v)[QrVec<T>::V], const T (&y)[QrVec<T>::V]) {
#pragma unroll
        for (int e = 0; e < QrVec<T>::V; ++e) a += tconj_mul(v[e], y[e]);
    }
    __device__ __forceinline__ T total() const { return a; }
};
template <>
struct QrAcc<float> {
    float2 a = {0.f, 0.f};
    __device__ __forceinline__ void add(const float (&v)[4], const float (&y)[4]) {
        a = __ffma2_rn(make_float2(v[0], v[1]), make_float2(y[0], y[1]), a);
        a = __ffma2_rn(make_float2(v[2], v[3]), make_float2(y[2], y[3]), a);
    }
    __device__ __forceinline__ float total() const { return a.x + a.y; }
};
template <class T>
__device__ __forceinline__ void qr_axpy(T (&y)[QrVec<T>::V], const T (&v)[QrVec<T>::V], T nw) {  // y += v nw
    if constexpr (std::is_same<T, float>::value) {
        const float2 w2 = make_float2(nw, nw);
        const float2 a = __ffma2_rn(make_float2(v[0], v[1]), w2, make_float2(y[0], y[1]));
        const float2 b = __ffma2_rn(make_float2(v[2], v[3]), w2, make_float2(y[2], y[3]));
        y[0] = a.x;
        y[1] = a.y;
        y[2] = b.x;
        y[3] = b.y;
    } else {
#pragma unroll
        for (int e = 0; e < QrVec<T>::V; ++e) y[e] += v[e] * nw;
    }
}

// Reduce-scatter of NV per-lane values over the warp: the lanes of group i
// (lane / (32 / NV)) return value i's total.
template <int NV, class T>
__device__ __forceinline__ T qr_reduce_scatter(T (&v)[NV]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int lev = 0; (1 << lev) < NV; ++lev) {
        const int o = 16 >> lev, half = (NV >> lev) / 2;
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < NV / 2; ++i) {
            if (i < half) {
                const T send = upper ? v[i] : v[half + i];
                const T keep = upper ? v[half + i] : v[i];
                v[i] = keep + shfl_xor(send, o);
            }
        }
    }
    T t = v[0];
#pragma unroll
    for (int o = 32 / NV / 2; o >= 1; o >>= 1) t += shfl_xor(t, o);
    return t;
}

// A warp's squared norm (float-float or float64), passed through shared memory
// and folded over the warps of a group.
template <class RT>
struct QrNorm;
template <>
struct QrNorm<double> {
    double s = 0.0;
    __device__ __forceinline__ void of(SqAcc<double> a) { s = warp_sum(a.s); }
    __device__ __forceinline__ void store(unsigned char* p) const { *reinterpret_cast<double*>(p) = s; }
    __device__ __forceinline__ void fold(const unsigned char* p) { s += *reinterpret_cast<const double*>(p); }
    __device__ __forceinline__ double value() const { return s; }
    __device__ __forceinline__ double wide() const { return s; }
};
template <>
struct QrNorm<float> {
    SqAcc<float> a;
    __device__ __forceinline__ void of(SqAcc<float> b) {
        b.warp_fold();
        a = b;
    }
    __device__ __forceinline__ void store(unsigned char* p) const {
        *reinterpret_cast<float2*>(p) = make_float2(a.hi, a.lo);
    }
    __device__ __forceinline__ void fold(const unsigned char* p) {
        const float2 t = *reinterpret_cast<const float2*>(p);
        SqAcc<float> b;
        b.hi = t.x;
        b.lo = t.y;
        a.merge(b);
    }
    __device__ __forceinline__ float value() const { return a.hi + a.lo; }
    __device__ __forceinline__ double wide() const { return (double)a.hi + (double)a.lo; }
    __device__ __forceinline__ float plus_square(float x) const {
        SqAcc<float> b = a;
        b.add(x);
        return b.hi + b.lo;
    }
};
template <class T>
__device__ __forceinline__ SqAcc<T> qr_real_acc(const SqAcc<T>& a) { return a; }
template <class R>
__device__ __forceinline__ SqAcc<R> qr_real_acc(const SqAcc<cplx<R>>& a) { return a.a; }

// sqrt(a2), (|x| + sqrt(a2)) / sqrt(a2) and 1 / (|x| + sqrt(a2)) for the reflector, from the
// hardware's float32 reciprocal (square root) and Newton / Halley steps: one
// short dependent chain instead of a square root and two divisions.  Worst relative errors
// measured against exact values over the range that comes here, in units of rounding
// (2^-24, 2^-53): root 1.0, quotient 2.0, reciprocal 2.3.  float64: a2 in float32's range.
__device__ __forceinline__ void qr_scalars(float a2, float ax, float& nrm, float& quo, float& inv) {
    float r = rsqrtf(a2);
    r = fmaf(0.5f * r, fmaf(-(a2 * r), r, 1.f), r);
    nrm = a2 * r;
    nrm = fmaf(0.5f * r, fmaf(-nrm, nrm, a2), nrm);
    const float d = ax + nrm;
    quo = d * r;
    quo = fmaf(r, fmaf(-quo, nrm, d), quo);
    inv = __fdividef(1.f, d);
    inv = fmaf(inv, fmaf(-d, inv, 1.f), inv);
}
__device__ __forceinline__ double qr_recip(double d) {
    const double r = (double)__fdividef(1.f, (float)d);
    const double e = fma(-d, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ double qr_root(double a2, double& r) {  // sqrt(a2) and r = 1 / sqrt(a2)
    r = (double)rsqrtf((float)a2);
    const double e = fma(-(a2 * r), r, 1.0);
    r = fma(r * e, fma(0.375, e, 0.5), r);
    const double n = a2 * r;
    return fma(0.5 * r, fma(-n, n, a2), n);
}
__device__ __forceinline__ void qr_scalars(double a2, double ax, double& nrm, double& quo, double& inv) {
    double r;
    nrm = qr_root(a2, r);
    const double d = ax + nrm;
    quo = d * r;
    quo = fma(r, fma(-quo, nrm, d), quo);
    inv = qr_recip(d);
}
// the exponents of a sum of squares and of its part leave room for the above
__device__ __forceinline__ bool qr_in_range(double part, double a2) {  // 2^-100 < part, a2 < 2^100
    return __double2hiint(part) > 923 << 20 && __double2hiint(a2) < 1123 << 20;
}

// What a warp knows of its place, and the CTA's shared arrays.
template <class T, int NB, int S, int NQ>
struct QrCtx {
    static constexpr int V = QrVec<T>::V;
    static constexpr int NG = NB / QR_NC;        // groups
    static constexpr int WARPS = NG * S;
    static constexpr int LDT = NB + 1;           // leading dimension of T and G
    static constexpr int GSZ = (S + 1) * QR_NC * NB;
    int ldp, grp, h, lane;
    T *P, *Tm, *G;  // V (column i at P + i ldp), T and G
    T *Wp, *W1;     // this group's W partials [h][c][i] and W [i][4]
    T* pd;          // panel dots [parity][warp][4]
    unsigned char *pn, *pa;  // norm partials [parity][warp], alpha [group] (16 bytes each)
    __device__ __forceinline__ int row(int q) const { return ((q * S + h) * 32 + lane) * V; }
    __device__ __forceinline__ void sync() const {  // the group's warps
        if constexpr (S == 1) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(32 * S) : "memory");
    }
};

// Four columns in registers.
template <class T, int NQ>
using QrQuad = T[QR_NC][NQ][QrVec<T>::V];

template <class T, int NB, int S, int NQ>
__device__ __forceinline__ void qr_load(const QrCtx<T, NB, S, NQ>& x, QrQuad<T, NQ>& y, T* const (&col)[QR_NC], int R) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int r = x.row(q);
#pragma unroll
        for (int c = 0; c < QR_NC; ++c) {
            if (r < R && col[c]) {
                qr_ld(y[c][q], col[c] + r);
            } else {
#pragma unroll
                for (int e = 0; e < QrVec<T>::V; ++e) y[c][q][e] = tzero<T>();
            }
        }
    }
}
template <class T, int NB, int S, int NQ>
__device__ __forceinline__ void qr_store(const QrCtx<T, NB, S, NQ>& x, const QrQuad<T, NQ>& y, T* const (&col)[QR_NC], int R) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int r = x.row(q);
        if (r < R) {
#pragma unroll
            for (int c = 0; c < QR_NC; ++c)
                if (col[c]) qr_st(col[c] + r, y[c][q]);
        }
    }
}

// Y <- (I - V T^H V^H) Y (adj: the factorisation) or (I - V T V^H) Y (forming
// Q) on a quad, by one group; NA chunks are worked on.
template <int NA, class T, int NB, int S, int NQ>
__device__ __forceinline__ void qr_apply_quad(const QrCtx<T, NB, S, NQ>& x, QrQuad<T, NQ>& y, int pw, bool adj) {
    constexpr int V = QrVec<T>::V, IB = 2;
    const T* vrow = x.P + x.row(0);
#pragma unroll 1
    for (int i0 = 0; i0 < pw; i0 += IB) {  // W = V^H Y (column pw of V, read when pw is odd, is discarded)
        QrAcc<T> acc[IB * QR_NC];
#pragma unroll
        for (int ii = 0; ii < IB; ++ii) {
            T v[NA][V];
#pragma unroll
            for (int q = 0; q < NA; ++q) qr_ld(v[q], vrow + (i0 + ii) * x.ldp + q * 32 * V * S);
#pragma unroll
            for (int q = 0; q < NA; ++q)
#pragma unroll
                for (int c = 0; c < QR_NC; ++c) acc[ii * QR_NC + c].add(v[q], y[c][q]);
        }
        T w[IB * QR_NC];
#pragma unroll
        for (int k = 0; k < IB * QR_NC; ++k) w[k] = acc[k].total();
        const T t = qr_reduce_scatter<IB * QR_NC>(w);
        constexpr int GL = 32 / (IB * QR_NC);  // lanes per value
        const int k = x.lane / GL;
        if (x.lane % GL == 0) x.Wp[(x.h * QR_NC + k % QR_NC) * NB + i0 + k / QR_NC] = t;
    }
    x.sync();
#pragma unroll 1
    for (int c = x.h; c < QR_NC; c += S) {  // W <- T^H W (T W): lane i forms row i
        const int i = x.lane;
        T w0 = tzero<T>(), w1 = tzero<T>();
        if (i < pw)
#pragma unroll
            for (int hh = 0; hh < S; ++hh) w0 += x.Wp[(hh * QR_NC + c) * NB + i];
        const T* t = adj ? x.Tm + (i < NB ? i : 0) : x.Tm + (i < NB ? i : 0) * x.LDT;
        const int st = adj ? x.LDT : 1;
#pragma unroll 8
        for (int l = 0; l < pw; ++l) {
            const T tl = t[l * st];
            w1 += (adj ? tconj(tl) : tl) * shfl(w0, l);
        }
        if (i < pw) x.W1[i * QR_NC + c] = tzero<T>() - w1;
    }
    x.sync();
#pragma unroll 2
    for (int i = 0; i < pw; ++i) {  // Y -= V W
        T w[QR_NC], v[NA][V];
#pragma unroll
        for (int q = 0; q < NA; ++q) qr_ld(v[q], vrow + i * x.ldp + q * 32 * V * S);
#pragma unroll
        for (int c = 0; c < QR_NC; c += V) {
            T t[V];
            qr_ld(t, x.W1 + i * QR_NC + c);
#pragma unroll
            for (int e = 0; e < V; ++e) w[c + e] = t[e];
        }
#pragma unroll
        for (int q = 0; q < NA; ++q)
#pragma unroll
            for (int c = 0; c < QR_NC; ++c) qr_axpy(y[c][q], v[q], w[c]);
    }
}

// Reflector of a column (y, held by the owner group), step j of the panel: its
// squared norm below row j in about twice the storage precision, beta, tau and
// the scaled v, which goes to V's column j (zeros above row j, 1 on it).  The
// registers keep R's rows above j, beta on row j and v below.
template <int NA, class T, int NB, int S, int NQ>
__device__ __forceinline__ void qr_reflect(const QrCtx<T, NB, S, NQ>& x, T (&y)[NQ][QrVec<T>::V], int j) {
    constexpr int V = QrVec<T>::V;
    using RT = real_t<T>;
    SqAcc<T> a[NA];
#pragma unroll
    for (int e = 0; e < V; ++e)
#pragma unroll
        for (int q = 0; q < NA; ++q) a[q].add(x.row(q) + e > j ? y[q][e] : tzero<T>());
#pragma unroll
    for (int q = 1; q < NA; ++q) a[0].merge(a[q]);
    const int par = j & 1;
    unsigned char* pn = x.pn + (size_t)(par * x.WARPS + x.grp * S) * 16;
    T* alpha_sh = reinterpret_cast<T*>(x.pa + (size_t)x.grp * 16);
    QrNorm<RT> nrm;
    nrm.of(qr_real_acc(a[0]));
    if (S > 1 && x.lane == 0) nrm.store(pn + x.h * 16);
    if (x.h == 0) {  // row j < 32 VEC lies in the first chunk of warp 0
#pragma unroll
        for (int e = 0; e < V; ++e)
            if (x.row(0) + e == j) *alpha_sh = y[0][e];
    }
    x.sync();
    if constexpr (S > 1) {
        nrm = QrNorm<RT>{};
#pragma unroll 1
        for (int hh = 0; hh < S; ++hh) nrm.fold(pn + hh * 16);
    }
    const T alpha = *alpha_sh;
    double xn2 = 0.0;
    bool tiny = false;
    if constexpr (sizeof(RT) == 4) tiny = nrm.value() < 1e-30f;
    if (tiny) {
        // squares of entries below ~1e-19 (residues of rank-deficient columns)
        // underflow in float32: such totals are recomputed from float64 squares
        double s = 0.0;
#pragma unroll 1
        for (int r = x.row(0), q = 0; q < NA; ++q, r += 32 * V * S)
#pragma unroll
            for (int e = 0; e < V; ++e) {
                T t = y[0][e];
#pragma unroll
                for (int k = 1; k < NA; ++k) t = q == k ? y[k][e] : t;
                s += r + e > j ? dabs2(t) : 0.0;
            }
        s = warp_sum(s);
        x.sync();
        if (x.lane == 0) *reinterpret_cast<double*>(pn + x.h * 16) = s;
        x.sync();
#pragma unroll 1
        for (int hh = 0; hh < S; ++hh) xn2 += *reinterpret_cast<const double*>(pn + hh * 16);
    }
    T tau = tzero<T>(), scale = tzero<T>(), beta = alpha;
    bool done = false;
    if constexpr (!is_complex_v<T>) {
        // short chain: float32 on the float-float sum alpha^2 + |x|^2, float64 where
        // the sum is in float32's range
        T a2;
        bool ok;
        if constexpr (sizeof(T) == 4) {
            a2 = nrm.plus_square(alpha);
            ok = !tiny;
        } else {
            a2 = fma(alpha, alpha, nrm.value());
            ok = qr_in_range(nrm.value(), a2);
        }
        if (ok) {
            if (sizeof(T) == 8 || nrm.value() > T(0)) {
                T nr, quo, inv;
                qr_scalars(a2, alpha < T(0) ? -alpha : alpha, nr, quo, inv);
                beta = tcopysign(nr, alpha);
                beta = -beta;
                tau = quo;
                scale = tcopysign(inv, alpha);
            }
            done = true;
        }
    }
    if (!done) {
        if (!tiny) xn2 = nrm.wide();
        const double a2 = dabs2(alpha) + xn2;
        // a sub-column below (1e-30)^2 (float32) is treated as zero
        if (xn2 > 0.0 && a2 > (sizeof(RT) == 4 ? 1e-60 : 0.0)) {
            if constexpr (is_complex_v<T>) {
                // beta = -sign(Re alpha) |(alpha, x)| (real), tau = (beta - alpha) / beta,
                // scale = 1 / (alpha - beta), evaluated in float64
                const double ar = alpha.x, ai = alpha.y;
                if (qr_in_range(xn2, a2)) {
                    double r;
                    const double nr = qr_root(a2, r), ab = fabs(ar), zr = ab + nr;
                    const double quo = zr * r, iz = qr_recip(fma(zr, zr, ai * ai));
                    tau = T{RT(fma(r, fma(-quo, nr, zr), quo)), RT(copysign(1.0, ar) * ai * r)};
                    scale = T{RT(copysign(zr * iz, ar)), RT(-ai * iz)};
                    beta = T{RT(-copysign(nr, ar)), RT(0)};
                } else {
                    const double bt = -copysign(sqrt(a2), ar);
                    tau = T{RT((bt - ar) / bt), RT(-ai / bt)};
                    const double zr = ar - bt, zi = ai, zz = zr * zr + zi * zi;
                    scale = T{RT(zr / zz), RT(-zi / zz)};
                    beta = T{RT(bt), RT(0)};
                }
            } else {
                const double al = alpha;
                const double bt = -copysign(sqrt(a2), al);
                tau = T((bt - al) / bt);
                scale = T(1.0 / (al - bt));
                beta = T(bt);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < NA; ++q) {
        T v[V];
#pragma unroll
        for (int e = 0; e < V; ++e) {
            v[e] = y[q][e] * scale;
            if (q == 0) {  // rows at and above j lie in the first chunk of warp 0
                const int r = x.row(0) + e;
                if (r <= j) v[e] = r == j ? tone<T>() : tzero<T>();
                y[0][e] = r > j ? v[e] : (r == j ? beta : y[0][e]);
            } else {
                y[q][e] = v[e];
            }
        }
        qr_st(x.P + j * x.ldp + x.row(q), v);
    }
    if (x.h == 0 && x.lane == 0) x.Tm[j * x.LDT + j] = tau;
}

// Order of a non-negative metric as an integer: float32's bits, float64's upper 32 (so
// metrics within 1e-6 are alike); NaN and negative values -1, a taken column (-2) -2.
// On integers throughout: a float64 comparison would hold the FP64 pipe for 16 clocks
// a warp in every step of the panel.
constexpr int QR_TAKEN = -2;
__device__ __forceinline__ int qr_metric_key(float v) {
    const int i = __float_as_int(v);
    return i == (int)0xc0000000u ? QR_TAKEN : i < 0 || i > 0x7f800000 ? -1 : i;
}
__device__ __forceinline__ int qr_metric_key(double v) {
    const int i = __double2hiint(v);
    return i == (int)0xc0000000u ? QR_TAKEN : i < 0 || i > 0x7ff00000 ? -1 : i;
}

// T of the compact WY form from tau on its diagonal and G = V^H V: with the
// columns in two halves, T = [T1, -T1 G12 T2; 0, T2], so blocks of 1, 2, 4, ...
// columns are joined pairwise by all threads (T is zero on entry but for its
// diagonal; X = G12 T2 is kept below T's diagonal, which is cleared at the end).
template <class T, int NB, int S, int NQ>
__device__ __forceinline__ void qr_t_matrix(const QrCtx<T, NB, S, NQ>& x, int pw) {
    constexpr int LDT = NB + 1;
    const int tid = (x.grp * S + x.h) * 32 + x.lane, nt = 32 * S * (NB / QR_NC);
#pragma unroll 1
    for (int b = 1; b < pw; b *= 2) {
        // element o: pair o / b^2, row i and column j of its b x b off-diagonal block
        for (int o = tid; o < NB / 2 * b; o += nt) {
            const int pr = o / (b * b), e = o - pr * b * b, i = e / b, j = e - i * b;
            const int r0 = 2 * b * pr, c0 = r0 + b;
            if (c0 + j < pw) {
                T s = tzero<T>();
                for (int l = 0; l <= j; ++l) s += x.G[(r0 + i) * LDT + c0 + l] * x.Tm[(c0 + l) * LDT + c0 + j];
                x.Tm[(c0 + j) * LDT + r0 + i] = s;  // X, transposed into the lower block
            }
        }
        __syncthreads();
        for (int o = tid; o < NB / 2 * b; o += nt) {
            const int pr = o / (b * b), e = o - pr * b * b, i = e / b, j = e - i * b;
            const int r0 = 2 * b * pr, c0 = r0 + b;
            if (c0 + j < pw) {
                T s = tzero<T>();
                for (int l = i; l < b; ++l) s += x.Tm[(r0 + i) * LDT + r0 + l] * x.Tm[(c0 + j) * LDT + r0 + l];
                x.Tm[(r0 + i) * LDT + c0 + j] = tzero<T>() - s;
            }
        }
        __syncthreads();
    }
    for (int o = tid; o < pw * pw; o += nt) {
        const int i = o / pw, j = o - i * pw;
        if (j < i) x.Tm[i * LDT + j] = tzero<T>();
    }
    __syncthreads();
}

// The metric of columns which (bits) of this group's quad, measured: their squared
// norms from row j down.
template <int NA, class T, int NB, int S, int NQ>
__device__ __forceinline__ void qr_remeasure(const QrCtx<T, NB, S, NQ>& x, const QrQuad<T, NQ>& y, int j, unsigned which,
                                             real_t<T>* met) {
    constexpr int V = QrVec<T>::V;
    using RT = real_t<T>;
    if (which == 0) return;  // the group's warps alike
    RT s2[QR_NC];
#pragma unroll
    for (int c = 0; c < QR_NC; ++c) {
        s2[c] = RT(0);
#pragma unroll
        for (int q = 0; q < NA; ++q)
#pragma unroll
            for (int e = 0; e < V; ++e)  // rows above j lie in the first chunk
                if (q > 0 || x.row(0) + e >= j) s2[c] += tabs2(y[c][q][e]);
    }
    RT t = qr_reduce_scatter<QR_NC>(s2);
    const int c = x.lane >> 3;
    if constexpr (S > 1) {
        RT* pd = reinterpret_cast<RT*>(x.pd + x.grp * S * QR_NC);
        if ((x.lane & 7) == 0) pd[x.h * QR_NC + c] = t;
        x.sync();
        t = RT(0);
#pragma unroll 1
        for (int hh = 0; hh < S; ++hh) t += pd[hh * QR_NC + c];
    }
    if (x.h == 0 && (x.lane & 7) == 0 && ((which >> c) & 1u)) met[x.grp * QR_NC + c] = t;
}

// A metric is measured again once less than sqrt(eps) (2^-12, 2^-27) of the value last
// measured is left (the rule of Drmac and Bujanovic for pivoted QR): the differences
// then have lost half of their digits.  As a distance of metric keys.
template <class RT>
constexpr int QR_STALE = sizeof(RT) == 4 ? 12 << 23 : 27 << 20;

// Householder factorisation of the panel: group g holds columns 4 g .. 4 g + 3
// of the pw panel columns in y (R rows).  Per step: the owner forms the
// reflector (qr_reflect), one CTA barrier, then every group takes the dots of
// v with its four columns and updates those not yet done; the dots with
// finished columns are the entries of G = V^H V, which give T at the end.  Pivoting
// (met != null): step j takes the remaining column with the largest metric, its
// squared norm: at the start of the panel a plain sum in the storage type, reduced by
// the squares of the R entries found since, and measured again from the quad's
// registers where that has cancelled (otherwise graded and rank-deficient panels are
// taken in the order of rounding noise, and their factors cost the Jacobi sweeps).
// float64 metrics are compared by their upper 32 bits (1e-6).  stp[c] is the step at
// which this group's column c was taken.
template <int NA, bool PIV, class T, int NB, int S, int NQ>
__device__ __forceinline__ void qr_panel(const QrCtx<T, NB, S, NQ>& x, QrQuad<T, NQ>& y, int pw, bool want_t,
                                         real_t<T>* met, int (&stp)[QR_NC]) {
    constexpr int V = QrVec<T>::V;
#pragma unroll
    for (int c = 0; c < QR_NC; ++c) stp[c] = NB;
    int ref = 0;  // lane's column: its metric's key when last measured
#pragma unroll 1
    for (int j = 0; j < pw; ++j) {
        int k = j;
        if (PIV) {
            int key = x.lane < pw ? qr_metric_key(met[x.lane]) : QR_TAKEN;
            if (j == 0) ref = key;
            const bool stale = key >= 0 && key < ref - QR_STALE<real_t<T>>;
            const unsigned which = __ballot_sync(0xffffffffu, stale);
            if (which) {  // the whole CTA alike: every warp reads the same metrics
                __syncthreads();
                qr_remeasure<NA>(x, y, j, (which >> (x.grp * QR_NC)) & 15u, met);
                __syncthreads();
                if (stale) ref = key = qr_metric_key(met[x.lane]);
            }
            const int best = __reduce_max_sync(0xffffffffu, key);
            k = __ffs(__ballot_sync(0xffffffffu, key == best)) - 1;
        }
        const int kc = x.grp == (k >> 2) ? (k & 3) : -1;  // the column of this quad that is taken
        if (kc >= 0) {
            // one copy of the code for the four columns: the step has to stay within
            // the instruction cache
            T z[NQ][V];
            auto take = [&](auto cc) {  // compile-time column: y stays in registers
                constexpr int c = decltype(cc)::value;
#pragma unroll
                for (int q = 0; q < NA; ++q)
#pragma unroll
                    for (int e = 0; e < V; ++e) z[q][e] = y[c][q][e];
            };
            auto give = [&](auto cc) {
                constexpr int c = decltype(cc)::value;
                stp[c] = j;
#pragma unroll
                for (int q = 0; q < NA; ++q)
#pragma unroll
                    for (int e = 0; e < V; ++e) y[c][q][e] = z[q][e];
            };
            switch (kc) {
                case 0: take(std::integral_constant<int, 0>{}); break;
                case 1: take(std::integral_constant<int, 1>{}); break;
                case 2: take(std::integral_constant<int, 2>{}); break;
                default: take(std::integral_constant<int, 3>{}); break;
            }
            qr_reflect<NA>(x, z, j);
            switch (kc) {
                case 0: give(std::integral_constant<int, 0>{}); break;
                case 1: give(std::integral_constant<int, 1>{}); break;
                case 2: give(std::integral_constant<int, 2>{}); break;
                default: give(std::integral_constant<int, 3>{}); break;
            }
        }
        __syncthreads();
        if (PIV && kc >= 0 && x.h == 0 && x.lane == 0) met[k] = real_t<T>(QR_TAKEN);
        // a group whose columns are all done has only its entries of G left to give
        const bool live = max(max(stp[0], stp[1]), max(stp[2], stp[3])) == NB || want_t;
        if (x.grp * QR_NC < pw && live) {
            const T tau = x.Tm[j * x.LDT + j];
            T v[NA][V];
            QrAcc<T> acc[QR_NC];
#pragma unroll
            for (int q = 0; q < NA; ++q) qr_ld(v[q], x.P + j * x.ldp + x.row(q));
#pragma unroll
            for (int q = 0; q < NA; ++q)
#pragma unroll
                for (int c = 0; c < QR_NC; ++c) acc[c].add(v[q], y[c][q]);
            T w[QR_NC];
#pragma unroll
            for (int c = 0; c < QR_NC; ++c) w[c] = acc[c].total();
            const T t = qr_reduce_scatter<QR_NC>(w);
            if constexpr (S == 1) {
#pragma unroll
                for (int c = 0; c < QR_NC; ++c) w[c] = shfl(t, 8 * c);
            } else {
                T* pd = x.pd + ((j & 1) * x.WARPS + x.grp * S) * QR_NC;
                if ((x.lane & 7) == 0) pd[x.h * QR_NC + (x.lane >> 3)] = t;
                x.sync();
#pragma unroll
                for (int c = 0; c < QR_NC; ++c) w[c] = pd[c];
#pragma unroll
                for (int hh = 1; hh < S; ++hh)
#pragma unroll
                    for (int c = 0; c < QR_NC; ++c) w[c] += pd[hh * QR_NC + c];
            }
            // y -= conj(tau) (v^H y) v on the columns not yet taken (factor 0 on the others)
            const T ntau = tzero<T>() - tconj(tau);
#pragma unroll
            for (int c = 0; c < QR_NC; ++c) {
                const T f = stp[c] == NB ? ntau * w[c] : tzero<T>();
                if (sizeof(real_t<T>) == 8 && stp[c] != NB) continue;  // float64 work is scarce
#pragma unroll
                for (int q = 0; q < NA; ++q) qr_axpy(y[c][q], v[q], f);
            }
            if (x.h == 0) {
                if (want_t) {  // dots with the finished columns: row stp[c] of G
                    T g = w[0];
                    int row = stp[0];
#pragma unroll
                    for (int c = 1; c < QR_NC; ++c) {
                        g = x.lane == c ? w[c] : g;
                        row = x.lane == c ? stp[c] : row;
                    }
                    if (x.lane < QR_NC && row < j) x.G[row * x.LDT + j] = tconj(g);
                }
                if (PIV) {
#pragma unroll
                    for (int e = 0; e < V; ++e)
                        if (x.row(0) + e == j) {
#pragma unroll
                            for (int c = 0; c < QR_NC; ++c) {
                                const int lc = x.grp * QR_NC + c;
                                const real_t<T> d = met[lc] - tabs2(y[c][0][e]);
                                if (stp[c] == NB) met[lc] = d > real_t<T>(0) || d != d ? d : real_t<T>(0);
                            }
                        }
                }
            }
        }
        if (PIV) __syncthreads();
    }
    __syncthreads();
    if (want_t) qr_t_matrix(x, pw);
}

template <class T, int NB, int S, int NQ, bool PIV>
__global__ void __launch_bounds__(32 * S * NB / QR_NC, S == 1 ? 2 : 1) k_qr(QRJob<T> job) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int V = QrVec<T>::V;
    using RT = real_t<T>;
    const int b = blockIdx.x;
    const int m = job.m, n = job.n, ld = job.ld;
    constexpr int nb = NB, nt = 32 * S * NB / QR_NC;
    const int kk = min(m, n);
    T* A = job.A + (long)b * job.strideA;
    T* Tw = job.Tw + (long)b * job.strideT;
    const int tid = threadIdx.x;
    const int lane = tid & 31, wid = tid >> 5;
    QrCtx<T, NB, S, NQ> x;
    x.ldp = qr_ldp<T>(m, S, NQ);
    x.grp = wid / S;
    // the warps of a quad by rank h; where chunks past the matrix are left out (below), the
    // last rank's empty first, and a warp's place in the CTA fixes its scheduler: ranks are
    // turned from quad to quad
    x.h = (wid + (sizeof(RT) < 8 ? 0 : S >= 4 ? x.grp : x.grp / 2)) % S;
    // Y's update.  The FP64 pipe bounds 64-bit types, so each warp takes only the chunks
    // that hold rows (at 1024 x 256, 12 to 16 of the quad's 16): 120 LQ launches of 16 terms
    // at L = 16, D = 128 float64 2717 -> 2597 ms, the pivoted QRs 788 -> 739 ms.  (A branch
    // per chunk in the loops gained nothing: 2755 ms.)  32-bit types keep two versions.
    auto update = [&](QrQuad<T, NQ>& yy, int pw, int R, bool adj) {
        if constexpr (sizeof(RT) == 8 && NQ == 4) {
            const int act = (ceil_div(R, 32 * V) - x.h + S - 1) / S;
            if (act >= 4) qr_apply_quad<4>(x, yy, pw, adj);
            else if (act == 3) qr_apply_quad<3>(x, yy, pw, adj);
            else if (act == 2) qr_apply_quad<2>(x, yy, pw, adj);
            else qr_apply_quad<1>(x, yy, pw, adj);
        } else if (qr_active(R, V, S, NQ) == NQ) {
            qr_apply_quad<NQ>(x, yy, pw, adj);
        } else {
            qr_apply_quad<NQ / 2>(x, yy, pw, adj);
        }
    };
    x.lane = lane;
    x.pn = smem_raw;
    x.pa = smem_raw + 2 * x.WARPS * 16;
    x.P = reinterpret_cast<T*>(x.pa + x.WARPS * 16);
    x.pd = x.P + (size_t)nb * x.ldp;
    T* grp0 = x.pd + 2 * x.WARPS * QR_NC;
    x.W1 = grp0 + x.grp * x.GSZ;
    x.Wp = x.W1 + QR_NC * nb;
    x.Tm = grp0 + x.NG * x.GSZ;
    x.G = x.Tm + nb * (nb + 4);
    RT* met = reinterpret_cast<RT*>(x.G + nb * (nb + 4));
    RT* cnrm = met + nb;
    int* pm = reinterpret_cast<int*>(cnrm + n);
    int* pm2 = pm + n;
    auto phys = [&](int c) { return PIV ? pm[c] : c; };

    if (PIV) {  // identity order and the columns' squared norms
        for (int c = tid; c < n; c += nt) pm[c] = c;
        for (int c = wid; c < n; c += x.WARPS) {
            const T* col = A + (long)c * ld;
            RT s2 = RT(0);
            for (int r = lane; r < m; r += 32) s2 += tabs2(col[r]);
            s2 = warp_sum(s2);
            if (lane == 0) cnrm[c] = s2;
        }
        __syncthreads();
    }

    QrQuad<T, NQ> y;
    T* col[QR_NC];
#pragma unroll 1
    for (int p0 = 0; p0 < kk; p0 += nb) {
        const int pw = min(nb, kk - p0);
        const int R = m - p0;
        if (PIV) {
            // block pivoting: order the remaining columns by their norm below row
            // p0 (ties by position; non-finite norms last), so the panel takes the
            // largest ones
            for (int c = p0 + tid; c < n; c += nt) {
                RT v = cnrm[c];
                if (!(v == v)) v = RT(-1);
                int rank = 0;
                for (int q = p0; q < n; ++q) {
                    RT w = cnrm[q];
                    if (!(w == w)) w = RT(-1);
                    rank += (w > v) || (w == v && q < c);
                }
                pm2[p0 + rank] = pm[c];
                if (rank < pw) met[rank] = v;
            }
            __syncthreads();
            for (int c = p0 + tid; c < n; c += nt) pm[c] = pm2[c];
            __syncthreads();
        }
        int lc[QR_NC], stp[QR_NC];
#pragma unroll
        for (int c = 0; c < QR_NC; ++c) {
            const int l = x.grp * QR_NC + c;
            lc[c] = l < pw ? phys(p0 + l) : -1;
            col[c] = l < pw ? A + (long)lc[c] * ld + p0 : nullptr;
        }
        qr_load<T, NB, S, NQ>(x, y, col, R);
        for (int o = tid; o < nb * x.LDT; o += nt) x.Tm[o] = tzero<T>();
        __syncthreads();
        const bool want_t = !PIV || p0 + pw < n;
        const bool full = qr_active(R, V, S, NQ) == NQ;
        if (full) qr_panel<NQ, PIV>(x, y, pw, want_t, met, stp);
        else qr_panel<NQ / 2, PIV>(x, y, pw, want_t, met, stp);
        // the factored panel (R above, reflectors below the diagonal) back to A
        qr_store<T, NB, S, NQ>(x, y, col, R);
        if (PIV && x.h == 0 && lane == 0) {
#pragma unroll
            for (int c = 0; c < QR_NC; ++c)
                if (lc[c] >= 0) pm[p0 + stp[c]] = lc[c];
        }
        // T for forming or applying Q
        if (!PIV)
            for (int o = tid; o < nb * nb; o += nt) Tw[(long)(p0 / nb) * nb * nb + o] = x.Tm[(o / nb) * x.LDT + o % nb];
        // --- trailing update of columns p0+pw .. n-1, a quad per group
#pragma unroll 1
        for (int c0 = p0 + pw + QR_NC * x.grp; c0 < n; c0 += QR_NC * x.NG) {
#pragma unroll
            for (int c = 0; c < QR_NC; ++c) col[c] = c0 + c < n ? A + (long)phys(c0 + c) * ld + p0 : nullptr;
            qr_load<T, NB, S, NQ>(x, y, col, R);
            update(y, pw, R, true);
            qr_store<T, NB, S, NQ>(x, y, col, R);
            if (PIV) {  // their norms below row p0 + pw, for the next panel
                RT s2[QR_NC];
#pragma unroll
                for (int c = 0; c < QR_NC; ++c) {
                    s2[c] = RT(0);
#pragma unroll
                    for (int q = 0; q < NQ; ++q)
#pragma unroll
                        for (int e = 0; e < V; ++e)
                            if (x.row(q) + e >= pw) s2[c] += tabs2(y[c][q][e]);
                }
                const RT t = qr_reduce_scatter<QR_NC>(s2);
                RT* pd = reinterpret_cast<RT*>(x.pd + x.grp * S * QR_NC);
                if ((lane & 7) == 0) pd[x.h * QR_NC + (lane >> 3)] = t;
                x.sync();
                if (x.h == 0 && lane < QR_NC && c0 + lane < n) {
                    RT s = RT(0);
#pragma unroll 1
                    for (int hh = 0; hh < S; ++hh) s += pd[hh * QR_NC + lane];
                    cnrm[c0 + lane] = s;
                }
            }
        }
        __syncthreads();
    }

    // --- outputs
    T* out = job.out + (long)b * job.strideOut;
    if constexpr (PIV) {
        for (int i = tid; i < n * n; i += nt) {
            const int r = i / n, c = i % n;
            out[i] = (r <= c && r < kk) ? A[(long)phys(c) * ld + r] : tzero<T>();
        }
        for (int c = tid; c < n; c += nt) job.colmap[(long)b * n + c] = pm[c];
    } else {
        // QR_L_AND_Q / QR_L_ONLY: L = R^T (n x kk)
#pragma unroll 4
        for (int i = tid; i < n * kk; i += nt) {
            const int r = i / kk, c = i % kk;
            out[i] = (c <= r) ? A[(long)r * ld + c] : tzero<T>();
        }
        if (job.mode == QR_L_ONLY) return;
        __syncthreads();
        // form Q in place, panels in reverse order: the panel's block reflector on the
        // later columns of Q and on the identity columns of its own
#pragma unroll 1
        for (int pi = (kk - 1) / nb; pi >= 0; --pi) {
            const int p0 = pi * nb;
            const int pw = min(nb, kk - p0);
            const int R = m - p0;
            for (int o = tid; o < pw * x.ldp; o += nt) {
                const int i = o / x.ldp, r = o % x.ldp;
                x.P[o] = r < i || r >= R ? tzero<T>() : (r == i ? tone<T>() : A[(long)(p0 + i) * ld + p0 + r]);
            }
            for (int o = tid; o < nb * nb; o += nt) x.Tm[(o / nb) * x.LDT + o % nb] = Tw[(long)pi * nb * nb + o];
            __syncthreads();
#pragma unroll 1
            for (int c0 = p0 + QR_NC * x.grp; c0 < kk; c0 += QR_NC * x.NG) {
                const bool own = c0 < p0 + pw;
#pragma unroll
                for (int c = 0; c < QR_NC; ++c) col[c] = c0 + c < kk ? A + (long)(c0 + c) * ld + p0 : nullptr;
                if (own) {
#pragma unroll
                    for (int c = 0; c < QR_NC; ++c)
#pragma unroll
                        for (int q = 0; q < NQ; ++q)
#pragma unroll
                            for (int e = 0; e < V; ++e)
                                y[c][q][e] = x.row(q) + e == c0 + c - p0 ? tone<T>() : tzero<T>();
                } else {
                    qr_load<T, NB, S, NQ>(x, y, col, R);
                }
                update(y, pw, R, false);
                qr_store<T, NB, S, NQ>(x, y, col, R);
            }
            for (int i = tid; i < pw * p0; i += nt) A[(long)(p0 + i / p0) * ld + i % p0] = tzero<T>();
            __syncthreads();
        }
    }
}

// f(kernel) for shape i of QR_SHAPES
template <class T, bool PIV, class F>
inline void qr_dispatch(int shape, F&& f) {
    if constexpr (qr_narrow<T>(PIV)) {
        if (shape == 6) return f(k_qr<T, 16, 2, 2, PIV>);
        if (shape == 7) return f(k_qr<T, 16, 2, 4, PIV>);
    }
    switch (shape) {
        case 0: return f(k_qr<T, 32, 1, 2, PIV>);
        case 1: return f(k_qr<T, 32, 1, 4, PIV>);
        case 2: return f(k_qr<T, 32, 2, 4, PIV>);
        case 3: return f(k_qr<T, 16, 4, 4, PIV>);
        case 4: return f(k_qr<T, 8, 8, 4, PIV>);
        case 5: return f(k_qr<T, 4, 16, 4, PIV>);
    }
}

}  // namespace thc
