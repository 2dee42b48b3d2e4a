// adjoint.cuh -- exact <phi|H|psi> and its derivatives with respect to t, chi,
// zeta and psi (the adjoint of the THC-MPO expectation value).
//
// Every term of H is a product of nl bond-2 ladder MPOs (Sec. 3.1): a Coulomb
// term G_{mu s, nu s'} = zeta^{mu nu} A+_{mu s} A_{mu s} A+_{nu s'} A_{nu s'}
// (Eq. G; four layers, A_{nu s'} applied first), a one-body term
// (sum_p t_pq a+_{p s}) a_{q s} (two layers, the first with coefficient e_q).
// A term's value <phi|W_{nl-1} ... W_0|psi> is contracted exactly (no
// compression) with environments over the composite MPO bond w in [0, 2^nl)
// (bit l = bond state of layer l):
//   left   E_{s+1}[a', w', b'] = sum phi_s[a, n', a'] M_s[w, w', n', n] E_s[a, w, b] psi_s[b, n, b']
//   right  R_s[a, w, b]       = sum phi_s[a, n', a'] M_s[w, w', n', n] R_{s+1}[a', w', b'] psi_s[b, n, b']
// with M_s the product of the layers' site-s tensors
// W = [[Z(x)Z, c_s b], [0, I4]] and boundary states w = 0 (left), w = all ones
// (right).  The derivatives follow from the two environments:
//   d value / d c^l_s = sum X_s[a, w, n, b'] (M'^l_s^T Q_s)[a, w, n, b'],
//       X_s = E_s psi_s, Q_s = phi_s R_{s+1}, M'^l_s = M_s with layer l's site-s
//       tensor replaced by dW/dc_s = [[0, b], [0, 0]];
//   d value / d psi_s = E_s^T (M_s^T Q_s).
// Each site is four batched GEMMs (the library's tiled GEMM) and two
// kernels that apply the layers in registers (forward, or transposed with the
// coefficient gradients; the transposed one of four float64 layers holds three blocks of
// 64 entries and spills 316 bytes of them).  Real MPS only.
#pragma once

#include "common.cuh"
#include "scalar.cuh"

namespace thc {

// per-term layer data: nl layers, op[b*nl + l] = sigma + 2*dagger, coef[(b*nl + l)*L + s]
template <class T>
struct AdjTerms {
    const int* op;
    const T* coef;
    int nl, L;
};

// The ladder operators' local matrices (c_src, c_sgn) for an operator known at
// compile time: two elements, n' = dst <- n = dst ^ flip.  A kernel branches once per
// layer (the whole CTA alike) to the code of its operator, so that all register
// indices are constants and only the two elements are multiplied: an entry that the
// operator does not reach is left alone, also by an infinity (a coefficient of zero
// would make it NaN).  Layer kernels of all terms at L = 8, N = 8, D = 64 against four
// products of which two have a zero coefficient: float64 4.51 -> 3.13 ms, float32
// (bound elsewhere) within 2 %.  Indices from a table would put the blocks into local
// memory: 35.6 against 5.9 ms for 1024 terms at L = 10, D = 64, float32.
__device__ __forceinline__ constexpr int adj_par(int n) { return n == 0 || n == 3 ? 1 : -1; }  // c_par
template <int O>  // O = sigma + 2 dagger
struct AdjMat {
    static constexpr int flip = O & 1 ? 1 : 2;
    // output n' has an element (annihilation: the mode is empty in n'), its sign
    static __device__ __forceinline__ constexpr bool has(int np) { return ((np & flip) != 0) == (O >= 2); }
    static __device__ __forceinline__ constexpr int sgn(int np) { return (O & 1) && (np & 2) ? -1 : 1; }
};
template <class F>
__device__ __forceinline__ void adj_by_op(int o, F f) {
    switch (o) {
        case 0: f(AdjMat<0>{}); break;
        case 1: f(AdjMat<1>{}); break;
        case 2: f(AdjMat<2>{}); break;
        default: f(AdjMat<3>{}); break;
    }
}
template <class T>
struct AdjOp {
    int o;
    T c;
};

// Layer l applied to the block Z[w][n] (2^NL x 4) at site s (input side bit l = a,
// output side bit l = b): Z'[b=0][n'] = par[n'] Z[a=0][n'],
// Z'[b=1][n'] = c sgn[n'] Z[a=0][src[n']] + Z[a=1][n'].
template <int L, class T, int NW>
__device__ __forceinline__ void adj_layer_fwd(T (&Z)[NW][4], const AdjOp<T>& op) {
    adj_by_op(op.o, [&](auto mat) {
        using M = decltype(mat);
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            if (w & (1 << L)) continue;
            const int w1 = w | (1 << L);
#pragma unroll
            for (int n = 0; n < 4; ++n)
                if (M::has(n)) Z[w1][n] += (M::sgn(n) < 0 ? -op.c : op.c) * Z[w][n ^ M::flip];
#pragma unroll
            for (int n = 0; n < 4; ++n)
                if (adj_par(n) < 0) Z[w][n] = -Z[w][n];
        }
    });
}

// Transposed layer l on the output-side block Z[w'][n'] -> input side:
// Z'[a=0][n] = par[n] Z[b=0][n] + sum_{n': src[n'] = n} c sgn[n'] Z[b=1][n'],
// Z'[a=1][n] = Z[b=1][n].  DERIV: the layer's derivative with respect to c
// (only the c b block, c = 1): Z'[a=0][n] = sum_{src[n'] = n} sgn[n'] Z[b=1][n'],
// Z'[a=1] = 0.  ZERO: bits of w whose blocks are zero (below a derivative) and skipped.
template <int L, bool DERIV, int ZERO, class T, int NW>
__device__ __forceinline__ void adj_layer_bwd(T (&Z)[NW][4], const AdjOp<T>& op) {
    adj_by_op(op.o, [&](auto mat) {
        using M = decltype(mat);
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            if ((w & (1 << L)) || (w & ZERO)) continue;
            const int w1 = w | (1 << L);
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                const int np = n ^ M::flip;
                const T z1 = M::sgn(np) < 0 ? -Z[w1][np] : Z[w1][np];
                if (DERIV) Z[w][n] = M::has(np) ? z1 : T(0);
                else if (M::has(np)) Z[w][n] = op.c * z1 + (adj_par(n) < 0 ? -Z[w][n] : Z[w][n]);
                else if (adj_par(n) < 0) Z[w][n] = -Z[w][n];
            }
            if (DERIV)
#pragma unroll
                for (int n = 0; n < 4; ++n) Z[w1][n] = T(0);
        }
    });
}
template <int L, int ZERO, class T, int NW, int NL>
__device__ __forceinline__ void adj_below(T (&Z)[NW][4], const AdjOp<T> (&op)[NL]) {  // layers L-1 .. 0
    if constexpr (L > 0) {
        adj_layer_bwd<L - 1, false, ZERO>(Z, op[L - 1]);
        adj_below<L - 1, ZERO>(Z, op);
    }
}

// A dot of float32 blocks in about 48 bits without the FP64 pipe (2 FMAs a clock
// and SM, which bounded the backward kernel): exact products and TwoSum in
// float-float.  That holds in float32's exponent range only: a product below 2^-149
// vanishes, one below 2^-102 has no exact error term, one above 2^128 is infinite.
// A thread loses at most 2^-150 for each of its up to 64 products and error terms, a
// CTA of 256 threads 2^-136: no more than a float64 sum's rounding beside one dot of
// at least 2^-82.  seen collects, per layer l, whether there is such a dot (bit l) and
// whether one is not finite (bit 8 + l); a CTA that misses the one or has the other
// takes its sums again in float64 (WIDE), as all sums of float64 blocks are.
template <bool WIDE, int NB>
__device__ __forceinline__ double adj_dot(const float (&x)[NB], const float (&z)[NB], int l, unsigned& seen) {
    if constexpr (WIDE) {
        double s = 0.0;
#pragma unroll
        for (int i = 0; i < NB; ++i) s += (double)x[i] * (double)z[i];
        return s;
    }
    float hi = 0.f, lo = 0.f;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const float p = x[i] * z[i], e = fmaf(x[i], z[i], -p), s = hi + p, bp = s - hi;
        lo += ((hi - (s - bp)) + (p - bp)) + e;
        hi = s;
    }
    const float t = fabsf(hi + lo);
    seen |= t >= 0x1p-82f ? 1u << l : 0u;
    seen |= t <= 0x1p126f ? 0u : 256u << l;
    return (double)hi + (double)lo;
}
template <bool WIDE, int NB>
__device__ __forceinline__ double adj_dot(const double (&x)[NB], const double (&z)[NB], int, unsigned&) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < NB; ++i) s += x[i] * z[i];
    return s;
}

// part[dl] = X . (M'^dl^T Q) for dl = L .. 0: Z holds Q taken through the layers
// above; a copy goes through the derivative of layer L and the layers below it,
// then Z through layer L.  Half of the copy's blocks are zero.
template <bool WIDE, int L, class T, int NW, int NL>
__device__ __forceinline__ void adj_derivs(T (&Z)[NW][4], const T (&X)[NW][4], const AdjOp<T> (&op)[NL],
                                           double (&part)[NL], unsigned& seen) {
    T D[NW][4];
#pragma unroll
    for (int w = 0; w < NW; ++w)
#pragma unroll
        for (int n = 0; n < 4; ++n) D[w][n] = Z[w][n];
    adj_layer_bwd<L, true, 0>(D, op[L]);
    adj_below<L, 1 << L>(D, op);
    T xs[2 * NW], ds[2 * NW];  // the entries that are not zero: w without bit L
#pragma unroll
    for (int i = 0; i < 2 * NW; ++i) {
        const int w = ((i / 4) >> L << (L + 1)) | ((i / 4) & ((1 << L) - 1));
        xs[i] = X[w][i % 4];
        ds[i] = D[w][i % 4];
    }
    part[L] = adj_dot<WIDE>(xs, ds, L, seen);
    adj_layer_bwd<L, false, 0>(Z, op[L]);
    if constexpr (L > 0) adj_derivs<WIDE, L - 1>(Z, X, op, part, seen);
}

// Y[b][a][n'][w'][bp] = (M_s X)[...] for X[b][a][w][n][bp]; one thread per
// (a, bp), blockIdx.y = term b; sb = the buffers' stride between terms.
template <class T, int NL>
__global__ void __launch_bounds__(256) k_adj_fwd(int Da, int Db, long sb, const T* X, T* Y, AdjTerms<T> tm, int s) {
    constexpr int NW = 1 << NL;
    const long per = (long)Da * Db;
    const long idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (idx >= per) return;
    const int b = blockIdx.y;
    const int a = (int)(idx / Db), bp = (int)(idx % Db);
    const T* x = X + (long)b * sb;
    T Z[NW][4];
#pragma unroll
    for (int w = 0; w < NW; ++w)
#pragma unroll
        for (int n = 0; n < 4; ++n) Z[w][n] = x[(((long)a * NW + w) * 4 + n) * Db + bp];
    auto op = [&](int l) { return AdjOp<T>{tm.op[b * NL + l], tm.coef[((long)b * NL + l) * tm.L + s]}; };
    adj_layer_fwd<0>(Z, op(0));
    adj_layer_fwd<1>(Z, op(1));
    if constexpr (NL == 4) {
        adj_layer_fwd<2>(Z, op(2));
        adj_layer_fwd<3>(Z, op(3));
    }
    T* y = Y + (long)b * sb;
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int w = 0; w < NW; ++w) y[(((long)a * 4 + n) * NW + w) * Db + bp] = Z[w][n];
}

// One thread's part of the backward kernel: P = M_s^T Q (PUT), and its coefficient
// gradients.
template <bool WIDE, bool PUT, class T, int NL>
__device__ __forceinline__ void adj_bwd_thread(int Db, const T* q, const T* x, T* p, const AdjTerms<T>& tm, int b, int s,
                                               int a, int bp, double (&part)[NL], unsigned& seen) {
    constexpr int NW = 1 << NL;
    T Z[NW][4], Zx[NW][4];
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int w = 0; w < NW; ++w) Z[w][n] = q[(((long)a * 4 + n) * NW + w) * Db + bp];
#pragma unroll
    for (int w = 0; w < NW; ++w)
#pragma unroll
        for (int n = 0; n < 4; ++n) Zx[w][n] = x[(((long)a * NW + w) * 4 + n) * Db + bp];
    auto op = [&](int l) { return AdjOp<T>{tm.op[b * NL + l], tm.coef[((long)b * NL + l) * tm.L + s]}; };
    if constexpr (NL == 4) {
        const AdjOp<T> ops[4] = {op(0), op(1), op(2), op(3)};
        adj_derivs<WIDE, 3>(Z, Zx, ops, part, seen);
    } else {
        const AdjOp<T> ops[2] = {op(0), op(1)};
        adj_derivs<WIDE, 1>(Z, Zx, ops, part, seen);
    }
    if (PUT)
#pragma unroll
        for (int w = 0; w < NW; ++w)
#pragma unroll
            for (int n = 0; n < 4; ++n) p[(((long)a * NW + w) * 4 + n) * Db + bp] = Z[w][n];
}

// P[b][a][w][n][bp] = (M_s^T Q)[...] for Q[b][a][n'][w'][bp], and
// g[b][l][s] += sum X . (M'^l^T Q) (the coefficient gradients, reduced per block,
// one float64 atomic per block and layer).  One thread per (a, bp), blockIdx.y = b.
template <class T, int NL>
__global__ void __launch_bounds__(256) k_adj_bwd(int Da, int Db, long sb, const T* Q, T* P, const T* X, double* g,
                                                AdjTerms<T> tm, int s) {
    __shared__ double red[NL][8];
    __shared__ unsigned seen_w[8];
    const long per = (long)Da * Db;
    const long idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
    const bool live = idx < per;
    const int b = blockIdx.y;
    const int a = live ? (int)(idx / Db) : 0, bp = live ? (int)(idx % Db) : 0;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const T *q = Q + (long)b * sb, *x = X + (long)b * sb;
    double part[NL];
    auto reduce = [&] {  // the warps' sums to red
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            const double v = warp_sum(part[l]);
            if (lane == 0) red[l][wid] = v;
        }
    };
    unsigned seen = 0;
#pragma unroll
    for (int l = 0; l < NL; ++l) part[l] = 0.0;
    if (live) adj_bwd_thread<false, true, T, NL>(Db, q, x, P + (long)b * sb, tm, b, s, a, bp, part, seen);
    reduce();
    if (sizeof(T) == 4) {
        seen = __reduce_or_sync(0xffffffffu, seen);
        if (lane == 0) seen_w[wid] = seen;
    }
    __syncthreads();
    if constexpr (sizeof(T) == 4) {
        seen = 0;
        for (int w = 0; w < nw; ++w) seen |= seen_w[w];
        if (seen != (1u << NL) - 1) {  // the whole CTA alike
            __syncthreads();
#pragma unroll
            for (int l = 0; l < NL; ++l) part[l] = 0.0;
            if (live) adj_bwd_thread<true, false, T, NL>(Db, q, x, nullptr, tm, b, s, a, bp, part, seen);
            reduce();
            __syncthreads();
        }
    }
    if (threadIdx.x < NL) {
        double v = 0.0;
        for (int w = 0; w < nw; ++w) v += red[threadIdx.x][w];
        atomicAdd(&g[((long)b * NL + threadIdx.x) * tm.L + s], v);
    }
}

// The value of every term: E_L[b][0][NW-1][0].
template <class T>
__global__ void k_adj_values(int B, const T* EL, long strideE, int NW, double* val) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) val[b] = (double)EL[(long)b * strideE + (NW - 1)];
}

// boundary environments: E_0[b][0][0][0] = 1 (w = 0); R_L[b][0][NW-1][0] = 1
template <class T>
__global__ void k_adj_boundary(int B, T* E0, long sE, T* RL, long sR, int NW) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    for (int w = 0; w < NW; ++w) {
        E0[(long)b * sE + w] = T(w == 0 ? 1 : 0);
        RL[(long)b * sR + w] = T(w == NW - 1 ? 1 : 0);
    }
}

// dpsi_s += sum_b weight_b G[b] (one site, n elements per term, terms sg apart)
template <class T>
__global__ void k_adj_accum_site(int B, const T* G, long sg, long n, const double* weight, T* out) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        double acc = 0.0;
        for (int b = 0; b < B; ++b) acc += weight[b] * (double)G[(long)b * sg + i];
        out[i] = T((double)out[i] + acc);
    }
}

// The terms of H as layers.  kind 0 (one-body, 2L terms): j -> (q = j % L,
// s = j / L): layer 0 = a_{q s} (coefficient e_q), layer 1 = sum_p t_pq a+_{p s};
// weight 1.  kind 1 (Coulomb, 4N^2 terms, index ((s'N + nu)2 + s)N + mu):
// layers A_{nu s'}, A+_{nu s'}, A_{mu s}, A+_{mu s} (coefficients chi^nu, chi^nu,
// chi^mu, chi^mu); weight zeta^{mu nu} / 2.
template <class T>
__global__ void k_adj_terms(int kind, long t0, int B, int L, int N, const double* t, const double* chi,
                            const double* zeta, int* op, T* coef, double* weight) {
    const int b = blockIdx.x;
    if (b >= B) return;
    const long tt = t0 + b;
    if (kind == 0) {
        const int q = (int)(tt % L), sg = (int)(tt / L);
        for (int s = threadIdx.x; s < L; s += blockDim.x) {
            coef[((long)b * 2 + 0) * L + s] = T(s == q ? 1.0 : 0.0);
            coef[((long)b * 2 + 1) * L + s] = T(t[(long)s * L + q]);
        }
        if (threadIdx.x == 0) {
            op[b * 2 + 0] = sg;
            op[b * 2 + 1] = sg + 2;
            weight[b] = 1.0;
        }
    } else {
        const int mu = (int)(tt % N);
        long rest = tt / N;
        const int sg = (int)(rest % 2);
        rest /= 2;
        const int nu = (int)(rest % N), sp = (int)(rest / N);
        for (int s = threadIdx.x; s < L; s += blockDim.x) {
            const double cn = chi[(long)s * N + nu], cm = chi[(long)s * N + mu];
            coef[((long)b * 4 + 0) * L + s] = T(cn);
            coef[((long)b * 4 + 1) * L + s] = T(cn);
            coef[((long)b * 4 + 2) * L + s] = T(cm);
            coef[((long)b * 4 + 3) * L + s] = T(cm);
        }
        if (threadIdx.x == 0) {
            op[b * 4 + 0] = sp;
            op[b * 4 + 1] = sp + 2;
            op[b * 4 + 2] = sg;
            op[b * 4 + 3] = sg + 2;
            weight[b] = 0.5 * zeta[(long)mu * N + nu];
        }
    }
}

// Fold a batch of terms into the value and the parameter gradients (float64
// atomics): value += w_b v_b; kind 0: dt[p][q] += g[b][1][p]; kind 1:
// dzeta[mu][nu] += v_b / 2, dchi[s][nu] += w_b (g0 + g1)[s], dchi[s][mu] += w_b (g2 + g3)[s].
static __global__ void k_adj_params(int kind, long t0, int B, int L, int N, const double* val, const double* g,
                             const double* weight, double* value, double* dt, double* dchi, double* dzeta) {
    const int b = blockIdx.x;
    if (b >= B) return;
    const long tt = t0 + b;
    const double w = weight[b], v = val[b];
    if (threadIdx.x == 0) atomicAdd(value, w * v);
    if (kind == 0) {
        const int q = (int)(tt % L);
        if (dt)
            for (int p = threadIdx.x; p < L; p += blockDim.x) atomicAdd(&dt[(long)p * L + q], g[((long)b * 2 + 1) * L + p]);
    } else {
        const int mu = (int)(tt % N);
        const int nu = (int)((tt / (2L * N)) % N);
        if (dzeta && threadIdx.x == 0) atomicAdd(&dzeta[(long)mu * N + nu], 0.5 * v);
        if (dchi)
            for (int s = threadIdx.x; s < L; s += blockDim.x) {
                const double* gb = g + (long)b * 4 * L;
                atomicAdd(&dchi[(long)s * N + nu], w * (gb[0 * L + s] + gb[1 * L + s]));
                atomicAdd(&dchi[(long)s * N + mu], w * (gb[2 * L + s] + gb[3 * L + s]));
            }
    }
}

}  // namespace thc
