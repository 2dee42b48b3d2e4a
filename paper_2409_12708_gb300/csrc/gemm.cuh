// gemm.cuh -- batched, shared-memory tiled SIMT GEMM with functor operands
// (real or complex accumulators).
//
// C[b](m, n) = sum_k A[b](m, k) * B[b](k, n), with A and B produced element by
// element by loader functors (so the bond-2 MPO expansion, transposes and dtype
// conversions happen while a tile is staged into shared memory and never touch
// HBM) and C written by a store functor.  blockIdx.z is the batch index,
// blockIdx.y / blockIdx.x the row / column tile.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "scalar.cuh"

namespace thc {

template <class Acc, int BM, int BN, int BK, int TM, int TN, class LA, class LB, class SC>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
k_gemm(int M, int N, int K, LA la, LB lb, SC sc) {
    constexpr int TX = BN / TN;          // threads along n
    constexpr int TY = BM / TM;          // threads along m
    constexpr int NT = TX * TY;
    __shared__ Acc As[BK][BM + 1];
    __shared__ Acc Bs[BK][BN + 1];
    const int b = blockIdx.z;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int tid = threadIdx.x;
    const int tx = tid % TX, ty = tid / TX;
    Acc acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = tzero<Acc>();

    for (int k0 = 0; k0 < K; k0 += BK) {
        // A tile: consecutive threads walk k (row-major A is contiguous in k)
        for (int i = tid; i < BM * BK; i += NT) {
            const int mm = i / BK, kk = i % BK;
            const int m = m0 + mm, k = k0 + kk;
            As[kk][mm] = (m < M && k < K) ? cvt<Acc>(la(b, m, k)) : tzero<Acc>();
        }
        // B tile: consecutive threads walk n (row-major B is contiguous in n)
        for (int i = tid; i < BK * BN; i += NT) {
            const int kk = i / BN, nn = i % BN;
            const int k = k0 + kk, n = n0 + nn;
            Bs[kk][nn] = (k < K && n < N) ? cvt<Acc>(lb(b, k, n)) : tzero<Acc>();
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            Acc av[TM], bv[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) av[i] = As[kk][ty + i * TY];
#pragma unroll
            for (int j = 0; j < TN; ++j) bv[j] = Bs[kk][tx + j * TX];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] += av[i] * bv[j];
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int m = m0 + ty + i * TY;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int n = n0 + tx + j * TX;
            if (n < N) sc(b, m, n, acc[i][j]);
        }
    }
}

// Which index consecutive threads walk when a tile of A is loaded: k (row-major
// A), or m where the loader says that A is stored transposed (walk_m).
template <class LA, class = void>
struct WalkM : std::false_type {};
template <class LA>
struct WalkM<LA, std::enable_if_t<LA::walk_m>> : std::true_type {};

// Large-tile float32 variant: BM x BN tile (64 or 128 each), 256 threads, each
// thread 4 x 4 quadrants of C (rows 4ty.. and, at 128, 64+4ty.., columns alike), so
// every k step at 128 x 128 reads its operands with four 16-byte shared-memory
// loads for 64 multiply-adds, done on packed pairs of columns (32 instructions).
// The next BK-slice of the operands is loaded into registers while this one is
// multiplied, and two CTAs share an SM, which caps a thread at 128 registers: at
// 128 x 128 with slices of 8 some loaders spill 16 to 56 bytes, with 16 all do, to 232.
// Bound by the FMA pipe and by the functors' index arithmetic.  Measured: expand +
// absorb of 608 terms at L = 16, D = 128 83.5 -> 61.6 ms; the products of a gradient
// at L = 10, N = 30, D = 64 (bond 64: the 64-wide tiles) 41.9 -> 26.9 ms against
// one 4 x 4 block a thread without the prefetch.
template <int BM, int BN, int BK, class LA, class LB, class SC>
__global__ void __launch_bounds__(256, 2) k_gemm_tile(int M, int N, int K, LA la, LB lb, SC sc) {
    constexpr int RM = BM / 16, RN = BN / 16, NLA = BM * BK / 256, NLB = BN * BK / 256;
    __shared__ __align__(16) float As[BK][BM + 4];
    __shared__ __align__(16) float Bs[BK][BN + 4];
    const int b = blockIdx.z;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    float2 acc[RM][RN / 2];
    float ra[NLA], rb[NLB];
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN / 2; ++j) acc[i][j] = make_float2(0.f, 0.f);
    auto place_a = [&](int l, int& mm, int& kk) {
        const int i = tid + 256 * l;
        mm = WalkM<LA>::value ? i % BM : i / BK;
        kk = WalkM<LA>::value ? i / BM : i % BK;
    };
    auto fetch = [&](int k0) {
#pragma unroll
        for (int l = 0; l < NLA; ++l) {
            int mm, kk;
            place_a(l, mm, kk);
            const int m = m0 + mm, k = k0 + kk;
            ra[l] = (m < M && k < K) ? float(la(b, m, k)) : 0.f;
        }
#pragma unroll
        for (int l = 0; l < NLB; ++l) {
            const int i = tid + 256 * l, k = k0 + i / BN, n = n0 + i % BN;
            rb[l] = (k < K && n < N) ? float(lb(b, k, n)) : 0.f;
        }
    };
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
        for (int l = 0; l < NLA; ++l) {
            int mm, kk;
            place_a(l, mm, kk);
            As[kk][mm] = ra[l];
        }
#pragma unroll
        for (int l = 0; l < NLB; ++l) {
            const int i = tid + 256 * l;
            Bs[i / BN][i % BN] = rb[l];
        }
        __syncthreads();
        if (k0 + BK < K) fetch(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float av[RM];
            float2 bv[RN / 2];
#pragma unroll
            for (int h = 0; h < RM / 4; ++h) {
                const float4 x = *reinterpret_cast<const float4*>(&As[kk][64 * h + 4 * ty]);
                av[4 * h] = x.x;
                av[4 * h + 1] = x.y;
                av[4 * h + 2] = x.z;
                av[4 * h + 3] = x.w;
            }
#pragma unroll
            for (int h = 0; h < RN / 4; ++h) {
                const float4 x = *reinterpret_cast<const float4*>(&Bs[kk][64 * h + 4 * tx]);
                bv[2 * h] = make_float2(x.x, x.y);
                bv[2 * h + 1] = make_float2(x.z, x.w);
            }
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int j = 0; j < RN / 2; ++j) acc[i][j] = __ffma2_rn(make_float2(av[i], av[i]), bv[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < RM; ++i) {
        const int m = m0 + 64 * (i / 4) + 4 * ty + i % 4;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < RN; ++j) {
            const int n = n0 + 64 * (j / 4) + 4 * tx + j % 4;
            const float2 v = acc[i][j / 2];
            if (n < N) sc(b, m, n, j & 1 ? v.y : v.x);
        }
    }
}

// Small-tile variant: a BT x BT tile by 256 threads ((BT / 16)^2 outputs each),
// with the next BK-slice of the operands loaded into registers while this one is
// multiplied.  Every output is the same chain of multiply-adds over k as in
// k_gemm, so the two give the same bits.  What bounds it: for float64 the FP64
// pipe (2 FMAs a clock and SM), which a 64 x 64 tile spends on padding when M or
// N is small; at one instance the load latency of a slice, which more and
// smaller CTAs share out.  Measured (GB300): the 12 products of <phi|psi> at L = 6,
// D = 16 in float64 take 0.084 ms (0.389 ms with 64 x 64 tiles), the 150 of a
// complex64 time step at L = 5 2.5 ms (23.6 ms), the compression's float64
// products of H|psi> at L = 6, D = 16 3.4 ms (10.8 ms).
template <class Acc, int BT, int BK, class LA, class LB, class SC>
__global__ void __launch_bounds__(256) k_gemm_small(int M, int N, int K, LA la, LB lb, SC sc) {
    constexpr int TT = BT / 16, NL = BT * BK / 256;  // outputs per side, loads per operand and thread
    __shared__ Acc As[BK][BT + 1];
    __shared__ Acc Bs[BK][BT + 1];
    const int b = blockIdx.z;
    const int m0 = blockIdx.y * BT, n0 = blockIdx.x * BT;
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    Acc acc[TT][TT], ra[NL], rb[NL];
#pragma unroll
    for (int i = 0; i < TT; ++i)
#pragma unroll
        for (int j = 0; j < TT; ++j) acc[i][j] = tzero<Acc>();
    auto fetch = [&](int k0) {
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            const int i = tid + 256 * l;
            const int m = m0 + i / BK, ka = k0 + i % BK;  // consecutive threads walk k
            ra[l] = (m < M && ka < K) ? cvt<Acc>(la(b, m, ka)) : tzero<Acc>();
            const int n = n0 + i % BT, kb = k0 + i / BT;  // consecutive threads walk n
            rb[l] = (kb < K && n < N) ? cvt<Acc>(lb(b, kb, n)) : tzero<Acc>();
        }
    };
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            const int i = tid + 256 * l;
            As[i % BK][i / BK] = ra[l];
            Bs[i / BT][i % BT] = rb[l];
        }
        __syncthreads();
        if (k0 + BK < K) fetch(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            Acc av[TT], bv[TT];
#pragma unroll
            for (int i = 0; i < TT; ++i) av[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < TT; ++j) bv[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < TT; ++i)
#pragma unroll
                for (int j = 0; j < TT; ++j) acc[i][j] += av[i] * bv[j];
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TT; ++i) {
        const int m = m0 + ty + 16 * i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < TT; ++j) {
            const int n = n0 + tx + 16 * j;
            if (n < N) sc(b, m, n, acc[i][j]);
        }
    }
}

// Launch helper.  float32: the large-tile kernel, 128 wide where the output fills
// it, else 64.  64-bit accumulators: tiles of 32 when the output is wider than 16
// both ways and 32-tiles alone give two CTAs per SM (the loads, through functors
// that decode their index, then are shared by more outputs), else tiles of 16.
// 32-bit accumulators: tiles of 32 when M or N is at most 32 (half or more of a
// 64-tile would be padding), of 16 when both are at most 16.
template <class Acc, class LA, class LB, class SC>
inline cudaError_t launch_gemm(int batch, int M, int N, int K, const LA& la, const LB& lb,
                               const SC& sc, cudaStream_t st) {
    if (batch <= 0 || M <= 0 || N <= 0) return cudaSuccess;
    auto small = [&](auto bt) {
        constexpr int BT = decltype(bt)::value, BK = 16;
        dim3 grid(ceil_div(N, BT), ceil_div(M, BT), batch);
        k_gemm_small<Acc, BT, BK><<<grid, 256, 0, st>>>(M, N, K, la, lb, sc);
        return cudaGetLastError();
    };
    using Tile16 = std::integral_constant<int, 16>;
    using Tile32 = std::integral_constant<int, 32>;
    if constexpr (sizeof(real_t<Acc>) == 8) {
        const long tiles = (long)batch * ceil_div(M, 32) * ceil_div(N, 32);
        return M > 16 && N > 16 && tiles >= 2 * GB300_SMS ? small(Tile32{}) : small(Tile16{});
    } else {
        if (M <= 16 && N <= 16) return small(Tile16{});
        if (M <= 32 || N <= 32) return small(Tile32{});
        if constexpr (sizeof(Acc) == 4) {
            auto large = [&](auto bm, auto bn) {
                constexpr int BM = decltype(bm)::value, BN = decltype(bn)::value;
                dim3 grid(ceil_div(N, BN), ceil_div(M, BM), batch);
                k_gemm_tile<BM, BN, 8><<<grid, 256, 0, st>>>(M, N, K, la, lb, sc);
                return cudaGetLastError();
            };
            using T64 = std::integral_constant<int, 64>;
            using T128 = std::integral_constant<int, 128>;
            if (M >= 128 && N >= 128) return large(T128{}, T128{});
            if (M >= 128) return large(T128{}, T64{});
            if (N >= 128) return large(T64{}, T128{});
            return large(T64{}, T64{});
        } else {  // complex64
            constexpr int BM = 64, BN = 64, TM = 4, TN = 4, BK = 8;
            dim3 grid(ceil_div(N, BN), ceil_div(M, BM), batch);
            k_gemm<Acc, BM, BN, BK, TM, TN><<<grid, (BM / TM) * (BN / TN), 0, st>>>(M, N, K, la, lb, sc);
            return cudaGetLastError();
        }
    }
}

}  // namespace thc
