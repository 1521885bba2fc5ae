// The coarse tail of the V-cycle as one dense operator.
//
// From a zero guess the V-cycle on levels t .. L-1 is a fixed linear map
// e = B b of level t's right-hand side (Sec. 2.2: stationary sweeps, R, P and
// the direct coarsest solve).  On levels of at most kTailRows rows every step
// of that chain is one launch of a few microseconds whose only cost is its
// dependent load chain, so B (n_t x n_t) is formed once per smoother and
// applied as one matrix-vector product instead of 7 launches per level.
// Measured on GB300 (per pass, before -> after): one V-cycle on 9k / 280k
// unstructured rows 71 -> 52 / 173 -> 138 us, on a 1025^2 grid (Jacobi)
// 209 -> 186 us; a whole FP64 solve on a 64^2 grid 926 -> 681 us; prediction
// and solve on the 50k mesh 4.43 -> 3.60 ms with B re-formed in every pass.
//
// The coarsest solve of an FP32 V-cycle is FP64, so B is held and applied in
// FP32 pairs (about 48 bits) and e is rounded once: PRECISION_FIGURES
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace amg {

// Largest level a tail starts on: at 1024 rows B is 4 MB (FP32), 27 KB an SM.
// Forming it costs n_t times the tail's entries: the next RS level (about 2300
// rows) would take five times the memory and the work, in every call that has
// new coefficients.
constexpr int kTailRows = 1024;
constexpr int kTailMaxLevels = 16;     // levels of a tail (kernel argument arrays)
constexpr int kTailCols = 4;           // columns of B a CTA forms at a time
constexpr int kTailThreads = 512;
constexpr size_t kTailSmem = 220 * 1024;         // shared memory a tail's level vectors may take
constexpr double kTailCoarseWork = 134217728.0;  // n_t n_L^2 bound: the FP64 coarsest solves of the n_t columns

// The FP32 V-cycle's B is formed in FP32 pairs (FloatPair): GB300 runs 64
// FP32 FMAs for each FP64 one, so the ten FP32 operations of a pair FMA are
// ~6x cheaper than a DFMA.
// acc += a x (Dekker / Knuth error-free product and sum)
__device__ __forceinline__ void tail_fma(FloatPair &acc, float a, const FloatPair &x) {
    const float p = __fmul_rn(a, x.h);
    const float e = __fmaf_rn(a, x.l, __fmaf_rn(a, x.h, -p));
    pair_add(acc, p, e);
}
__device__ __forceinline__ void tail_fma(double &acc, double a, const double &x) { acc = fma(a, x, acc); }

__device__ __forceinline__ FloatPair tail_norm(const FloatPair &v) {
    const float h = __fadd_rn(v.h, v.l);
    return {h, __fadd_rn(v.l, -__fadd_rn(h, -v.h))};
}
__device__ __forceinline__ double tail_norm(double v) { return v; }

__device__ __forceinline__ void tail_set(FloatPair &v, double x) {
    v.h = static_cast<float>(x);
    v.l = static_cast<float>(x - static_cast<double>(v.h));
}
__device__ __forceinline__ void tail_set(double &v, double x) { v = x; }
__device__ __forceinline__ double tail_get(const FloatPair &v) { return static_cast<double>(v.h) + static_cast<double>(v.l); }
__device__ __forceinline__ double tail_get(double v) { return v; }
__device__ __forceinline__ float tail_round(const FloatPair &v) { return __fadd_rn(v.h, v.l); }
__device__ __forceinline__ double tail_round(double v) { return v; }
// B's entry k (and, `lo` entries behind it, a pair's low word)
__device__ __forceinline__ void tail_store(float *B, size_t lo, size_t k, const FloatPair &v) {
    B[k] = v.h;
    B[lo + k] = v.l;
}
__device__ __forceinline__ void tail_store(double *B, size_t, size_t k, double v) { B[k] = v; }
__device__ __forceinline__ void tail_add(FloatPair &a, const FloatPair &b) { pair_add(a, b.h, b.l); }
__device__ __forceinline__ void tail_add(double &a, double b) { a += b; }
__device__ __forceinline__ FloatPair tail_shfl(const FloatPair &v, int o) {
    return {__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)};
}
__device__ __forceinline__ double tail_shfl(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }

// What T's values are held in while B is formed and applied.
template <class T> struct TailValue {
    using type = double;
};
template <> struct TailValue<float> {
    using type = FloatPair;
};

template <class T> struct TailCsr {
    const int *rp, *col;
    const T *val;
};

template <class T> struct TailLevel {
    int n, off;                 // rows; start of the level's b, u, r in shared memory (elements)
    TailCsr<T> A, P, R;
    const T *m;                 // Q^-1 on A's pattern (pseudo-inverse) or omega / a_ii (Jacobi)
};

template <class T> struct TailArgs {
    int nlev, nu1, nu2, pinv, ld;
    TailLevel<T> lev[kTailMaxLevels];
    const double *Linv, *LinvT;
    T *B;                       // n_t rows of ld entries (FP32: the low words n_t ld entries behind)
};

// acc[c] = (NEG ? -1 : 1) sum_k m_ik x_kc of one CSR row and kTailCols columns
template <bool NEG, class T, class V>
__device__ __forceinline__ void tail_row(const TailCsr<T> &M, int row, const V *__restrict__ x, V (&acc)[kTailCols]) {
    const int e = __ldg(M.rp + row + 1);
    for (int p = __ldg(M.rp + row); p < e; p += 4) {
        int c[4];
        T v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            c[j] = p + j < e ? __ldg(M.col + p + j) : 0;
            v[j] = p + j < e ? __ldg(M.val + p + j) : T(0);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (p + j >= e) break;
            const T a = NEG ? -v[j] : v[j];
#pragma unroll
            for (int k = 0; k < kTailCols; ++k) tail_fma(acc[k], a, x[c[j] * kTailCols + k]);
        }
    }
}

// One smoothing sweep u += M (b - A u) on a level's columns (all threads).
template <class T, class V>
__device__ void tail_sweep(const TailLevel<T> &L, int pinv, const V *b, V *u, V *r) {
    for (int i = threadIdx.x; i < L.n; i += kTailThreads) {
        V acc[kTailCols];
#pragma unroll
        for (int k = 0; k < kTailCols; ++k) acc[k] = b[i * kTailCols + k];
        tail_row<true>(L.A, i, u, acc);
#pragma unroll
        for (int k = 0; k < kTailCols; ++k) r[i * kTailCols + k] = tail_norm(acc[k]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < L.n; i += kTailThreads) {
        V acc[kTailCols];
#pragma unroll
        for (int k = 0; k < kTailCols; ++k) acc[k] = u[i * kTailCols + k];
        if (pinv) {
            tail_row<false>(TailCsr<T>{L.A.rp, L.A.col, L.m}, i, r, acc);
        } else {
            const T j = L.m[i];
#pragma unroll
            for (int k = 0; k < kTailCols; ++k) tail_fma(acc[k], j, r[i * kTailCols + k]);
        }
#pragma unroll
        for (int k = 0; k < kTailCols; ++k) u[i * kTailCols + k] = tail_norm(acc[k]);
    }
    __syncthreads();
}

// Columns kTailCols blockIdx.x .. of B: the V-cycle of the tail run on unit
// vectors, every level's b, u, r for those columns in shared memory, so one
// launch forms B without grid-wide steps (each CTA re-reads the levels'
// matrices from L2).  Dynamic shared memory: 3 sum_l n_l kTailCols values.
template <class T, class V>
__global__ void __launch_bounds__(kTailThreads) k_tail_build(const __grid_constant__ TailArgs<T> A) {
    extern __shared__ __align__(16) unsigned char tail_smem[];
    V *sm = reinterpret_cast<V *>(tail_smem);
    const int j0 = blockIdx.x * kTailCols, nt = A.lev[0].n, last = A.nlev - 1;
    V zero;
    tail_set(zero, 0.0);
    {
        V *b = sm + A.lev[0].off;
        V one;
        tail_set(one, 1.0);
        for (int e = threadIdx.x; e < nt * kTailCols; e += kTailThreads)
            b[e] = (e / kTailCols == j0 + e % kTailCols) ? one : zero;
    }
    __syncthreads();
    for (int l = 0; l < last; ++l) {
        const TailLevel<T> &L = A.lev[l];
        V *b = sm + L.off, *u = b + L.n * kTailCols, *r = u + L.n * kTailCols;
        for (int i = threadIdx.x; i < L.n; i += kTailThreads) {   // first sweep from zero: u = M b
            V acc[kTailCols];
#pragma unroll
            for (int k = 0; k < kTailCols; ++k) acc[k] = zero;
            if (A.nu1 > 0 && A.pinv) {
                tail_row<false>(TailCsr<T>{L.A.rp, L.A.col, L.m}, i, b, acc);
            } else if (A.nu1 > 0) {
                const T j = L.m[i];
#pragma unroll
                for (int k = 0; k < kTailCols; ++k) tail_fma(acc[k], j, b[i * kTailCols + k]);
            }
#pragma unroll
            for (int k = 0; k < kTailCols; ++k) u[i * kTailCols + k] = tail_norm(acc[k]);
        }
        __syncthreads();
        for (int s = 1; s < A.nu1; ++s) tail_sweep<T, V>(L, A.pinv, b, u, r);
        for (int i = threadIdx.x; i < L.n; i += kTailThreads) {   // r = b - A u
            V acc[kTailCols];
#pragma unroll
            for (int k = 0; k < kTailCols; ++k) acc[k] = b[i * kTailCols + k];
            tail_row<true>(L.A, i, u, acc);
#pragma unroll
            for (int k = 0; k < kTailCols; ++k) r[i * kTailCols + k] = tail_norm(acc[k]);
        }
        __syncthreads();
        const TailLevel<T> &C = A.lev[l + 1];
        V *bc = sm + C.off;
        for (int i = threadIdx.x; i < C.n; i += kTailThreads) {   // b_{l+1} = R r
            V acc[kTailCols];
#pragma unroll
            for (int k = 0; k < kTailCols; ++k) acc[k] = zero;
            tail_row<false>(L.R, i, r, acc);
#pragma unroll
            for (int k = 0; k < kTailCols; ++k) bc[i * kTailCols + k] = tail_norm(acc[k]);
        }
        __syncthreads();
    }
    {   // coarsest level: u = L^-T (L^-1 b) in FP64; y is kept in r as doubles
        const int n = A.lev[last].n;
        const V *b = sm + A.lev[last].off;
        V *u = sm + A.lev[last].off + n * kTailCols;
        static_assert(sizeof(V) == sizeof(double), "y shares r's storage");
        double *y = reinterpret_cast<double *>(u + n * kTailCols);
        for (int e = threadIdx.x; e < n * kTailCols; e += kTailThreads) {
            const int i = e / kTailCols, k = e % kTailCols;
            double acc = 0.0;
            for (int q = 0; q <= i; ++q) acc = fma(A.Linv[static_cast<size_t>(i) * n + q], tail_get(b[q * kTailCols + k]), acc);
            y[e] = acc;
        }
        __syncthreads();
        for (int e = threadIdx.x; e < n * kTailCols; e += kTailThreads) {
            const int i = e / kTailCols, k = e % kTailCols;
            double acc = 0.0;
            for (int q = i; q < n; ++q) acc = fma(A.LinvT[static_cast<size_t>(i) * n + q], y[q * kTailCols + k], acc);
            tail_set(u[e], acc);
        }
        __syncthreads();
    }
    for (int l = last - 1; l >= 0; --l) {
        const TailLevel<T> &L = A.lev[l];
        V *b = sm + L.off, *u = b + L.n * kTailCols, *r = u + L.n * kTailCols;
        const V *e = sm + A.lev[l + 1].off + A.lev[l + 1].n * kTailCols;
        for (int i = threadIdx.x; i < L.n; i += kTailThreads) {   // u += P e
            V acc[kTailCols];
#pragma unroll
            for (int k = 0; k < kTailCols; ++k) acc[k] = u[i * kTailCols + k];
            tail_row<false>(L.P, i, e, acc);
#pragma unroll
            for (int k = 0; k < kTailCols; ++k) u[i * kTailCols + k] = tail_norm(acc[k]);
        }
        __syncthreads();
        for (int s = 0; s < A.nu2; ++s) tail_sweep<T, V>(L, A.pinv, b, u, r);
    }
    const V *u = sm + A.lev[0].off + nt * kTailCols;
    for (int e = threadIdx.x; e < nt * kTailCols; e += kTailThreads) {
        const int i = e / kTailCols, j = j0 + e % kTailCols;
        if (j < nt) tail_store(A.B, static_cast<size_t>(nt) * A.ld, static_cast<size_t>(i) * A.ld + j, u[e]);
    }
}

// e = B b: a warp per row, its whole row of B (J 16-byte loads per lane, and
// as many of the low words) in registers before the grid-dependency wait (B is
// constant during a solve), so only the loads of b follow the previous
// kernel.  ld is n rounded up to 512 bytes; the padding of B is zero.
template <class T, int J>
__global__ void __launch_bounds__(kBlock) k_tail_apply(int n, int ld, const T *__restrict__ B,
                                                       const T *__restrict__ b, T *__restrict__ e) {
    constexpr bool kPair = sizeof(T) == 4;
    constexpr int W = 16 / sizeof(T);          // entries per 16-byte load
    using V = typename TailValue<T>::type;
    struct alignas(16) Vec { T v[W]; };
    const int row = blockIdx.x * (kBlock / 32) + static_cast<int>(threadIdx.x >> 5), lane = threadIdx.x & 31;
    Vec m[J], ml[kPair ? J : 1];
    const T *Br = B + static_cast<size_t>(row) * ld, *Bl = Br + static_cast<size_t>(n) * ld;
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int k = (j * 32 + lane) * W;
        const bool in = row < n && k < ld;
#pragma unroll
        for (int q = 0; q < W; ++q) m[j].v[q] = T(0);
        if (in) m[j] = *reinterpret_cast<const Vec *>(Br + k);
        if constexpr (kPair) {
#pragma unroll
            for (int q = 0; q < W; ++q) ml[j].v[q] = T(0);
            if (in) ml[j] = *reinterpret_cast<const Vec *>(Bl + k);
        }
    }
    pdl_wait_and_release();
    if (row >= n) return;
    V acc[W];
#pragma unroll
    for (int q = 0; q < W; ++q) tail_set(acc[q], 0.0);
    auto add = [&](int j, int q, T x) {
        if constexpr (kPair) tail_fma(acc[q], x, FloatPair{m[j].v[q], ml[j].v[q]});
        else tail_fma(acc[q], x, m[j].v[q]);
    };
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int k = (j * 32 + lane) * W;
        if (k + W <= n) {
            const Vec x = *reinterpret_cast<const Vec *>(b + k);
#pragma unroll
            for (int q = 0; q < W; ++q) add(j, q, x.v[q]);
        } else {
#pragma unroll
            for (int q = 0; q < W; ++q)
                if (k + q < n) add(j, q, b[k + q]);
        }
    }
    V s = acc[0];
#pragma unroll
    for (int q = 1; q < W; ++q) tail_add(s, acc[q]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tail_add(s, tail_shfl(s, o));
    if (lane == 0) e[row] = tail_round(s);
}

}  // namespace amg
