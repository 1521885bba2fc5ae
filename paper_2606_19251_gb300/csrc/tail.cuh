// The coarse tail of the V-cycle as one dense operator.
//
// From a zero guess the V-cycle on levels t .. L-1 is a fixed linear map
// e = B b of level t's right-hand side (Sec. 2.2: stationary sweeps, R, P and
// the direct coarsest solve).  On levels of at most kTailRows rows every step
// of that chain is one launch of a few microseconds whose only cost is its
// dependent load chain, so B (n_t x n_t) is formed once per smoother and
// applied as one matrix-vector product instead of 7 launches per level.
// Measured on GB300 (per pass, levels one by one -> with the tail): one V-cycle
// launched kernel by kernel on 9k / 280k unstructured rows 71 -> 52 / 173 ->
// 138 us, on a 1025^2 grid (Jacobi) 209 -> 186 us; a whole FP64 solve on a 64^2
// grid 926 -> 681 us; prediction and solve on the 50k mesh 4.43 -> 3.60 ms with
// B re-formed in every pass.  What forming B costs, and where the tail of a
// pseudo-inverse may start for it: kTailWork.
//
// The coarsest solve of an FP32 V-cycle is FP64, so B is held and applied in
// FP32 pairs (about 48 bits) and e is rounded once.  V-cycle error against
// 64 bits relative to the levels one by one, geometric mean of 48 seeds: 9k
// unstructured rows 0.99 (learned smoother) and 0.85 (Jacobi), 20k rows with
// cells of 100:1 0.96 and 0.78, 5-point grid of 10k rows 0.96 and 0.99; with B
// in FP32 and FP32 sums 0.97, 0.99, 0.99, 0.84, 0.96, 1.00.  The pairs cost 0 to
// 1.5 us a V-cycle (280k rows 136.2 -> 137.7).
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace amg {

// Largest level a tail starts on: at 1024 rows B is 8 MB, 54 KB an SM.  The
// next RS level (about 2300 rows) would take five times the memory and the
// work.
constexpr int kTailRows = 1024;
constexpr int kTailMaxLevels = 16;     // levels of a tail (kernel argument arrays)
constexpr int kTailCols = 4;           // columns of B a CTA forms at a time
constexpr int kTailThreads = 1024;
constexpr size_t kTailSmem = 220 * 1024;         // shared memory a tail's level vectors may take
// Bound of n_t x (entries of the tail's levels) where B is formed again with
// new values, in the first V-cycle or solve after them: always for the
// pseudo-inverse, for Jacobi after a change of omega.  The work is 8 passes
// over those entries for n_t columns (4 with Jacobi).  Measured, the
// pseudo-inverse's B: 280 rows, n_t x entries 1.3e6, 42 us; 513 rows, 3.0e6, 67
// us; 978 rows, 15.6e6, 220 us (FP64 409); 525 rows of a 3-D mesh, 18.7e6, 182 us
// (463).  Against that stand 5 to 10 us a V-cycle for a level of 500 to 1000
// rows more in the tail: it pays after 25 to 35 V-cycles, more than a solve with
// conjugate gradients takes.  Within the bounds amg_set_coeffs and a prediction
// with 0, 1, 2, ... V-cycles after them take no longer than with the levels one
// by one (9k rows, amg_set_coeffs and one V-cycle: 139 us one by one, 381 with
// the tail from 978 rows, 126 from 231 rows; FP64 168, 525, 167).  Jacobi's B
// is formed with the hierarchy, where 0.1 to 0.5 ms stand beside 5 to 50 ms of
// setup (1025^2 grid 45.5 -> 45.8 ms, 262k rows of a 3-D grid 28.2 -> 28.6), and
// is not bounded there.
constexpr double kTailWork = 4e6, kTailWork64 = 1.5e6;
constexpr int kTailLongRows = 32;      // FP64: four lanes a row from this mean length on
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

// Column g = tid % 4 of the sum over the row's four lanes (each holds its
// share of every column).
template <class V>
__device__ __forceinline__ V tail_scatter(const V (&acc)[kTailCols], int g) {
    static_assert(kTailCols == 4, "two exchange steps");
    const bool hi = g & 2;
    V a = hi ? acc[2] : acc[0], b = hi ? acc[3] : acc[1];
    tail_add(a, tail_shfl(hi ? acc[0] : acc[2], 2));
    tail_add(b, tail_shfl(hi ? acc[1] : acc[3], 2));
    const bool odd = g & 1;
    V s = odd ? b : a;
    tail_add(s, tail_shfl(odd ? a : b, 1));
    return s;
}

// f(k, M x at k) for every entry k = row kTailCols + column: LANES (1 or 4)
// lanes share a row's entries; of four, each then takes one column.
template <int LANES, class T, class V, class F>
__device__ __forceinline__ void tail_rows(int n, const TailCsr<T> &M, const V *x, const F &f) {
    struct alignas(16) Two { V a, b; };      // 16-byte loads: a level's vectors start at multiples of kTailCols
    const int g = threadIdx.x % LANES;
    for (int base = 0; base < n; base += kTailThreads / LANES) {
        const int row = base + static_cast<int>(threadIdx.x) / LANES;
        V acc[kTailCols];
#pragma unroll
        for (int k = 0; k < kTailCols; ++k) tail_set(acc[k], 0.0);
        if (row < n) {
            const int e = __ldg(M.rp + row + 1);
            for (int p0 = __ldg(M.rp + row) + g; p0 < e; p0 += 4 * LANES) {
                int c[4];
                T v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int p = p0 + j * LANES;
                    c[j] = p < e ? __ldg(M.col + p) : 0;
                    v[j] = p < e ? __ldg(M.val + p) : T(0);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (p0 + j * LANES >= e) break;
                    const Two *xr = reinterpret_cast<const Two *>(x + c[j] * kTailCols);
                    const Two lo = xr[0], hi = xr[1];
                    tail_fma(acc[0], v[j], lo.a);
                    tail_fma(acc[1], v[j], lo.b);
                    tail_fma(acc[2], v[j], hi.a);
                    tail_fma(acc[3], v[j], hi.b);
                }
            }
        }
        if constexpr (LANES == 1) {
            if (row < n) {
#pragma unroll
                for (int k = 0; k < kTailCols; ++k) f(row * kTailCols + k, acc[k]);
            }
        } else {
            const V s = tail_scatter(acc, g);
            if (row < n) f(row * kTailCols + g, s);
        }
    }
    __syncthreads();
}

// y = y + s with s negated on demand, renormalised
__device__ __forceinline__ FloatPair tail_sum(FloatPair y, const FloatPair &s, bool neg = false) {
    if (neg) pair_add(y, -s.h, -s.l);
    else pair_add(y, s.h, s.l);
    return tail_norm(y);
}
__device__ __forceinline__ double tail_sum(double y, double s, bool neg = false) { return neg ? y - s : y + s; }

// r = b - A u
template <int LANES, class T, class V>
__device__ __forceinline__ void tail_resid(const TailLevel<T> &L, const V *b, const V *u, V *r) {
    tail_rows<LANES>(L.n, L.A, u, [&](int k, const V &s) { r[k] = tail_sum(b[k], s, true); });
}

// u = (add ? u : 0) + M r
template <int LANES, class T, class V>
__device__ __forceinline__ void tail_smooth(const TailLevel<T> &L, int pinv, const V *r, V *u, bool add) {
    V zero;
    tail_set(zero, 0.0);
    if (pinv) {
        tail_rows<LANES>(L.n, TailCsr<T>{L.A.rp, L.A.col, L.m}, r, [&](int k, const V &s) { u[k] = tail_sum(add ? u[k] : zero, s); });
        return;
    }
    for (int k = threadIdx.x; k < L.n * kTailCols; k += kTailThreads) {
        V acc = add ? u[k] : zero;
        tail_fma(acc, __ldg(L.m + k / kTailCols), r[k]);
        u[k] = tail_norm(acc);
    }
    __syncthreads();
}

// Columns kTailCols blockIdx.x .. of B: the V-cycle of the tail run on unit
// vectors, every level's b, u, r for those columns in shared memory, so one
// launch forms B without grid-wide steps (each CTA re-reads the levels'
// matrices from L2).  Dynamic shared memory: 3 sum_l n_l kTailCols values.
// A step's time is its longest row's (coarse rows have 10 to 100 entries), so
// with FP32 pairs four lanes share a row and exchange their columns' sums at
// its end (one thread a row: 978 rows 285 -> 220 us, 525 rows of 60 entries 431
// -> 182, 280 rows 56 -> 42).  In FP64 the exchange costs as much of the narrow
// FP64 unit as a short row (978 rows of 13 entries 409 -> 509 us), so there four
// lanes take rows of kTailLongRows entries on average (525 rows 637 -> 463).
template <class T, class V, int LANES>
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
        if (A.nu1 > 0) {
            tail_smooth<LANES>(L, A.pinv, b, u, false);                      // first sweep from zero: u = M b
        } else {
            for (int k = threadIdx.x; k < L.n * kTailCols; k += kTailThreads) u[k] = zero;
            __syncthreads();
        }
        for (int s = 1; s < A.nu1; ++s) {
            tail_resid<LANES>(L, b, u, r);
            tail_smooth<LANES>(L, A.pinv, r, u, true);
        }
        tail_resid<LANES>(L, b, u, r);
        V *bc = sm + A.lev[l + 1].off;
        tail_rows<LANES>(A.lev[l + 1].n, L.R, r, [&](int k, const V &s) { bc[k] = tail_norm(s); });
    }
    {   // coarsest level: u = L^-T (L^-1 b) in FP64; y is kept in r as doubles
        const int n = A.lev[last].n;
        const V *b = sm + A.lev[last].off;
        V *u = sm + A.lev[last].off + n * kTailCols;
        static_assert(sizeof(V) == sizeof(double), "y shares r's storage");
        double *y = reinterpret_cast<double *>(u + n * kTailCols);
        // a warp's lanes take 32 / kTailCols terms of a row and its columns
        constexpr int kParts = 32 / kTailCols;
        const int k = threadIdx.x % kTailCols, part = threadIdx.x % 32 / kTailCols;
        auto total = [&](double v) {
#pragma unroll
            for (int o = kTailCols; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            return v;
        };
        for (int i = threadIdx.x / 32; i < n; i += kTailThreads / 32) {
            const double *row = A.Linv + static_cast<size_t>(i) * n;
            double acc = 0.0;
            for (int q = part; q <= i; q += kParts) acc = fma(row[q], tail_get(b[q * kTailCols + k]), acc);
            acc = total(acc);
            if (part == 0) y[i * kTailCols + k] = acc;
        }
        __syncthreads();
        for (int i = threadIdx.x / 32; i < n; i += kTailThreads / 32) {
            const double *row = A.LinvT + static_cast<size_t>(i) * n;
            double acc = 0.0;
            for (int q = i + part; q < n; q += kParts) acc = fma(row[q], y[q * kTailCols + k], acc);
            acc = total(acc);
            if (part == 0) tail_set(u[i * kTailCols + k], acc);
        }
        __syncthreads();
    }
    for (int l = last - 1; l >= 0; --l) {
        const TailLevel<T> &L = A.lev[l];
        V *b = sm + L.off, *u = b + L.n * kTailCols, *r = u + L.n * kTailCols;
        const V *e = sm + A.lev[l + 1].off + A.lev[l + 1].n * kTailCols;
        tail_rows<LANES>(L.n, L.P, e, [&](int k, const V &s) { u[k] = tail_sum(u[k], s); });
        for (int s = 0; s < A.nu2; ++s) {
            tail_resid<LANES>(L, b, u, r);
            tail_smooth<LANES>(L, A.pinv, r, u, true);
        }
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
