// The coarse levels of the training V-cycle and of its adjoint, each as one
// CTA's kernel.
//
// The training loss needs every sweep's residual of every level, so its
// V-cycle cannot take the coarse levels as one operator (tail.cuh).  As
// launches they are ten a level and direction of 2 to 2.5 us each, all of it
// launch and dependent loads on levels of a few hundred rows.  Here one CTA
// keeps the levels' vectors in shared memory and steps with __syncthreads, the
// matrices in its L1.  Every row is summed by as many lanes and in the same
// order as in the launched passes, so the V-cycle, its adjoint and with them
// the loss (one FP32-rounded number: another order would move it by its
// rounding) keep their bits.  The sums of dL/dc run over this one CTA's threads
// and over a level's sweeps before they are reduced, another order than the
// launched passes'; in FP32 pairs or FP64 they agree to about 1e-14.
// 12k-row mesh, three cycles: 739 -> 711 us a call; five-mesh training batch
// 5104 -> 4966.  The line: with levels up to 512 rows in the one CTA 725 -> 738
// us, up to 1024 rows 734 -> 745 (batch 5076 -> 5357): there the SMs that the
// launched passes spread over are worth more than the launches.
#pragma once
#include "tail.cuh"

namespace amg {

constexpr int kTrainTailRows = 256;     // largest level the CTA takes
constexpr int kTtThreads = 1024;
constexpr int kTtCoarse = 64;           // largest coarsest level
constexpr int kTtLd = kTtCoarse + 1;    // row stride of its factors in shared memory

// u r v for the row's own values u, r and a basis value v
__device__ __forceinline__ FloatPair adj_prod(float u, float r, const FloatPair &v) {
    const float t = __fmul_rn(u, r), tl = __fmaf_rn(u, r, -t);
    FloatPair o{__fmul_rn(t, v.h), 0.f};
    o.l = __fmaf_rn(t, v.l, __fmaf_rn(tl, v.h, __fmaf_rn(t, v.h, -o.h)));
    return o;
}
__device__ __forceinline__ double adj_prod(double u, double r, double v) { return u * r * v; }
// u v
__device__ __forceinline__ FloatPair adj_scale(float u, const FloatPair &v) {
    FloatPair o{__fmul_rn(u, v.h), 0.f};
    o.l = __fmaf_rn(u, v.l, __fmaf_rn(u, v.h, -o.h));
    return o;
}
__device__ __forceinline__ double adj_scale(double u, double v) { return u * v; }

template <class T, class V> struct TrainTailLevel {
    int n, off;                         // rows; first row in the concatenated level vectors
    int la, lp, lr;                     // log2 of the lanes per row of A, P and R
    TailCsr<T> A, P, R;
    const T *q;                         // Q^-1 on A's pattern
    const V *o1, *o2, *d;               // basis of dL/dc (AdjBasis)
    T *ck;                              // this cycle's checkpoints
    long long stride;                   // elements between them
    double *partial;                    // five sums of dL/dc
    T us;                               // the basis's scale (k_adj_sweep), inverted
};
template <class T, class V> struct TrainTailArgs {
    int nlev, nu1, nu2, rows;           // rows: all levels together
    TrainTailLevel<T, V> lev[kTailMaxLevels];
    const double *Linv, *LinvT;
    const T *in;                        // b (forward) or dL/d(output) (adjoint) of the first level
    T *out;                             // u (forward) or dL/db (adjoint) of the first level
    const float *scale;                 // r's and ubar's scale in the gradient sums (adjoint)
};

// One row's sum over `tpr` lanes, in the order of row_dot and group_sum.
template <class T> __device__ __forceinline__ T tt_group_sum(T v, int tpr) {
    for (int o = tpr / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// f(row, sum of M x) for every row, in lane 0 of the row's 2^lt lanes.
template <class T, class F>
__device__ __forceinline__ void tt_rows(int n, int lt, const TailCsr<T> &M, const T *x, const F &f) {
    const int tpr = 1 << lt, lane = threadIdx.x & (tpr - 1);
    for (int base = 0; base < n; base += kTtThreads >> lt) {
        const int row = base + (static_cast<int>(threadIdx.x) >> lt);
        T acc = T(0);
        if (row < n) {
            const int e = __ldg(M.rp + row + 1);
            for (int p0 = __ldg(M.rp + row) + lane; p0 < e; p0 += 4 * tpr) {
                int c[4];
                T v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int p = p0 + j * tpr;
                    c[j] = p < e ? __ldg(M.col + p) : 0;
                    v[j] = p < e ? __ldg(M.val + p) : T(0);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (p0 + j * tpr < e) acc += v[j] * x[c[j]];
            }
        }
        acc = tt_group_sum(acc, tpr);
        if (row < n && lane == 0) f(row, acc);
    }
    __syncthreads();
}

// The coarsest level's factors into shared memory (constant: ahead of the
// grid-dependency wait), zero where they have no entry.
__device__ __forceinline__ void tt_stage(int n, const double *__restrict__ Linv, const double *__restrict__ LinvT,
                                         double *sL) {
    for (int k = threadIdx.x; k < kTtCoarse * kTtCoarse; k += kTtThreads) {
        const int i = k / kTtCoarse, j = k % kTtCoarse;
        sL[i * kTtLd + j] = (i < n && j <= i) ? Linv[i * n + j] : 0.0;
        sL[(kTtCoarse + i) * kTtLd + j] = (i < n && j >= i && j < n) ? LinvT[i * n + j] : 0.0;
    }
}

// x = L^-T (L^-1 b) in FP64, summed as in k_coarse_warp (n <= 32) or k_coarse_64
template <class T>
__device__ __forceinline__ void tt_coarse(int n, const double *sL, const T *b, T *x) {
    __shared__ double sb[kTtCoarse], sy[kTtCoarse];
    const double *sLT = sL + kTtCoarse * kTtLd;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (threadIdx.x < kTtCoarse) {
        sb[threadIdx.x] = static_cast<int>(threadIdx.x) < n ? static_cast<double>(b[threadIdx.x]) : 0.0;
        sy[threadIdx.x] = 0.0;
    }
    __syncthreads();
    if (n <= 32) {
        if (warp == 0) {
            double y = 0.0, v = 0.0;
            if (lane < n)
                for (int k = 0; k <= lane; ++k) y = fma(sL[lane * kTtLd + k], sb[k], y);
            sy[lane] = y;
            __syncwarp();
            if (lane < n)
                for (int k = lane; k < n; ++k) v = fma(sLT[lane * kTtLd + k], sy[k], v);
            if (lane < n) x[lane] = static_cast<T>(v);
        }
    } else {
        for (int i = warp; i < n; i += kTtThreads / 32) {
            const double v = warp_sum(fma(sL[i * kTtLd + lane + 32], sb[lane + 32], sL[i * kTtLd + lane] * sb[lane]));
            if (lane == 0) sy[i] = v;
        }
        __syncthreads();
        for (int i = warp; i < n; i += kTtThreads / 32) {
            const double v = warp_sum(fma(sLT[i * kTtLd + lane + 32], sy[lane + 32], sLT[i * kTtLd + lane] * sy[lane]));
            if (lane == 0) x[i] = static_cast<T>(v);
        }
    }
    __syncthreads();
}

// One V-cycle from the tail's first level on, keeping b_l (slot 0, with
// pre-smoothing) and every later sweep's residual (slot k).  Dynamic shared
// memory: the coarsest factors, then 3 x rows of T.
template <class T, class V>
__global__ void __launch_bounds__(kTtThreads) k_train_tail_fwd(const __grid_constant__ TrainTailArgs<T, V> A) {
    extern __shared__ __align__(16) unsigned char tt_smem[];
    const int last = A.nlev - 1;
    double *sL = reinterpret_cast<double *>(tt_smem);
    T *sb = reinterpret_cast<T *>(sL + 2 * kTtCoarse * kTtLd), *su = sb + A.rows, *sr = su + A.rows;
    tt_stage(A.lev[last].n, A.Linv, A.LinvT, sL);
    pdl_wait_and_release();
    for (int i = threadIdx.x; i < A.lev[0].n; i += kTtThreads) sb[i] = A.in[i];
    __syncthreads();
    auto resid = [&](const TrainTailLevel<T, V> &L, T *ck) {      // r = b - A u, kept in ck
        const T *b = sb + L.off, *u = su + L.off;
        T *r = sr + L.off;
        tt_rows(L.n, L.la, L.A, u, [&](int i, T s) {
            const T v = b[i] - s;
            r[i] = v;
            if (ck) ck[i] = v;
        });
    };
    auto apply = [&](const TrainTailLevel<T, V> &L) {             // u += Q^-1 r
        T *u = su + L.off;
        tt_rows(L.n, L.la, TailCsr<T>{L.A.rp, L.A.col, L.q}, sr + L.off, [&](int i, T s) { u[i] = u[i] + s; });
    };
    for (int l = 0; l < last; ++l) {
        const TrainTailLevel<T, V> &L = A.lev[l];
        T *u = su + L.off;
        if (A.nu1 > 0) {
            if (l > 0)
                for (int i = threadIdx.x; i < L.n; i += kTtThreads) L.ck[i] = sb[L.off + i];
            tt_rows(L.n, L.la, TailCsr<T>{L.A.rp, L.A.col, L.q}, sb + L.off, [&](int i, T s) { u[i] = s; });
        } else {
            for (int i = threadIdx.x; i < L.n; i += kTtThreads) u[i] = T(0);
            __syncthreads();
        }
        for (int k = 1; k < A.nu1; ++k) {
            resid(L, L.ck + k * L.stride);
            apply(L);
        }
        resid(L, nullptr);
        T *bc = sb + A.lev[l + 1].off;
        tt_rows(A.lev[l + 1].n, L.lr, L.R, sr + L.off, [&](int i, T s) { bc[i] = s; });
    }
    tt_coarse<T>(A.lev[last].n, sL, sb + A.lev[last].off, su + A.lev[last].off);
    for (int l = last - 1; l >= 0; --l) {
        const TrainTailLevel<T, V> &L = A.lev[l];
        T *u = su + L.off;
        tt_rows(L.n, L.lp, L.P, su + A.lev[l + 1].off, [&](int i, T s) { u[i] = u[i] + s; });
        for (int k = A.nu1; k < A.nu1 + A.nu2; ++k) {
            resid(L, L.ck + k * L.stride);
            apply(L);
        }
    }
    for (int i = threadIdx.x; i < A.lev[0].n; i += kTtThreads) A.out[i] = su[i];
}

// The adjoint of that V-cycle: out = dL/db from in = dL/du, the levels'
// gradient sums added to `partial`.  Dynamic shared memory: the coarsest
// factors, then 4 x rows of T.
template <class T, class V>
__global__ void __launch_bounds__(kTtThreads) k_train_tail_adj(const __grid_constant__ TrainTailArgs<T, V> A) {
    extern __shared__ __align__(16) unsigned char tt_smem[];
    __shared__ V red[5][kTtThreads / 32];
    const int last = A.nlev - 1;
    double *sL = reinterpret_cast<double *>(tt_smem);
    T *sub = reinterpret_cast<T *>(sL + 2 * kTtCoarse * kTtLd), *sbb = sub + A.rows, *srb = sbb + A.rows, *sk = srb + A.rows;
    V zero;
    tail_set(zero, 0.0);
    V g[5];
    auto clear = [&]() {
#pragma unroll
        for (int k = 0; k < 5; ++k) g[k] = zero;
    };
    auto flush = [&](const TrainTailLevel<T, V> &L) {             // g into the level's five sums, fixed order
#pragma unroll
        for (int k = 0; k < 5; ++k) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) tail_add(g[k], tail_shfl(g[k], o));
            if (threadIdx.x % 32 == 0) red[k][threadIdx.x / 32] = g[k];
        }
        __syncthreads();
        if (threadIdx.x < 5) {
            V t = red[threadIdx.x][0];
            for (int k = 1; k < kTtThreads / 32; ++k) tail_add(t, red[threadIdx.x][k]);
            L.partial[threadIdx.x] += tail_get(t);
        }
        __syncthreads();
    };
    T sr = T(1), su = T(1);
    // rbar = M ubar, bbar (+)= rbar, and the sweep's share of dL/dc with the checkpoint ck
    auto sweep = [&](const TrainTailLevel<T, V> &L, const T *ck, bool assign) {
        const T *ub = sub + L.off;
        T *bb = sbb + L.off, *rb = srb + L.off, *r = sk + L.off;
        for (int i = threadIdx.x; i < L.n; i += kTtThreads) r[i] = ck[i] * sr;
        __syncthreads();
        const int tpr = 1 << L.la, lane = threadIdx.x & (tpr - 1);
        for (int base = 0; base < L.n; base += kTtThreads >> L.la) {
            const int row = base + (static_cast<int>(threadIdx.x) >> L.la);
            T acc = T(0);
            if (row < L.n) {
                V s3 = zero, s4 = zero;
                const int e = __ldg(L.A.rp + row + 1);
                for (int p = __ldg(L.A.rp + row) + lane; p < e; p += tpr) {
                    const int j = __ldg(L.A.col + p);
                    acc += __ldg(L.q + p) * ub[j];
                    tail_fma(s3, r[j], L.o1[p]);
                    tail_fma(s4, r[j], L.o2[p]);
                }
                const T ui = ub[row] * (su * L.us);
                tail_add(g[3], adj_scale(ui, s3));
                tail_add(g[4], adj_scale(ui, s4));
                if (lane == 0) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) tail_add(g[k], adj_prod(ui, r[row], L.d[3 * static_cast<size_t>(row) + k]));
                }
            }
            acc = tt_group_sum(acc, tpr);
            if (row < L.n && lane == 0) {
                rb[row] = acc;
                bb[row] = assign ? acc : bb[row] + acc;
            }
        }
        __syncthreads();
    };
    auto minus_a = [&](const TrainTailLevel<T, V> &L) {           // ubar -= A rbar
        T *ub = sub + L.off;
        tt_rows(L.n, L.la, L.A, srb + L.off, [&](int i, T s) { ub[i] = ub[i] - s; });
    };
    tt_stage(A.lev[last].n, A.Linv, A.LinvT, sL);
    pdl_wait_and_release();
    sr = A.scale[0];
    su = A.scale[1];
    for (int i = threadIdx.x; i < A.lev[0].n; i += kTtThreads) sub[i] = A.in[i];
    __syncthreads();
    for (int l = 0; l < last; ++l) {
        const TrainTailLevel<T, V> &L = A.lev[l];
        clear();
        for (int k = A.nu1 + A.nu2 - 1; k >= A.nu1; --k) {
            sweep(L, L.ck + k * L.stride, k == A.nu1 + A.nu2 - 1);
            minus_a(L);
        }
        flush(L);
        T *uc = sub + A.lev[l + 1].off;                            // ebar = P^T ubar = R ubar
        tt_rows(A.lev[l + 1].n, L.lr, L.R, sub + L.off, [&](int i, T s) { uc[i] = s; });
    }
    tt_coarse<T>(A.lev[last].n, sL, sub + A.lev[last].off, sbb + A.lev[last].off);
    for (int l = last - 1; l >= 0; --l) {
        const TrainTailLevel<T, V> &L = A.lev[l];
        T *bb = sbb + L.off, *rb = srb + L.off;
        const bool assign = A.nu2 == 0;
        tt_rows(L.n, L.lp, L.P, sbb + A.lev[l + 1].off, [&](int i, T s) {   // rhobar = R^T bbar_c
            rb[i] = s;
            bb[i] = assign ? s : bb[i] + s;
        });
        minus_a(L);
        clear();
        for (int k = A.nu1 - 1; k >= 1; --k) {
            sweep(L, L.ck + k * L.stride, false);
            minus_a(L);
        }
        if (A.nu1 >= 1) sweep(L, L.ck, false);   // first sweep from zero: u = M b
        flush(L);
    }
    for (int i = threadIdx.x; i < A.lev[0].n; i += kTtThreads) A.out[i] = sbb[i];
}

}  // namespace amg
